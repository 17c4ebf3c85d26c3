"""Kept features of attention heads by clusters of eight blocks (attn_features.cu), against the general score pass."""
import pytest
import torch

import paper_2608_13426_b200 as rmm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B, Hq, Hkv, Lq, Dh", [
    (1, 32, 8, 40, 128), (1, 8, 8, 17, 256), (1, 3, 1, 129, 72), (2, 2, 2, 1001, 64), (1, 1, 1, 4096, 128), (1, 1, 1, 4097, 128),
    (1, 33, 1, 64, 64), (1, 9, 9, 130, 136), (3, 5, 1, 300, 8), (1, 4, 2, 2048, 256), (1, 2, 1, 65000, 8),
    (1, 3, 1, 2560, 128), (1, 3, 1, 2561, 128), (1, 28, 4, 4352, 128), (1, 28, 4, 4353, 128), (1, 2, 1, 5120, 128), (1, 2, 1, 5121, 128), (1, 40, 8, 90, 64), (1, 41, 1, 90, 64),
    (1, 8, 8, 512, 256), (1, 8, 8, 513, 256)])   # either side of each line of attn_features_eligible
@pytest.mark.parametrize("rho", [0.5, 0.13, 1.0])
def test_features_are_those_of_the_general_pass(B, Hq, Hkv, Lq, Dh, rho):
    g = torch.Generator(device="cuda").manual_seed(Lq)
    Q = torch.randn(B, Hq, Lq, Dh, generator=g, device="cuda") * torch.rand(B, Hq, 1, Dh, generator=g, device="cuda")
    Q[..., 1] = Q[..., 4]                                     # equal energies: the lower index
    Q[:, 0, :, 2] = 0
    if Hq > 1:
        Q[:, 1, 0, 3], Q[:, 1, 0, 5] = float("inf"), float("nan")
    wide = torch.zeros(B, Lq, Hq, Dh + 8, dtype=torch.bfloat16, device="cuda")
    wide[..., :Dh] = Q.transpose(1, 2)
    K = torch.randn(B, Hkv, 64, Dh, generator=g, device="cuda").bfloat16()
    for q in (Q.bfloat16(), wide[..., :Dh].transpose(1, 2)):  # contiguous; rows and heads elsewhere
        _, feat, _ = rmm.rmm_reduced_attn(q, K, K, False, rho, 1.0, want_idx=True)
        want = rmm.rmm_score_select(q.reshape(B * Hq, Lq, Dh), rho=rho)[0].reshape(feat.shape)
        assert torch.equal(feat, want)
    assert rmm.rmm_status_read() == 0
