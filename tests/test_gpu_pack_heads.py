"""Packing of Q and K for the fused attention kernels, rows of 64, 128 and 256 columns (pack_heads_kernel in pack.cu)."""
import pytest
import torch

import paper_2608_13426_b200 as rmm
from paper_2608_13426_b200 import synth
from test_gpu_masked_tiles import padded
from test_gpu_parity import check_attention

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Dh, rho_d", [(64, 0.5), (64, 1.0), (128, 0.13), (128, 1.0), (256, 0.5), (256, 0.7), (256, 0.02)])
@pytest.mark.parametrize("Lq, Lk", [(17, 127), (128, 128), (129, 64), (65, 257)])   # edges of blocks of 64 and 128 rows
def test_packed_heads(oracle, Dh, rho_d, Lq, Lk):
    assert check_attention(oracle, 2, 4, 2, Lq, Lk, Dh, False, rho_d, 1.0, seed=Lq)
    Q, K, V = synth.attention_qkv(2, 4, 2, Lq, Lk, Dh, seed=Lk, device="cuda")
    mask = padded(2, Lq, Lk, [Lk - 3, 40]).cuda()                                 # the pass over it runs beside the packing
    want = [rmm.rmm_reduced_attn(Q, K, V, False, rho_d, mask=m) for m in (None, mask)]
    wide = [torch.randn(2, n, h, Dh + 8, device="cuda").bfloat16() for n, h in ((Lq, 4), (Lk, 2))]
    for t, x in zip(wide, (Q, K)):
        t[..., :Dh] = x.transpose(1, 2)
    q, k = (t[..., :Dh].transpose(1, 2) for t in wide)                            # rows and heads elsewhere
    for m, w in zip((None, mask), want):
        assert torch.equal(rmm.rmm_reduced_attn(q, k, V, False, rho_d, mask=m), w)
    mask.fill_(0)                                                                 # a new mask in the same place
    assert torch.equal(rmm.rmm_reduced_attn(Q, K, V, False, rho_d, mask=mask), want[0])
    assert rmm.rmm_status_read() == 0
