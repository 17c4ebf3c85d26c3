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


@pytest.mark.parametrize("B, Hq, Hkv, L, Dh, causal", [(2, 16, 4, 512, 128, True), (1, 4, 2, 1500, 64, False), (2, 40, 8, 390, 128, False)])
def test_masked_calls_in_flight(B, Hq, Hkv, L, Dh, causal):
    """Calls with different masks right behind one another: the pass over a mask runs beside the packing, while the attention kernel of
    the call before, which reads what that pass wrote for it, must be done."""
    Q, K, V = synth.attention_qkv(B, Hq, Hkv, L, L, Dh, seed=L, device="cuda")
    masks = [padded(B, L, L, [n, L - n // 2][:B]).cuda() for n in (40, 129, 300, L - 1)] + [torch.zeros(1, 1, L, L, device="cuda")]
    want = []
    for m in masks:
        want.append(rmm.rmm_reduced_attn(Q, K, V, causal, 0.5, mask=m))
        torch.cuda.synchronize()
    rmm.binding.poison_outputs(False)                                             # its fills would keep the calls apart
    try:
        got = [rmm.rmm_reduced_attn(Q, K, V, causal, 0.5, mask=masks[i * 2 % 5]) for i in range(60)]
    finally:
        rmm.binding.poison_outputs(True)
    for i, o in enumerate(got):
        assert torch.equal(o, want[i * 2 % 5])
    assert rmm.rmm_status_read() == 0
