"""Attention outputs that lie anywhere: rows and heads in either order, backwards, strides of axes of one (the C entry point)."""
import ctypes

import pytest
import torch

import paper_2608_13426_b200 as rmm
from paper_2608_13426_b200 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rho_t", [1.0, 0.5])
@pytest.mark.parametrize("Hq, Lq, Lk, order, signs", [
    (4, 150, 150, "hl", (1, 1)), (4, 150, 150, "lh", (1, 1)),       # [head, row] and [row, head]
    (4, 150, 150, "hl", (1, -1)), (4, 150, 150, "lh", (-1, 1)), (4, 300, 200, "hl", (-1, -1)),
    (4, 1, 90, "hl", (1, 0)), (1, 140, 140, "hl", (0, 1)), (1, 1, 77, "hl", (0, 0)),
])
def test_any_strides(Hq, Lq, Lk, order, signs, rho_t):
    Dh = 64
    Q, K, V = synth.attention_qkv(1, Hq, Hq, Lq, Lk, Dh, seed=Lq, device="cuda")
    want = rmm.rmm_reduced_attn(Q, K, V, True, 0.5, rho_t)
    sh, sr = (Lq * (Dh + 8), Dh + 8) if order == "hl" else (Dh + 8, Hq * (Dh + 8))
    buf = torch.full((Hq * Lq * (Dh + 8),), float("nan"), dtype=torch.bfloat16, device="cuda")
    first = sum((n - 1) * s for n, s, sign in ((Hq, sh, signs[0]), (Lq, sr, signs[1])) if sign < 0)
    s3 = lambda *s: (ctypes.c_int64 * 3)(*s)  # noqa: E731
    d = binding.rmm_attn_desc_t(1, Hq, Hq, Lq, Lk, Dh, 1, 0.5, rho_t, s3(*Q.stride()[:3]), s3(*K.stride()[:3]), s3(*V.stride()[:3]),
                                s3(0, signs[0] * sh, signs[1] * sr), None, s3(0, 0, 0))
    need = binding.lib().rmm_reduced_attn_workspace_bytes(d)
    ws = binding.workspace(need, Q.device)
    p, nb = binding._ws_ptr(ws)
    binding._check(binding.lib().rmm_reduced_attn(d, Q.data_ptr(), K.data_ptr(), V.data_ptr(), buf.data_ptr() + 2 * first, None, None, p, nb,
                                                  binding._stream()))
    at = (torch.arange(Hq)[:, None] * signs[0] * sh + torch.arange(Lq) * signs[1] * sr + first)[..., None] + torch.arange(Dh)
    got = buf[at.cuda()]
    assert torch.equal(got, want[0])
    buf[at.cuda()] = float("nan")
    assert torch.isnan(buf).all()                                   # nothing beside the outputs was written
    assert rmm.rmm_status_read() == 0
