"""One-pass attention whose row maxima move from tile to tile: the reference that weights are taken against is renewed, or
lets them grow to 2^40 (attn_fused.cu), whatever the size of the values that they weigh."""
import math

import pytest
import torch

import paper_2608_13426_b200 as rmm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("peak", [0, 30])        # one key of the highest tile stands out by so much
@pytest.mark.parametrize("v_scale", [1.0, 1e-20, 1e20, 1e-26, 1e-33])
@pytest.mark.parametrize("levels", [
    [0, 35, 70, 79],            # within the margin: never renewed
    [0, 79, 81, 160, 162],      # just below and above it
    [0, 300, 0, -300, 500],     # far beyond, and back
    [-400, -400, 40, 39.5, 0],  # low first
    [0, 2, 4, 6, 8],            # a row is spread over several tiles
])
def test_row_maxima_that_grow(levels, v_scale, peak):
    g = torch.Generator().manual_seed(len(levels))
    Lq, Lk, Dh = 300, 128 * len(levels) - 5, 64
    Q, K, V = (torch.randn(1, 2, n, Dh, generator=g) for n in (Lq, Lk, Lk))
    # logits: level of the tile in powers of two, for most rows a little more or less than the next row's
    Q[..., 0] = 8.0 + torch.arange(Lq) % 7 / 16
    for t, x in enumerate(levels):
        K[:, :, 128 * t:128 * (t + 1), 0] = x / math.log2(math.e)
    K[:, :, 128 * levels.index(max(levels)) + 77, 0] += peak / math.log2(math.e)
    Q, K, V = Q.bfloat16(), K.bfloat16(), (V * v_scale).bfloat16()
    O = rmm.rmm_reduced_attn(Q.cuda(), K.cuda(), V.cuda(), False, 1.0).cpu().double()
    P = torch.softmax(Q.double() @ K.double().mT / math.sqrt(Dh), -1)
    want = P @ V.double()
    assert torch.isfinite(O).all()
    # a rounding of P and one of O, 2^-9 each, over the row's norm
    assert ((O - want).norm(dim=-1) <= 2.5e-2 * want.norm(dim=-1)).all()
    # a row that one key dominates gets that key's value: the rounding of O alone
    alone = P.max(-1).values > 1 - 1e-5
    assert peak == 0 or alone.double().mean() > 0.9
    assert ((O - want).norm(dim=-1) <= 2.0 ** -8 * want.norm(dim=-1))[alone].all()
    assert rmm.rmm_status_read() == 0
