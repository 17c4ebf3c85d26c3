"""Additive masks whose 128 x 128 tiles are skipped, left alone or added (attn_fused.cu)."""
import numpy as np
import pytest
import torch

import paper_2608_13426_b200 as rmm
from paper_2608_13426_b200 import synth
from test_gpu_parity import check_attention, dev

pytestmark = pytest.mark.gpu
HIDE = -float("inf")


def padded(B, Lq, Lk, lengths, value=HIDE):
    M = torch.zeros(B, 1, Lq, Lk)
    for b, n in enumerate(lengths):
        M[b, :, :, n:] = value
    return M


def blocks(L, size):
    """Block-diagonal: whole tiles hidden between visible ones, left and right of the diagonal."""
    i = torch.arange(L) // size
    return torch.where(i[:, None] == i[None, :], 0.0, HIDE)


def sliding(L, width):
    i = torch.arange(L)
    return torch.where((i[:, None] - i[None, :]).abs() <= width, 0.0, HIDE)


CASES = {
    # B, Hq, Hkv, Lq, Lk, Dh, causal, mask
    "padding per sequence, shared by heads": (2, 4, 2, 300, 300, 128, True, padded(2, 300, 300, [300, 129])),
    "rows of odd length": (2, 4, 2, 261, 261, 64, True, padded(2, 261, 261, [131, 256])),
    "no value is zero or hides": (1, 2, 2, 257, 263, 64, False, torch.randn(1, 1, 257, 263, generator=torch.Generator().manual_seed(1))),
    "an odd pitch per head": (2, 2, 1, 140, 275, 128, False, torch.randn(2, 2, 140, 275, generator=torch.Generator().manual_seed(2)).round()),
    "one row for all queries": (2, 4, 4, 400, 385, 128, False, padded(2, 1, 385, [128, 300])),
    "the lowest finite value": (2, 4, 2, 300, 300, 128, True, padded(2, 300, 300, [140, 256], torch.finfo(torch.float32).min)),
    "first sequence sees nothing": (2, 4, 2, 300, 300, 128, False, padded(2, 300, 300, [0, 200])),
    "blocks": (1, 4, 2, 1280, 1280, 128, False, blocks(1280, 320)),
    "window": (1, 2, 1, 1500, 1500, 64, True, sliding(1500, 150)),
    "wide heads": (1, 2, 1, 700, 700, 256, True, sliding(700, 200)),
    "all zero": (1, 2, 1, 513, 513, 128, False, torch.zeros(513, 513)),
    "every second key block, over more than eight tiles": (1, 2, 2, 256, 2300, 64, False,
                                                             torch.where((torch.arange(2300) // 128) % 2 == 1, 0.0, HIDE).expand(256, 2300)),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_masked_attention_by_tiles(oracle, name):
    B, Hq, Hkv, Lq, Lk, Dh, causal, M = CASES[name]
    M = M.contiguous()
    mask = M if M.dim() == 4 else M[None, None]
    assert check_attention_or_zero(oracle, B, Hq, Hkv, Lq, Lk, Dh, causal, mask)
    assert rmm.rmm_status_read() == 0


def check_attention_or_zero(oracle, B, Hq, Hkv, Lq, Lk, Dh, causal, mask):
    if not (mask[0] < -1e30).all():
        low = mask.clone()
        low[low < -1e30] = HIDE          # the lowest finite value hides a key as -inf does
        Q, K, V = synth.attention_qkv(B, Hq, Hkv, Lq, Lk, Dh, seed=171)
        O, feat, _ = rmm.rmm_reduced_attn(dev(Q), dev(K), dev(V), causal, 0.5, 1.0, want_idx=True, mask=dev(mask))
        want = oracle.attn(Q, K, V, causal, 0.5, 1.0, idx_feat=feat.cpu().numpy(), mask=low.numpy().astype(np.float64))[0]
        got = O.float().cpu().numpy()
        assert np.isfinite(got).all()
        return bool((np.linalg.norm(got - want, axis=(2, 3)) <= 1e-2 * np.linalg.norm(want, axis=(2, 3))).all())
    Q, K, V = synth.attention_qkv(B, Hq, Hkv, Lq, Lk, Dh, seed=171)
    O = rmm.rmm_reduced_attn(dev(Q), dev(K), dev(V), causal, 0.5, 1.0, mask=dev(mask))
    alone = rmm.rmm_reduced_attn(dev(Q[1:]), dev(K[1:]), dev(V[1:]), causal, 0.5, 1.0, mask=dev(mask[1:]))
    return torch.count_nonzero(O[0]) == 0 and torch.equal(O[1:], alone)


def test_masked_attention_folds_only_even_sequences(oracle):
    """Sequences that are not evenly spaced in memory run one by one against their own planes of the mask."""
    M = padded(3, 200, 200, [200, 90, 140])
    Q, K, V = synth.attention_qkv(3, 4, 2, 200, 200, 64, seed=172)
    wide = torch.zeros(3, 5, 200, 64, dtype=torch.bfloat16)
    wide[:, :4] = Q
    a = rmm.rmm_reduced_attn(dev(wide)[:, :4], dev(K), dev(V), True, 0.5, 1.0, mask=dev(M))
    b = rmm.rmm_reduced_attn(dev(Q), dev(K), dev(V), True, 0.5, 1.0, mask=dev(M))
    assert torch.equal(a, b)
    assert check_attention(oracle, 3, 4, 2, 200, 200, 64, True, 0.5, 1.0, seed=172, mask=M)


@pytest.mark.parametrize("L", [300, 301, 2052])                 # rows of whole vectors, rows of odd length, more than eight tiles
@pytest.mark.parametrize("value", [torch.finfo(torch.float32).min, -1e30, -1e9, -1e4])
def test_rows_that_see_nothing_but_large_finite_values(oracle, L, value):
    """A finite mask value hides no key: rows that hold nothing else weigh their keys by the sums S~ + M as fp32 has them,
    and rows with one ordinary key are as if -inf stood there.  Left padding: rows before n see padding keys only."""
    n, B, Hq, Dh = 140, 2, 4, 64
    M = torch.zeros(B, 1, L, L)
    M[1, :, :, :n] = value
    Q, K, V = synth.attention_qkv(B, Hq, 2, L, L, Dh, seed=173)
    O, feat, _ = rmm.rmm_reduced_attn(dev(Q), dev(K), dev(V), True, 0.5, 1.0, want_idx=True, mask=dev(M))
    low = M.double()
    if value < -1e8:
        low[low < 0] = HIDE
    want = oracle.attn(Q, K, V, True, 0.5, 1.0, idx_feat=feat.cpu().numpy(), mask=low.numpy())[0]
    if value < -1e10:                                            # S~ is lost next to the mask: equal weights
        mean = (torch.cumsum(V[1].double(), 1) / torch.arange(1, L + 1)[:, None]).numpy()
        want[1, :, :n] = np.repeat(mean, 2, axis=0)[:, :n]
    got = O.float().cpu().numpy()
    assert np.isfinite(got).all()
    rows = np.linalg.norm(got - want, axis=3) / np.maximum(np.linalg.norm(want, axis=3), 1e-30)
    if -1e10 < value < -1e8:                                     # S~ + M in steps of 64: not compared
        rows[1, :, :n] = 0.0
    # one rounding of P and one of O, 2^-9 each, over the row's norm; S~ + M in steps of 2^-10 at -1e4
    assert rows.max() <= 2.5e-2, np.unravel_index(rows.argmax(), rows.shape)
    assert rmm.rmm_status_read() == 0


def test_low_tiles_are_skipped_only_where_every_row_has_another_key(oracle):
    """One row of a block keeps its low values while the other rows' tiles could go."""
    L, low = 384, torch.finfo(torch.float32).min
    M = torch.zeros(1, 1, L, L)
    M[..., :128] = low
    M[0, 0, 200] = low                                           # the only row of its block without an ordinary key
    M[0, 0, 300, 1:] = low                                       # its ordinary key: outside the evenly spread look
    M[0, 0, 300, 0] = low
    M[0, 0, 300, 131] = 0.5
    Q, K, V = synth.attention_qkv(1, 2, 1, L, L, 128, seed=174)
    O, feat, _ = rmm.rmm_reduced_attn(dev(Q), dev(K), dev(V), False, 0.5, 1.0, want_idx=True, mask=dev(M))
    hide = M.double()
    hide[hide < -1e30] = HIDE
    want = oracle.attn(Q, K, V, False, 0.5, 1.0, idx_feat=feat.cpu().numpy(), mask=hide.numpy())[0]
    want[0, :, 200] = V[0, 0].double().mean(0).numpy()
    got = O.float().cpu().numpy()
    assert (np.linalg.norm(got - want, axis=3) <= 2.5e-2 * np.linalg.norm(want, axis=3)).all()


def test_a_mask_over_more_row_blocks_than_a_grid_has_rows():
    """65536 blocks of 128 queries; one mask row stands for all of them.  Every row's result is its own."""
    Lq, Lk = 65536 * 128 + 5, 200
    g = torch.Generator(device="cuda").manual_seed(175)
    Q = torch.randn(1, 1, Lq, 8, generator=g, device="cuda").to(torch.bfloat16)
    K, V = (torch.randn(1, 1, Lk, 8, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    M = torch.zeros(1, 1, 1, Lk, device="cuda")
    M[..., 130:] = HIDE
    M[..., 7] = 1.5
    O = rmm.rmm_reduced_attn(Q, K, V, False, 1.0, 1.0, mask=M)
    for lo, hi in ((0, 300), (Lq // 2, Lq // 2 + 300), (Lq - 261, Lq)):
        part = rmm.rmm_reduced_attn(Q[:, :, lo:hi], K, V, False, 1.0, 1.0, mask=M)
        assert ((O[:, :, lo:hi].float() - part.float()).abs().max() <= 2.0 ** -7 * part.float().abs().max()).item()
    assert rmm.rmm_status_read() == 0
