"""Attention with a few query rows against a long cache (attn_decode.cu)."""
import numpy as np
import pytest
import torch

import paper_2608_13426_b200 as rmm
from paper_2608_13426_b200 import synth
from test_gpu_parity import check_attention, dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [
    # B, Hq, Hkv, Lq, Lk, Dh, causal, rho_d
    (1, 2, 2, 1, 1, 128, True, 0.5),           # one key
    (1, 2, 1, 4, 2, 64, True, 0.5),            # more queries than keys: the first rows see nothing
    (2, 8, 2, 1, 127, 128, True, 0.5),         # one key short of a tile
    (2, 8, 2, 1, 129, 128, False, 1.0),        # one key more
    (3, 4, 4, 2, 1000, 64, True, 0.25),        # a cache that ends inside a warp's 16 keys
    (1, 8, 1, 2, 4099, 128, True, 0.8),        # 16 rows on one kv head, one head over many blocks
    (5, 8, 8, 1, 700, 256, True, 0.5),         # wide heads, several heads per block
    (1, 12, 2, 4, 900, 256, True, 0.3),        # 24 rows: two row tiles, wide heads
    (2, 6, 2, 7, 333, 72, False, 0.5),         # a row tile that ends inside a head, head_dim off 64
    (40, 8, 8, 1, 130, 8, True, 0.5),          # more heads than blocks, the smallest head_dim
    (1, 4, 2, 16, 600, 128, True, 0.5),        # the longest step of this form
])
def test_decode_attention_matches_the_oracle(oracle, shape):
    B, Hq, Hkv, Lq, Lk, Dh, causal, rho_d = shape
    assert check_attention(oracle, B, Hq, Hkv, Lq, Lk, Dh, causal, rho_d, 1.0, seed=130 + Lk % 11, n_outlier=min(4, Dh // 4))
    assert rmm.rmm_status_read() == 0


def test_decode_attention_ties_and_strides(oracle):
    """Equal feature scores go to the lower index; K rows may be strided, O and the index list match the general form."""
    Q, K, V = synth.attention_qkv(2, 4, 2, 1, 300, 64, seed=9)
    Q = Q.sign() * 2.0
    wide = torch.zeros(2, 300, 2, 64 + 8, dtype=torch.bfloat16)
    wide[..., :64] = K.transpose(1, 2)
    O, feat, _ = rmm.rmm_reduced_attn(dev(Q), dev(wide)[..., :64].transpose(1, 2), dev(V), True, 0.5, want_idx=True)
    assert torch.equal(feat.cpu(), torch.arange(32, dtype=torch.int32).expand(2, 4, 32))
    want = oracle.attn(Q, K, V, True, 0.5, 1.0, idx_feat=feat.cpu().numpy())[0]
    assert np.linalg.norm(O.float().cpu().numpy() - want) <= 1e-2 * np.linalg.norm(want)


def test_decode_attention_ignores_what_dropped_features_hold(oracle):
    Q, K, V = synth.attention_qkv(1, 4, 2, 2, 500, 128, seed=15)
    Q[..., 100] = 0.0                           # the lowest score of every head: never kept
    want, feat, _ = rmm.rmm_reduced_attn(dev(Q), dev(K), dev(V), True, 0.5, want_idx=True)
    assert not (feat == 100).any()
    K[:, :, ::7, 100] = float("inf")
    K[:, :, 3, 100] = float("nan")
    got = rmm.rmm_reduced_attn(dev(Q), dev(K), dev(V), True, 0.5)
    assert torch.isfinite(got.float()).all()
    # the steps that hold such a key sum their products in another order: fp32 rounding before the bf16 rounding of P
    assert ((got.float() - want.float()).norm() / want.float().norm()).item() <= 4e-3


@pytest.mark.parametrize("B, Hkv, Lk", [(40, 8, 60), (1, 1, 6000)])   # whole jobs per block; one job over many blocks
def test_decode_attention_shows_a_nan(B, Hkv, Lk):
    """A NaN (or an infinity's inf - inf) among a row's logits makes the row NaN, wherever its key lies; rows that see no
    key stay zero and the other heads are untouched."""
    Q, K, V = synth.attention_qkv(B, Hkv, Hkv, 2, Lk, 64, seed=16)
    want = rmm.rmm_reduced_attn(dev(Q), dev(K), dev(V), True, 1.0)
    for key in (0, Lk // 2, Lk - 2):
        for bad in (float("nan"), float("inf")):
            Kb, Qb = K.clone(), Q.clone()
            Kb[0, 0, key, 5], Qb[0, 0, :, 5] = bad, 1.0
            got = rmm.rmm_reduced_attn(dev(Qb), dev(Kb), dev(V), True, 1.0)
            assert torch.isnan(got[0, 0]).all(), (key, bad)
            assert torch.equal(got.flatten(0, 1)[1:], want.flatten(0, 1)[1:])
    Qb = Q.clone()
    Qb[0, 0, 1, 7] = float("nan")                 # every logit of this row
    got = rmm.rmm_reduced_attn(dev(Qb), dev(K), dev(V), True, 1.0)
    assert torch.isnan(got[0, 0, 1]).all() and torch.isfinite(got[0, 0, 0].float()).all()
    Qb = Q.repeat(1, 1, 2, 1)                     # four queries on two keys: the first two see nothing
    Qb[0, 0] = float("nan")
    got = rmm.rmm_reduced_attn(dev(Qb), dev(K[:, :, :2]), dev(V[:, :, :2]), True, 1.0)
    assert torch.count_nonzero(got[:, :, :2]) == 0 and torch.isnan(got[0, 0, 2:]).all()
