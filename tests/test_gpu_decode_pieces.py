"""Decode attention cut into pieces: few of them meet in the last block of a job, many in a second launch (attn_decode.cu)."""
import pytest
import torch

import paper_2608_13426_b200 as rmm
from paper_2608_13426_b200 import synth
from test_gpu_parity import check_attention

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B, Hq, Hkv, Lq, Lk, Dh, launches", [
    (8, 32, 8, 1, 1000, 128, 1),     # four pieces of four rows
    (4, 16, 8, 1, 1500, 64, 1),      # eight pieces of two rows, half a warp per row
    (8, 24, 8, 1, 1000, 128, 1),     # three rows: a warp without one
    (9, 2, 2, 1, 2000, 64, 1),       # sixteen pieces of one row, shared out among the warps
    (20, 4, 2, 1, 1100, 256, 1),     # two rows of wide heads
    (20, 4, 2, 4, 4000, 256, 1),     # long pieces of eight rows, wide heads
    (20, 4, 2, 4, 1100, 256, 2),     # short ones
    (10, 4, 2, 4, 1100, 256, 2),
    (30, 16, 2, 2, 900, 128, 2),     # sixteen rows a block
    (4, 4, 4, 1, 6092, 128, 2),      # pieces of six tiles
    (4, 4, 4, 1, 6092, 64, 1),
    (2, 4, 2, 1, 3000, 128, 2),      # one row per warp, more than 32 pieces
    (1, 32, 2, 1, 4000, 64, 2),      # sixteen rows, many pieces
])
def test_pieces_meet(oracle, B, Hq, Hkv, Lq, Lk, Dh, launches):
    assert check_attention(oracle, B, Hq, Hkv, Lq, Lk, Dh, True, 0.5, 1.0, seed=Lk, n_outlier=4)
    Q, K, V = (t.cuda() for t in synth.attention_qkv(B, Hq, Hkv, Lq, Lk, Dh, seed=Lk + 1))
    first = rmm.rmm_reduced_attn(Q, K, V, True, 0.5)
    n0 = rmm.rmm_launch_count()
    again = rmm.rmm_reduced_attn(Q, K, V, True, 0.5)         # pieces are added in order, and the counters are back at zero
    assert rmm.rmm_launch_count() - n0 == launches
    assert torch.equal(first, again) and rmm.rmm_status_read() == 0
