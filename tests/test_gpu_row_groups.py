"""Fused attention by blocks of one and of two groups of 128 rows (attn_fused.cu: one where such blocks do not outnumber the SMs)."""
import pytest
import torch

import paper_2608_13426_b200 as rmm
from test_gpu_masked_tiles import padded
from test_gpu_parity import check_attention

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rho_t, masked", [(1.0, False), (0.5, False), (1.0, True)])
@pytest.mark.parametrize("B, Hq, Hkv, Lq, Lk, Dh, causal", [
    (1, 74, 37, 256, 256, 64, True),     # 148 blocks of 128 rows, each its own
    (1, 75, 25, 129, 129, 64, True),     # 150: two groups, the second of one row
    (1, 74, 74, 130, 385, 64, True),     # a chunk of a longer prompt
    (2, 4, 2, 17, 300, 128, False),      # one short block a head
    (1, 4, 4, 500, 260, 128, True),      # rows that see nothing
    (1, 2, 1, 900, 900, 256, False),     # two passes over the columns
    (1, 50, 25, 500, 500, 64, True),     # 200 blocks of 128 rows: two rounds of one group
    (1, 60, 20, 300, 700, 64, True),     # 180, all of them long: two groups
    (2, 50, 50, 140, 100, 64, True),     # 200, rows that see nothing among them
])
def test_one_and_two_groups(oracle, B, Hq, Hkv, Lq, Lk, Dh, causal, rho_t, masked):
    mask = padded(B, Lq, Lk, [Lk, 128][:B] if B > 1 else [Lk - 30]) if masked else None
    assert check_attention(oracle, B, Hq, Hkv, Lq, Lk, Dh, causal, 0.5, rho_t, seed=Lq, mask=mask)
    assert rmm.rmm_status_read() == 0
