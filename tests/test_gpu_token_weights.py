"""Token-reduced attention: weights partly by ex2_fma, O through tile stores (attn_fused.cu, GATHERED and STATS)."""
import math

import numpy as np
import pytest
import torch

import paper_2608_13426_b200 as rmm
from paper_2608_13426_b200 import synth
from test_gpu_parity import check_attention

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B, Hq, Hkv, Lq, Lk, Dh, causal", [
    (1, 1, 1, 17, 40, 64, False), (1, 3, 1, 33, 129, 72, True), (2, 2, 2, 161, 161, 128, True),   # rows and columns that tiles clip
    (1, 2, 1, 96, 700, 256, False),                                                               # two passes over the columns
    (1, 80, 8, 200, 260, 64, True),                                                               # blocks of two groups
])
@pytest.mark.parametrize("rho_t", [0.3, 0.9])
def test_outputs_of_odd_sizes(oracle, B, Hq, Hkv, Lq, Lk, Dh, causal, rho_t):
    assert check_attention(oracle, B, Hq, Hkv, Lq, Lk, Dh, causal, 0.5, rho_t, seed=Lk)
    assert rmm.rmm_status_read() == 0


def test_weights_over_the_whole_range():
    """Logits from far below to far above, so that weights run from 1 to nothing, and a row that holds a NaN."""
    g = torch.Generator().manual_seed(5)
    Lq, Lk, Dh = 256, 512, 64
    Q, K, V = (torch.randn(1, 1, n, Dh, generator=g) for n in (Lq, Lk, Lk))
    Q[..., 0] = 8.0
    K[..., 0] = torch.linspace(-120, 40, Lk) / math.log2(math.e)
    Q, K, V = Q.bfloat16(), K.bfloat16(), V.bfloat16()
    Q[0, 0, 7, 3] = float("nan")
    O, _, tok = rmm.rmm_reduced_attn(Q.cuda(), K.cuda(), V.cuda(), False, 1.0, 0.75, want_idx=True)
    P = torch.softmax(Q.double() @ K.double().mT / math.sqrt(Dh), -1).bfloat16().double()
    t = tok.cpu().long()[0, 0]
    want = P[0, 0][:, t] @ V.double()[0, 0][t]
    got = O.cpu().double()[0, 0]
    assert torch.isnan(got[7]).all()
    rest = torch.arange(Lq) != 7
    # weights rounded at a tie and the output: 2^-8 over the row's norm
    assert ((got - want).norm(dim=1) <= 2.0 ** -7 * want.norm(dim=1))[rest].all()
    assert rmm.rmm_status_read() == 0
