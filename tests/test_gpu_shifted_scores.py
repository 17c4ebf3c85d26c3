"""Scores of bf16 rows that start off 16 bytes (score_shift_kernel)."""
import numpy as np
import pytest
import torch

import paper_2608_13426_b200 as rmm
from paper_2608_13426_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,pitch,offset", [
    (100, 64, 65, 0), (449, 65, 65, 0), (777, 1001, 1001, 3), (333, 130, 134, 1), (1000, 4095, 4095, 0), (5000, 71, 79, 5),
    (300, 9001, 9001, 7), (130, 200, 200, 1), (40, 63, 63, 0),      # an aligned pitch off the base; below one block of columns
])
def test_scores_of_rows_off_sixteen_bytes(oracle, M, K, pitch, offset):
    A = synth.heavy_tailed_activations(M, K, seed=M + K)
    # what lies between, before and after the rows must not be counted
    flat = torch.full((offset + M * pitch + 64,), float("nan"), dtype=torch.bfloat16, device="cuda")
    view = flat[offset:offset + M * pitch].view(M, pitch)[:, :K]
    view.copy_(A)
    idx, s, e, _ = rmm.rmm_score_select(view, rho=0.5, want_scores=True, want_energy=True)
    e64, s64 = oracle.score(A)
    # fp32 chains of 16 exact squares, fp64 above, one rounding to fp32
    assert np.allclose(e.cpu().numpy(), e64, rtol=3e-7, atol=0) and np.allclose(s.cpu().numpy(), s64, rtol=3e-7, atol=0)
    assert np.array_equal(idx.cpu().numpy(), oracle.select(e.double().cpu().numpy(), idx.numel())[0])
    assert rmm.rmm_status_read() == 0


def test_scores_of_a_batch_whose_entries_differ_in_alignment(oracle):
    A = synth.heavy_tailed_activations(3 * 201, 333, seed=8).view(3, 201, 333)
    _, _, e, _ = rmm.rmm_score_select(A.cuda(), rho=0.3, want_energy=True)
    for b in range(3):
        assert np.allclose(e[b].cpu().numpy(), oracle.score(A[b])[0], rtol=3e-7, atol=0)
