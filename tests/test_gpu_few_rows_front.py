"""Scores, selection and gather of a few rows in one launch (select_cluster_kernel on a matrix)."""
import numpy as np
import pytest
import torch

import paper_2608_13426_b200 as rmm
from paper_2608_13426_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [1, 3, 5, 8, 9, 32, 33])
@pytest.mark.parametrize("K", [1, 9, 500, 1024, 1025, 4096, 4097, 8192, 8193, 16385, 32769, 65536, 65537])
def test_few_rows_scores_and_sets(oracle, M, K):
    A = synth.heavy_tailed_activations(M, K, seed=M + K)
    idx, s, e, kept = rmm.rmm_score_select(A.cuda(), rho=0.37, want_scores=True, want_energy=True, want_retained=True)
    e64, s64 = oracle.score(A)
    want = e64.astype(np.float32)
    assert np.allclose(e.cpu().numpy(), want, rtol=1.2e-7, atol=0) and np.allclose(s.cpu().numpy(), s64, rtol=1.2e-7, atol=0)
    sel, _ = oracle.select(e.double().cpu().numpy(), idx.numel())            # the set of the energies as returned, ties included
    assert np.array_equal(idx.cpu().numpy(), sel)
    assert abs(float(kept) - e64[sel].sum() / e64.sum()) <= 2e-6


def test_few_rows_batches_and_odd_pitch(oracle):
    A = synth.heavy_tailed_activations(3 * 7, 1003, seed=5).view(3, 7, 1003)   # rows start off 16 bytes
    idx, _, e, _ = rmm.rmm_score_select(A.cuda(), k=400, want_energy=True)
    for b in range(3):
        e64, _ = oracle.score(A[b])
        assert np.allclose(e[b].cpu().numpy(), e64, rtol=1.2e-7, atol=0)
        assert np.array_equal(idx[b].cpu().numpy(), oracle.select(e[b].double().cpu().numpy(), 400)[0])


@pytest.mark.parametrize("M,K,N,k", [(5, 1001, 264, 333), (24, 8192, 512, 2048), (33, 9000, 136, 4001), (32, 512, 256, 256), (32, 20000, 1032, 77)])
def test_whole_product_of_few_rows(M, K, N, k):
    """The gathered columns come from the selecting kernel: same result as from the list it returned."""
    A, B = synth.mlp_product(M, K, N, seed=K)
    A, B = A.cuda(), B.cuda()
    Y, idx = rmm.rmm_product(A, B, k=k)
    assert torch.equal(idx, rmm.rmm_score_select(A, k=k)[0])
    assert torch.equal(Y, rmm.rmm_reduced_gemm(A, B, idx))
    wide = torch.zeros(M, K + 8, dtype=torch.bfloat16, device="cuda")[:, :K].copy_(A)
    assert torch.equal(rmm.rmm_product(wide, B, k=k)[0], Y)
    assert rmm.rmm_status_read() == 0
