"""Scores inside the whole product of small operands (small.cu): the index set is the one that rmm_score_select gives."""
import pytest
import torch

import paper_2608_13426_b200 as rmm

pytestmark = pytest.mark.gpu

SHAPES = [(5, 8), (16, 511), (24, 1000), (16, 2047), (32, 512), (33, 513), (48, 1024), (64, 512), (64, 640)]


@pytest.mark.parametrize("M, K", SHAPES)
def test_columns_of_the_same_values_in_another_order_tie(M, K):
    """Every column holds the same heavy-tailed values: sums in fp64 are exact here, so all keys are equal and the lowest indices
    stay; sums in fp32 depend on the order."""
    g = torch.Generator().manual_seed(M + K)
    values = ((1 + torch.randint(0, 128, (M,), generator=g) / 128) * 2.0 ** torch.randint(-5, 4, (M,), generator=g)).bfloat16()
    A = torch.zeros(M, (K + 7) // 8 * 8, dtype=torch.bfloat16)
    for c in range(K):
        A[:, c] = values[torch.randperm(M, generator=g)]
    A, B, k = A.cuda()[:, :K], torch.ones(K, 256, device="cuda", dtype=torch.bfloat16), (K + 1) // 2
    first = torch.arange(k, dtype=torch.int32, device="cuda")
    n0 = rmm.rmm_launch_count()
    idx = rmm.rmm_product(A, B, k=k)[1]
    assert rmm.rmm_launch_count() - n0 == 1
    assert torch.equal(idx, first) and torch.equal(rmm.rmm_score_select(A, k=k)[0], first)


@pytest.mark.parametrize("M, K", SHAPES)
def test_the_index_set_is_that_of_the_score_pass(M, K):
    """Column energies a rounding of fp32 apart: the keys have to be the same numbers, not only nearly so."""
    g = torch.Generator().manual_seed(7 * M + K)
    one = torch.randn(M, generator=g) * 8.0 ** torch.rand(M, generator=g)
    A = torch.zeros(M, (K + 7) // 8 * 8, dtype=torch.bfloat16)
    for c in range(K):
        A[:, c] = one[torch.randperm(M, generator=g)]
        A[c % M, c] += (torch.rand(1, generator=g) * 2.0 ** -6).bfloat16()[0]     # about one unit in the last place of the sum
    A, B = A.cuda()[:, :K], torch.ones(K, 64, device="cuda", dtype=torch.bfloat16)
    for k in sorted({1, K // 3, K // 2, K - 1}):
        assert torch.equal(rmm.rmm_product(A, B, k=k)[1], rmm.rmm_score_select(A, k=k)[0]), k


@pytest.mark.parametrize("M, K", SHAPES)
def test_the_kept_share_changes_nothing_else(M, K):
    """Asking for the kept share of the energies leaves Y and the list as they are, and so does the list when it is given."""
    g = torch.Generator().manual_seed(M * K)
    wide = (K + 7) // 8 * 8
    A, B = torch.randn(M, wide, generator=g).bfloat16().cuda()[:, :K], torch.randn(K, 264, generator=g).bfloat16().cuda()
    for k in sorted({1, K // 2, K}):
        Y, idx = rmm.rmm_product(A, B, k=k, out=torch.empty(M, 264, device="cuda"))
        Y2, idx2, kept = rmm.rmm_product(A, B, k=k, out=torch.empty(M, 264, device="cuda"), want_retained=True)
        assert torch.equal(Y, Y2) and torch.equal(idx, idx2)
        assert torch.equal(Y, rmm.rmm_reduced_gemm(A, B, idx, out_dtype=torch.float32))
        want_idx, _, energy, want = rmm.rmm_score_select(A, k=k, want_energy=True, want_retained=True)
        assert torch.equal(idx, want_idx) and abs(float(kept) - float(want)) <= 2.0 ** -23
        share = float(energy[idx.long()].double().sum() / energy.double().sum())
        assert abs(float(kept) - share) <= 2.0 ** -23          # fp64 sums, rounded once to fp32
    assert rmm.rmm_status_read() == 0
