"""Products of 5 to 256 rows that fetch the kept rows of B themselves (gemm_skinny.cu, the cut tiles of gemm_sm100.cu)."""
import pytest
import torch

import paper_2608_13426_b200 as rmm

pytestmark = pytest.mark.gpu


def ints(shape, seed):
    """Small whole numbers: products and fp32 sums are exact, so the only rounding is that of the output."""
    return torch.randint(-3, 4, shape, generator=torch.Generator().manual_seed(seed)).to(torch.bfloat16)


@pytest.mark.parametrize("M", [5, 8, 9, 24, 31, 32, 33, 100, 128, 129, 256])
@pytest.mark.parametrize("K,N,k", [
    (40, 136, 17),        # less than two groups of kept rows; columns that end inside a tile
    (512, 256, 256),
    (1000, 264, 501),     # k off 8 and 16
    (6000, 1032, 4000),   # few tiles, a long contraction: it is cut
    (3000, 8200, 1111),   # many tiles
])
def test_few_rows_are_exact_on_whole_numbers(M, K, N, k):
    A, B = ints((M, K), 1), ints((K, N), 2)
    idx = torch.randperm(K, generator=torch.Generator().manual_seed(3))[:k].sort().values
    want = A[:, idx].float() @ B[idx].float()
    for dt in (torch.float32, torch.bfloat16):
        Y = rmm.rmm_reduced_gemm(A.cuda(), B.cuda(), idx.int().cuda(), scale=0.5, out_dtype=dt)
        assert torch.equal(Y.cpu(), (0.5 * want).to(dt))
    Y, e = rmm.rmm_reduced_gemm(A.cuda(), B.cuda(), idx.int().cuda(), want_energy=True)
    assert torch.equal(Y.cpu(), want.to(torch.bfloat16))
    assert torch.allclose(e.cpu().double(), Y.cpu().double().square().sum(0), rtol=3e-7)   # fp64 sums rounded to fp32
    assert rmm.rmm_status_read() == 0


@pytest.mark.parametrize("M", [6, 40])
def test_few_rows_batches_strides_and_bad_indices(M):
    A, B = ints((3, M, 700), 4), ints((3, 700, 520), 5)
    lists = torch.stack([torch.randperm(700, generator=torch.Generator().manual_seed(s))[:333].sort().values for s in range(3)])
    wide = torch.zeros(3, 700, 528, dtype=torch.bfloat16).index_copy_(2, torch.arange(520), B).cuda()
    want = torch.stack([A[b][:, lists[b]].float() @ B[b][lists[b]].float() for b in range(3)])
    Y = rmm.rmm_reduced_gemm(A.cuda(), wide[:, :, :520], lists.int().cuda(), out_dtype=torch.float32)
    assert torch.equal(Y.cpu(), want)
    shared = rmm.rmm_reduced_gemm(A.cuda(), B[0].cuda(), lists.int().cuda(), out_dtype=torch.float32)
    assert torch.equal(shared.cpu(), torch.stack([A[b][:, lists[b]].float() @ B[0][lists[b]].float() for b in range(3)]))
    bad = lists[0].clone()
    bad[7], bad[100] = 700, -5                                    # reported, and worth nothing
    keep = torch.ones(333, dtype=torch.bool)
    keep[[7, 100]] = False
    Y = rmm.rmm_reduced_gemm(A[0].cuda(), B[0].cuda(), bad.int().cuda(), out_dtype=torch.float32)
    assert torch.equal(Y.cpu(), A[0][:, lists[0][keep]].float() @ B[0][lists[0][keep]].float())
    assert rmm.rmm_status_read() == 6


@pytest.mark.parametrize("M", [24, 25, 32])
@pytest.mark.parametrize("k", [40, 111, 600])
def test_wide_outputs_by_either_kernel_are_exact_on_whole_numbers(M, k):
    """19208 columns: from 25 rows on whole 128-row tiles take over, for the longer of these contractions."""
    A, B = ints((M, 700), 6), ints((700, 19208), 7)
    idx = torch.randperm(700, generator=torch.Generator().manual_seed(8))[:k].sort().values
    Y = rmm.rmm_reduced_gemm(A.cuda(), B.cuda(), idx.int().cuda(), out_dtype=torch.float32)
    assert torch.equal(Y.cpu(), A[:, idx].float() @ B[idx].float())
    assert rmm.rmm_status_read() == 0
