"""Products of 5 to 256 rows that fetch the kept rows of B themselves (gemm_skinny.cu, the cut tiles of gemm_sm100.cu)."""
import numpy as np
import pytest
import torch

import paper_2608_13426_b200 as rmm
from paper_2608_13426_b200 import binding, synth

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


@pytest.mark.parametrize("M, K, N, k, apart", [
    (64, 1024, 28672, 512, False),     # tiles enough for the GPU: the epilogue leaves the energies
    (200, 512, 264, 100, False),       # two row tiles, a last tile of eight columns, a ragged k-block
    (24, 1024, 14336, 512, False),     # few rows, as above
    (24, 4096, 2048, 2048, True),      # the few-row kernel and a pass over Y
    (48, 8192, 2048, 4096, True),      # cut tiles and a pass over Y
])
def test_scored_products_of_few_rows_keep_their_energies_where_tiles_are_whole(oracle, M, K, N, k, apart):
    A, B = synth.mlp_product(M, K, N, seed=M + k)
    idx = torch.randperm(K, generator=torch.Generator().manual_seed(k))[:k].sort().values.int()
    Ad, Bd, ix = A.cuda(), B.cuda(), idx.cuda()
    rmm.rmm_reduced_gemm(Ad, Bd, ix, want_energy=True)
    timer = binding.KernelTimer(16)
    with timer:
        Y, e = rmm.rmm_reduced_gemm(Ad, Bd, ix, want_energy=True)
    assert any("score" in name for name, _ in timer.times_ms()) == apart
    cols = np.r_[0:min(N, 300), N - 40:N]
    want = oracle.reduced_gemm(A, B[:, cols].contiguous(), idx.numpy())
    got = Y.float().cpu().numpy()
    assert np.linalg.norm(got[:, cols] - want) <= 1e-2 * np.linalg.norm(want)
    # exact squares, fp32 chains of 16: 16 roundings of 2^-24 at most
    assert np.allclose(e.cpu().numpy(), (got.astype(np.float64) ** 2).sum(0), rtol=1e-6, atol=0)
    assert rmm.rmm_status_read() == 0
