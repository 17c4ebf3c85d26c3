"""Whole products of small operands in one launch (small.cu), and the same kernel on a given index list."""
import numpy as np
import pytest
import torch

import paper_2608_13426_b200 as rmm

pytestmark = pytest.mark.gpu


def ints(shape, seed):
    """Small whole numbers: products and fp32 sums are exact, so any order of summation gives the same."""
    return torch.randint(-4, 5, shape, generator=torch.Generator().manual_seed(seed)).float()


# rows around a 16-row tile and the largest count; axes around one, two and four keys a thread, odd ones in wider rows; columns of
# one vector, of a partial last block, and past the width of one 16-column block per SM
@pytest.mark.parametrize("M, K, N, k", [(5, 8, 8, 1), (15, 511, 40, 255), (16, 512, 264, 256), (17, 513, 24, 513), (64, 512, 256, 256), (33, 777, 2384, 17),
                                        (48, 1024, 1000, 1023), (5, 1025, 4096, 700), (16, 2048, 136, 1024), (6, 2047, 2048, 16)])
def test_small_product_is_exact_on_whole_numbers(oracle, M, K, N, k):
    A, B = ints((M, K), M + K), ints((K, N), N + 1)
    wide = torch.full((M, (K + 7) // 8 * 8 + 8), float("nan"), dtype=torch.bfloat16, device="cuda")   # what lies beside a row is not read
    wide[:, :K] = A.to(torch.bfloat16)
    Ad, Bd = wide[:, :K], B.to(torch.bfloat16).cuda()
    n0 = rmm.rmm_launch_count()
    out = torch.empty(M, N, dtype=torch.float32, device="cuda")
    Y, idx = rmm.rmm_product(Ad, Bd, k=k, scale=0.5, out=out)
    assert rmm.rmm_launch_count() - n0 == 1
    e64, _ = oracle.score(A.to(torch.bfloat16))
    assert np.array_equal(idx.cpu().numpy(), oracle.select(e64, k)[0])     # whole energies: equal keys included
    kept = idx.cpu().long()
    want = 0.5 * (A[:, kept].double() @ B[kept].double()).float()
    assert torch.equal(Y.cpu(), want)
    assert torch.equal(rmm.rmm_reduced_gemm(Ad, Bd, idx, scale=0.5).cpu(), want.to(torch.bfloat16))
    # a list of the caller's: any order, repeats; an index out of range is reported and contributes nothing
    own = torch.randint(0, K, (k,), generator=torch.Generator().manual_seed(k), dtype=torch.int32)
    Yo = rmm.rmm_reduced_gemm(Ad, Bd, own.cuda(), out_dtype=torch.float32)
    assert torch.equal(Yo.cpu(), (A[:, own.long()].double() @ B[own.long()].double()).float())
    assert rmm.rmm_status_read() == 0
    own[0] = K
    Yb = rmm.rmm_reduced_gemm(Ad, Bd, own.cuda(), out_dtype=torch.float32)
    assert torch.equal(Yb.cpu(), (A[:, own[1:].long()].double() @ B[own[1:].long()].double()).float())
    assert rmm.rmm_status_read() == 6 and rmm.rmm_status_read() == 0


def test_dropped_rows_and_columns_weigh_nothing():
    """NaN and infinities in rows of B that are not kept leave the output alone; kept ones come through."""
    A, B = torch.ones(8, 256, device="cuda", dtype=torch.bfloat16), torch.ones(256, 64, device="cuda", dtype=torch.bfloat16)
    A[:, 100:] = 0.5
    B[100:] = float("nan")
    Y, idx = rmm.rmm_product(A, B, k=100)
    assert torch.equal(idx.cpu(), torch.arange(100, dtype=torch.int32)) and torch.equal(Y, torch.full_like(Y, 100.0))
    B[7, 3] = float("inf")
    Y = rmm.rmm_product(A, B, k=100)[0]
    assert torch.isinf(Y[:, 3]).all() and torch.equal(Y[:, 4:], torch.full_like(Y[:, 4:], 100.0))


def test_scored_output_of_a_small_product_is_the_plain_one():
    A, B = torch.randn(40, 640, device="cuda").bfloat16(), torch.randn(640, 512, device="cuda").bfloat16()
    idx = rmm.rmm_score_select(A, rho=0.5)[0]
    Y, e = rmm.rmm_reduced_gemm(A, B, idx, want_energy=True)
    assert torch.equal(Y, rmm.rmm_reduced_gemm(A, B, idx))
    assert torch.allclose(e.double(), Y.double().square().sum(0), rtol=3e-7, atol=0)
