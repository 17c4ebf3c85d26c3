"""Products of few CTA-pair tiles, cut along the contraction (gemm_sm100.cu): pieces that a second kernel adds up."""
import pytest
import torch

import paper_2608_13426_b200 as rmm

pytestmark = pytest.mark.gpu


def ints(shape, seed, dtype=torch.bfloat16):
    """Small whole numbers: products and fp32 sums are exact, so any cut of the contraction gives the same."""
    return torch.randint(-2, 3, shape, generator=torch.Generator().manual_seed(seed)).to(dtype).cuda()


# one tile to two thirds of a round (the last rows and columns of a tile outside Y), shares of less than a tile and of more
SHAPES = [(385, 9000, 520, 8001), (600, 9000, 1000, 8000), (900, 9000, 3000, 8999), (257, 16384, 264, 16000), (300, 9000, 136, 8999)]


@pytest.mark.parametrize("M, K, N, k", SHAPES)
def test_cut_tiles_are_exact_on_whole_numbers(M, K, N, k):
    A, B = ints((M, K), M), ints((K, N), N)
    idx = torch.randperm(K, generator=torch.Generator().manual_seed(k))[:k].sort().values.int().cuda()
    want = (A[:, idx.long()].float() @ B[idx.long()].float()) * 0.5        # whole numbers below 2^24: exact in fp32
    n0 = rmm.rmm_launch_count()
    Y = rmm.rmm_reduced_gemm(A, B, idx, scale=0.5, out_dtype=torch.float32)
    assert rmm.rmm_launch_count() - n0 == 3                                 # gathers, product, meeting
    assert torch.equal(Y, want)
    assert torch.equal(rmm.rmm_reduced_gemm(A, B, idx, scale=0.5), want.bfloat16())
    Bt = B.t().contiguous().t()                                            # K-major operand
    assert torch.equal(rmm.rmm_reduced_gemm(A, Bt, idx, scale=0.5, out_dtype=torch.float32), want)
    # a caller's workspace without room for the pieces: whole tiles
    ws = torch.zeros(4096 + 512 + (M * (k + 7) // 8 * 8 + k * N) * 2 + 1024, dtype=torch.uint8, device="cuda")
    assert torch.equal(rmm.rmm_reduced_gemm(A, B, idx, scale=0.5, ws=ws), want.bfloat16())
    Ys, e = rmm.rmm_reduced_gemm(A, B, idx, scale=0.5, want_energy=True)
    assert torch.equal(Ys, want.bfloat16())
    assert torch.allclose(e.double(), Ys.double().square().sum(0), rtol=3e-7, atol=0)
    assert rmm.rmm_status_read() == 0


def test_cut_tiles_with_8_bit_operands_and_in_the_one_call_form():
    M, K, N, k = 700, 8192, 768, 8000
    A, W = ints((M, K), 1), ints((N, K), 2)
    A[:, 0] = 448.0                                                         # every row's step is 1
    idx = torch.arange(k, dtype=torch.int32, device="cuda")
    Y = rmm.rmm_reduced_gemm_q8(A, W.to(torch.float8_e4m3fn), 1.0, idx, out_dtype=torch.float32)
    assert torch.equal(Y, A[:, :k].float() @ W[:, :k].float().t())
    B = W.t().contiguous()
    Y1, i1 = rmm.rmm_product(A, B, k=5000)
    assert torch.equal(Y1, rmm.rmm_reduced_gemm(A, B, i1)) and torch.equal(Y1, (A[:, i1.long()].float() @ B[i1.long()].float()).bfloat16())
    assert rmm.rmm_status_read() == 0
