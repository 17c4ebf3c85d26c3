"""fp32 products as sums of bf16 products on the tensor cores (gemm_split.cu)."""
import pytest
import torch

import paper_2608_13426_b200 as rmm

pytestmark = pytest.mark.gpu

# sizes at which the split form is the cheaper one: edges of its 128 x 128 tiles, 64-index k-blocks, 8-column rows of the packed
# parts; few tiles (the contraction cut into shares) and many
SIZES = [(777, 3000, 1500, 1500), (385, 9000, 520, 8191), (384, 8192, 512, 8192), (1024, 1025, 1023, 1025), (2048, 2048, 1280, 449), (600, 4100, 513, 4097)]


def operands(M, K, N, form, seed=0):
    g = torch.Generator().manual_seed(seed + M + N)
    A, B = torch.randn(M, K, generator=g).cuda(), (torch.randn(K, N, generator=g) * 0.02).cuda()
    if form == "wide":                      # rows of B off 16 bytes, columns of A apart
        return torch.stack([A, A], 2)[:, :, 0], torch.cat([B, B[:, :1]], 1)[:, :N]
    if form == "columns":                   # both with the other axis contiguous
        return A.t().contiguous().t(), B.t().contiguous().t()
    return A, B


def fma(A, B, idx):
    """The same product by the FMA kernel: a workspace of the header only."""
    ws = torch.zeros(4096 + 256, dtype=torch.uint8, device="cuda")
    return rmm.rmm_reduced_gemm(A, B, idx, ws=ws)


@pytest.mark.parametrize("form", ["rows", "wide", "columns"])
@pytest.mark.parametrize("M, K, N, k", SIZES)
def test_split_product_is_as_close_as_the_fma_kernel(M, K, N, k, form):
    A, B = operands(M, K, N, form)
    idx = torch.randperm(K, generator=torch.Generator().manual_seed(k))[:k].sort().values.int().cuda()
    n0 = rmm.rmm_launch_count()
    Y = rmm.rmm_reduced_gemm(A, B, idx)
    assert rmm.rmm_launch_count() - n0 == 3
    want = A[:, idx.long()].double() @ B[idx.long()].double()
    err, ref = [float((y.double() - want).norm() / want.norm()) for y in (Y, fma(A, B, idx))]
    assert err <= ref * 1.05 and err <= 2.0 ** -22, (err, ref)
    assert torch.equal(Y, rmm.rmm_reduced_gemm(A, B, idx))          # pieces are added in order
    half = rmm.rmm_reduced_gemm(A, B, idx, scale=0.5, out_dtype=torch.bfloat16)
    assert torch.equal(half, (Y * 0.5).bfloat16())
    assert rmm.rmm_status_read() == 0


VALUES = {"uniform": lambda t: t.uniform_(), "exponential": lambda t: t.exponential_(), "absolute": lambda t: t.normal_().abs_(),
          "spread": lambda t: t.normal_().mul_(2).exp_()}


@pytest.mark.parametrize("k", [51, 64, 96, 449, 1024, 4100])
@pytest.mark.parametrize("values", sorted(VALUES))
def test_operands_of_one_sign(values, k):
    """The tensor cores' sums round toward zero, which operands of one sign show: an accumulator of 64 indices is cut four times at its
    full size (16 indices an instruction), half a unit of 2^-23 each, so 2^-22 whatever k is.  Where values lie far apart each of an
    instruction's 17 terms is cut at a unit of the largest: 17 times that at the most."""
    M = N = 2048 if k < 1024 else 1024
    fill = VALUES[values]
    A, B = torch.empty(M, k, device="cuda"), torch.empty(k, N, device="cuda")
    torch.manual_seed(k)
    fill(A), fill(B)
    n0 = rmm.rmm_launch_count()
    Y = rmm.rmm_reduced_gemm(A, B, None)
    assert rmm.rmm_launch_count() - n0 == 3
    want = A.double() @ B.double()
    err = float((Y.double() - want).norm() / want.norm())
    assert err <= 2.0 ** -22 * (17 if values == "spread" else 1), err


def test_batches_shared_weights_and_no_list():
    A, B = torch.randn(3, 500, 2000, device="cuda"), torch.randn(3, 2000, 400, device="cuda")
    idx = torch.stack([torch.randperm(2000)[:1500].sort().values for _ in range(3)]).int().cuda()
    for b in (B, B[0]):
        Y = rmm.rmm_reduced_gemm(A, b, idx)
        for i in range(3):
            want = A[i][:, idx[i].long()].double() @ (b if b.dim() == 2 else b[i])[idx[i].long()].double()
            assert float((Y[i].double() - want).norm() / want.norm()) <= 2.0 ** -22
    Y = rmm.rmm_reduced_gemm(A[0], B[0], None)
    want = A[0].double() @ B[0].double()
    assert float((Y.double() - want).norm() / want.norm()) <= 2.0 ** -22


def fma_rows(A, B, idx):
    """The same product by the FMA kernel with room for the slices that it takes behind the split product."""
    M, N, k = A.shape[0], B.shape[1], len(idx)
    # the split product wants the header and its flags besides
    ws = torch.zeros(6 * (M + N) * k + 2 * 148 * 65536, dtype=torch.uint8, device="cuda")
    n0 = rmm.rmm_launch_count()
    Y = rmm.rmm_reduced_gemm(A, B, idx, ws=ws)
    assert rmm.rmm_launch_count() - n0 == 1
    return Y


# the last two of either side lie just inside 2^-50 .. 2^40, the ones before them just outside
@pytest.mark.parametrize("value", [float("inf"), -float("inf"), float("nan"), 3e38, 1e-38, 1e-44, -(2.0 ** 40) * (1 + 2.0 ** -23), 2.0 ** -50 * (1 - 2.0 ** -24)])
@pytest.mark.parametrize("where", ["A", "B", "B by columns"])
def test_elements_that_cannot_be_split_take_the_fma_kernel(value, where):
    """The outputs that see such an element, in tiles of 64 x 128, are the FMA kernel's bit for bit; the others stay.  (A product of
    several rounds of the FMA kernel's blocks; a smaller one is all its.)"""
    M, K, N, k = 4000, 3000, 4100, 1500
    A, B = operands(M, K, N, "rows", seed=5)
    if where == "B by columns":
        B = B.t().contiguous().t()
    X = A if where == "A" else B
    idx = torch.arange(0, 3000, 2, dtype=torch.int32, device="cuda")
    plain = rmm.rmm_reduced_gemm(A, B, idx)
    X[501 if where == "A" else 1001, 1001 if where == "A" else 501] = value    # not kept: nothing changes
    assert torch.equal(rmm.rmm_reduced_gemm(A, B, idx), plain)
    X[500, 500] = value
    Y, want = rmm.rmm_reduced_gemm(A, B, idx), fma_rows(A, B, idx)
    left = torch.zeros(M, N, dtype=torch.bool, device="cuda")
    if where == "A":
        left[448:512] = True                                                    # rows 496 .. 511 share a flag, a tile has 64
    elif where == "B":
        left[:, 256:512] = True                                                # 256 columns share a flag
    else:
        left[:, 384:512] = True                                                 # 16 columns do, a tile has 128
    same = (Y == want) | (Y.isnan() & want.isnan())
    assert bool(same[left].all()) and torch.equal(Y[~left], plain[~left])
    assert not bool(same[~left].all())                                          # the two forms do differ
    A, B = A[:777], B[:, :1500]
    Y, want = rmm.rmm_reduced_gemm(A, B, idx), fma_rows(A, B, idx)
    assert bool(((Y == want) | (Y.isnan() & want.isnan())).all()) and rmm.rmm_status_read() == 0


@pytest.mark.parametrize("value", [2.0 ** 40, -(2.0 ** 40), 2.0 ** -50, 0.0])
@pytest.mark.parametrize("where", ["A", "B"])
def test_elements_at_the_ends_of_the_range_are_split(value, where):
    M, K, N, k = 777, 3000, 1500, 1500
    A, B = operands(M, K, N, "rows", seed=5)
    idx = torch.arange(0, 3000, 2, dtype=torch.int32, device="cuda")
    (A if where == "A" else B)[500, 500] = value
    Y, other = rmm.rmm_reduced_gemm(A, B, idx), fma_rows(A, B, idx)
    rows = slice(500, 501) if where == "A" else slice(None)
    cols = slice(500, 501) if where == "B" else slice(None)
    assert not torch.equal(Y[448:512, 256:512], other[448:512, 256:512])
    # per output, against the sum of the products' magnitudes (3 parts: 2^-22 of it, as everywhere)
    want = A[rows][:, idx.long()].double() @ B[idx.long()][:, cols].double()
    size = A[rows][:, idx.long()].double().abs() @ B[idx.long()][:, cols].double().abs()
    assert bool(((Y[rows, cols].double() - want).abs() <= size * 2.0 ** -22).all())


@pytest.mark.parametrize("M, K, N, every", [(777, 3000, 1500, 1), (777, 3000, 1500, 40), (1100, 2000, 640, 1), (4000, 3000, 4100, 64)])
def test_many_elements_that_cannot_be_split(M, K, N, every):
    """From half of the tiles on, everything is the FMA kernel's."""
    A, B = operands(M, K, N, "rows", seed=6)
    idx = torch.arange(0, K, 2, dtype=torch.int32, device="cuda")
    A[::every, 0] = 1e-30
    Y, want = rmm.rmm_reduced_gemm(A, B, idx), fma_rows(A, B, idx)
    assert torch.equal(Y, want)
    exact = A[:, ::2].double() @ B[::2].double()
    assert bool(((Y.double() - exact).norm(dim=1) <= exact.norm(dim=1) * 2.0 ** -22).all())     # every row by itself
    again = rmm.rmm_reduced_gemm(A, B, idx)
    assert torch.equal(Y, again) and rmm.rmm_status_read() == 0


def test_bad_index_is_reported():
    A, B = operands(777, 3000, 1500, "rows", seed=6)
    idx = torch.arange(0, 3000, 2, dtype=torch.int32, device="cuda")
    idx[3], idx[700] = -1, 3000
    Y = rmm.rmm_reduced_gemm(A, B, idx)
    assert rmm.rmm_status_read() == 6 and rmm.rmm_status_read() == 0
    keep = torch.ones(1500, dtype=torch.bool)
    keep[3] = keep[700] = False
    kept = idx.cpu().long()[keep].cuda()
    want = A[:, kept].double() @ B[kept].double()
    assert float((Y.double() - want).norm() / want.norm()) <= 2.0 ** -22
