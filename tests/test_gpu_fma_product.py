"""The product on the FMA pipes (gemm_simt.cu): tile edges, sliced contraction axes, every kind of load."""
import pytest
import torch

import paper_2608_13426_b200 as rmm

pytestmark = pytest.mark.gpu


def ints(shape, seed, dtype=torch.float32):
    """Small whole numbers: every product and partial sum is exact in fp32, so any order of summation gives the same."""
    return torch.randint(-3, 4, shape, generator=torch.Generator().manual_seed(seed)).to(dtype)


@pytest.mark.parametrize("M,K,N,k", [
    (1, 1, 1, 1), (31, 17, 5, 16), (32, 40, 64, 33), (33, 100, 127, 65), (63, 3000, 128, 2000), (64, 64, 129, 63),
    (65, 9000, 132, 8192), (777, 300, 260, 48), (130, 5000, 1500, 1023), (2048, 70, 1000, 70), (5, 7373, 4096, 7372),
])
@pytest.mark.parametrize("form", ["rows", "columns of B", "columns of A", "odd pitch"])
def test_fp32_product_is_exact_on_whole_numbers(M, K, N, k, form):
    A, B = ints((M, K), 1), ints((K, N), 2)
    idx = torch.randperm(K, generator=torch.Generator().manual_seed(3))[:k].sort().values
    Ad, Bd = A.cuda(), B.cuda()
    if form == "columns of B":
        Bd = B.t().contiguous().cuda().t()
    elif form == "columns of A":
        Ad = A.t().contiguous().cuda().t()
    elif form == "odd pitch":
        Bd = torch.zeros(K, N + 1, device="cuda")[:, :N].copy_(Bd)
    out = torch.full((M, N + (form == "odd pitch")), float("nan"), device="cuda")[:, :N]
    Y = rmm.rmm_reduced_gemm(Ad, Bd, idx.int().cuda(), scale=0.5, out=out)
    assert torch.equal(Y.cpu(), 0.5 * (A[:, idx].double() @ B[idx].double()).float())
    again = rmm.rmm_reduced_gemm(Ad, Bd, idx.int().cuda(), scale=0.5)          # the arrival counters are back at zero
    assert torch.equal(again, Y)
    assert rmm.rmm_status_read() == 0


def test_bf16_product_off_the_tensor_core_rules_and_bad_indices():
    A, B = ints((70, 901), 4, torch.bfloat16), ints((901, 131), 5, torch.bfloat16)   # 131 columns: not a multiple of 8
    idx = torch.arange(0, 901, 2)
    want = A[:, idx].double() @ B[idx].double()
    Y = rmm.rmm_reduced_gemm(A.cuda(), B.cuda(), idx.int().cuda(), out_dtype=torch.float32)
    assert torch.equal(Y.cpu().double(), want)
    A, B = ints((3, 40, 60), 6), ints((3, 60, 50), 7)                                # one list per batch entry
    lists = torch.stack([torch.randperm(60, generator=torch.Generator().manual_seed(s))[:37].sort().values for s in range(3)])
    Y = rmm.rmm_reduced_gemm(A.cuda(), B.cuda(), lists.int().cuda())
    assert torch.equal(Y.cpu(), torch.stack([A[b][:, lists[b]] @ B[b][lists[b]] for b in range(3)]))
    bad = lists[:1].clone()
    bad[0, 5], bad[0, 6] = 60, -1                                                    # reported, and worth nothing
    keep = torch.ones(37, dtype=torch.bool)
    keep[5:7] = False
    Y = rmm.rmm_reduced_gemm(A[0].cuda(), B[0].cuda(), bad[0].int().cuda())
    assert torch.equal(Y.cpu(), A[0][:, lists[0][keep]] @ B[0][lists[0][keep]])
    assert rmm.rmm_status_read() == 6
    assert rmm.rmm_status_read() == 0
