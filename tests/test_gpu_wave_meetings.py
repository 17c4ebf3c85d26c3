"""Products of several waves of tiles, whose blocks meet before each tile where a contraction holds 16 KB or more (gemm_sm100.cu)."""
import pytest
import torch

import paper_2608_13426_b200 as rmm

pytestmark = pytest.mark.gpu

M = N = 2304   # 81 pair tiles on 74 pairs of multiprocessors


def check(Y, A, B, k):
    A, B = A.double(), B.double()
    # k additions in fp32 that round toward zero
    assert ((Y.double() - A @ B).abs() <= k * 2.0 ** -23 * (A.abs() @ B.abs())).all()
    assert rmm.rmm_status_read() == 0


@pytest.mark.parametrize("k", [8191, 8192, 8200])
def test_bf16(k):
    g = torch.Generator(device="cuda").manual_seed(k)
    A = torch.randn(M, 8704, generator=g, device="cuda").bfloat16()
    B = torch.randn(8704, N, generator=g, device="cuda").bfloat16()
    idx = torch.randperm(8704, generator=g, device="cuda")[:k].sort().values.int()
    Y = rmm.rmm_reduced_gemm(A, B, idx, out_dtype=torch.float32)
    check(Y, A[:, idx.long()], B[idx.long()], k)
    assert torch.equal(rmm.rmm_reduced_gemm(A, B, idx, out_dtype=torch.float32), Y)   # the meeting's counters are back at zero


@pytest.mark.parametrize("k", [8192, 16368, 16383, 16384, 16400])
def test_8_bit(k):
    g = torch.Generator(device="cuda").manual_seed(k)
    K = 16640
    A = (torch.randn(M, K, generator=g, device="cuda") * 64).to(torch.float8_e4m3fn).bfloat16()
    B = torch.randn(N, K, generator=g, device="cuda").to(torch.float8_e4m3fn)
    idx = torch.randperm(K, generator=g, device="cuda")[:k].sort().values.int()
    A[:, idx[0].long()] = 448                                                         # every row's step is one: the codes are A itself
    Y, step = rmm.rmm_reduced_gemm_q8(A, B, 1.0, idx, out_dtype=torch.float32, want_scales=True)
    assert (step == 1).all()
    check(Y, A[:, idx.long()], B.bfloat16()[:, idx.long()].T, k)
    assert torch.equal(rmm.rmm_reduced_gemm_q8(A, B, 1.0, idx, out_dtype=torch.float32), Y)
