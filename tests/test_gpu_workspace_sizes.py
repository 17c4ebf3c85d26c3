"""A workspace that was sized for one shape serves the smaller ones: the forms that cut the contraction axis into pieces take
fewer of them where their partial sums do not fit."""
import ctypes

import numpy as np
import pytest
import torch

import paper_2608_13426_b200 as rmm
from paper_2608_13426_b200 import binding, synth

pytestmark = pytest.mark.gpu


def buffer(nbytes):
    return torch.zeros(nbytes, dtype=torch.uint8, device="cuda")


def sized_for(A, B, k):
    Y = torch.empty(A.shape[0], B.shape[1], dtype=A.dtype, device="cuda")
    return binding.lib().rmm_reduced_gemm_workspace_bytes(*(ctypes.byref(binding.as_mat(x)) for x in (A, B)), k, ctypes.byref(binding.as_mat(Y)))


def kept(K, k):
    return torch.arange(0, K, K // k, dtype=torch.int32, device="cuda")[:k]


@pytest.mark.parametrize("dtype, K, N, tol", [(torch.bfloat16, 4096, 264, 1e-2), (torch.float32, 4096, 264, 1e-5)])
def test_a_workspace_for_more_rows_serves_fewer(oracle, dtype, K, N, tol):
    A, B = synth.mlp_product(1024, K, N, seed=181, dtype=dtype)
    Ad, Bd, idx = A.cuda(), B.cuda(), kept(K, K // 2)
    want = oracle.reduced_gemm(A[:256], B, idx.cpu().numpy())
    ws = buffer(sized_for(Ad, Bd, K // 2))
    for M in (256, 129, 128, 33, 32, 9, 5, 1):
        for nbytes in (len(ws), len(ws) if dtype == torch.bfloat16 else 4096):     # (fp32 operands are read in place)
            Y = rmm.rmm_reduced_gemm(Ad[:M].contiguous(), Bd, idx, ws=ws[:nbytes])
            rel = np.linalg.norm(Y.float().cpu().numpy() - want[:M]) / np.linalg.norm(want[:M])
            assert rel <= tol, (M, nbytes, rel)
    assert rmm.rmm_status_read(ws=ws) == 0


@pytest.mark.parametrize("K", [8192, 128])
@pytest.mark.parametrize("M", [8, 32, 48, 128, 200])
def test_what_packed_operands_take_is_enough_where_rows_are_fetched_in_place(oracle, M, K):
    N, k = 256, K // 2                         # few columns: the pieces' sums are what a full workspace is made of
    A, B = synth.mlp_product(M, K, N, seed=182)
    Ad, Bd, idx = A.cuda(), B.cuda(), kept(K, k)
    full = sized_for(Ad, Bd, k)
    need = 4096 + (M * k * 2 + 255) // 256 * 256 + min(full, k * N * 2)
    want = oracle.reduced_gemm(A, B, idx.cpu().numpy())
    for nbytes in (full, min(full, need)):
        ws = buffer(nbytes)
        Y = rmm.rmm_reduced_gemm(Ad, Bd, idx, ws=ws)
        assert np.linalg.norm(Y.float().cpu().numpy() - want) <= 1e-2 * np.linalg.norm(want)
        assert rmm.rmm_status_read(ws=ws) == 0
    with pytest.raises(binding.RmmError) as e:
        rmm.rmm_reduced_gemm(Ad, Bd, idx, ws=buffer(4096 + M * k * 2 - 512))
    assert e.value.code == binding.RMM_ERR_WORKSPACE


def test_the_reserve_follows_the_problem():
    """48 rows of a small product do not ask for what 148 SMs could fill."""
    A, B = torch.empty(48, 512, dtype=torch.bfloat16, device="cuda"), torch.empty(512, 256, dtype=torch.bfloat16, device="cuda")
    assert sized_for(A, B, 256) <= 4096 + 48 * 512 * 2 + 4 * 48 * 1024
    sizes = [sized_for(A, B, k) for k in (64, 128, 256, 512)]
    assert sizes == sorted(sizes)


def test_a_small_scored_product_in_what_whole_tiles_take():
    """Packed A and the epilogue's column energies: no room for a pass over the output."""
    M, K, N, k = 64, 512, 256, 256
    A, B = synth.mlp_product(M, K, N, seed=183)
    Ad, Bd, idx = A.cuda(), B.cuda(), kept(K, k)
    Y, e = rmm.rmm_reduced_gemm(Ad, Bd, idx, want_energy=True)
    ws = buffer(4096 + M * k * 2 + M // 32 * N * 4)
    Y2, e2 = rmm.rmm_reduced_gemm(Ad, Bd, idx, want_energy=True, ws=ws)
    assert float((Y2.double() - Y.double()).norm() / Y.double().norm()) <= 2.0 ** -8        # a rounding to bf16 apart
    assert torch.allclose(e2.double(), Y2.double().square().sum(0), rtol=3e-7, atol=0) and rmm.rmm_status_read(ws=ws) == 0
