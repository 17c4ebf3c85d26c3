"""fp32 products whose parts would take more memory than the split form allows itself: panels in the same scratch (gemm_split.cu)."""
import pytest
import torch

import paper_2608_13426_b200 as rmm
from paper_2608_13426_b200 import binding

pytestmark = pytest.mark.gpu

LIMIT = 4096 + (512 << 20) + 2 * 148 * 65536 + (4 << 20)     # the parts, the cut tiles' sums and the flags of the largest panel


def close(Y, A, B, idx):
    for r in range(0, A.shape[0], 1024):
        want = A[r:r + 1024][:, idx.long()].double() @ B[idx.long()].double()
        err = (Y[r:r + 1024].double() - want).norm(dim=1) / want.norm(dim=1)
        assert float(err.max()) <= 2.0 ** -21, r          # every row by itself


# rows cut; columns cut, both operands the other way round; several of both
@pytest.mark.parametrize("M, K, N, columns", [(6000, 10000, 3001, False), (2049, 12000, 6100, True), (9000, 24000, 5000, False)])
def test_panels(M, K, N, columns):
    g = torch.Generator(device="cuda").manual_seed(M)
    A, B = torch.randn(M, K, generator=g, device="cuda"), torch.randn(K, N, generator=g, device="cuda")
    if columns:
        A, B = A.t().contiguous().t(), B.t().contiguous().t()
    idx = torch.arange(0, K, 4, dtype=torch.int32, device="cuda")
    A[M - 1, 4], A[0, 8] = 1e-30, 1e-20                   # cannot be split, in the last panel and in the first
    Y = torch.empty(M, N, device="cuda")
    need = binding.lib().rmm_reduced_gemm_workspace_bytes(*(binding.as_mat(x) for x in (A, B)), len(idx), binding.as_mat(Y))
    assert need <= LIMIT
    n0 = rmm.rmm_launch_count()
    rmm.rmm_reduced_gemm(A, B, idx, out=Y)
    launches = rmm.rmm_launch_count() - n0
    assert launches % 3 == 0 and launches >= 6
    close(Y, A, B, idx)
    assert torch.equal(Y, rmm.rmm_reduced_gemm(A, B, idx)) and rmm.rmm_status_read() == 0


def test_panels_of_a_batch():
    g = torch.Generator(device="cuda").manual_seed(1)
    A, B = torch.randn(3, 2000, 10000, generator=g, device="cuda"), torch.randn(3, 10000, 1500, generator=g, device="cuda")
    idx = torch.stack([torch.randperm(10000, generator=torch.Generator().manual_seed(b))[:2500].sort().values for b in range(3)]).int().cuda()
    for b in (B, B[1]):
        n0 = rmm.rmm_launch_count()
        Y = rmm.rmm_reduced_gemm(A, b, idx)
        assert rmm.rmm_launch_count() - n0 == 6
        for i in range(3):
            close(Y[i], A[i], b if b.dim() == 2 else b[i], idx[i])
    assert rmm.rmm_status_read() == 0


def test_a_product_asks_for_what_its_kept_count_takes():
    """rmm_product through the binding: the workspace is sized by k, and the split form runs in it."""
    g = torch.Generator(device="cuda").manual_seed(2)
    A, B = torch.randn(2048, 8192, generator=g, device="cuda"), torch.randn(8192, 2048, generator=g, device="cuda")
    kept, cache = binding._ws_cache, {}
    binding._ws_cache = cache
    try:
        n0 = rmm.rmm_launch_count()
        Y, idx = rmm.rmm_product(A, B, k=2048)
        assert rmm.rmm_launch_count() - n0 == 4            # scores and selection, then gather, product, what is left of it
        assert max(ws.numel() for ws in cache.values()) <= 6 * 4096 * 2048 + 2 * 148 * 65536 + (2 << 20)
        assert torch.equal(Y, rmm.rmm_reduced_gemm(A, B, idx))
        close(Y, A, B, idx)
    finally:
        binding._ws_cache = kept
