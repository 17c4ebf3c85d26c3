"""The decode-step product whose slices of the kept rows fill one staging buffer, just miss it or take several (gemv.cu)."""
import pytest
import torch

import paper_2608_13426_b200 as rmm
from paper_2608_13426_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [1, 2, 3, 4])
@pytest.mark.parametrize("k", [3 * 512 - 1, 3 * 512, 3 * 512 + 1, 3 * 1024 - 2, 3 * 1024, 3 * 1024 + 1, 3 * 2048 + 5])
def test_slices_around_the_buffer(M, k):
    K, N = 6200, 149 * 256                                     # three slices of the kept rows
    A, B = synth.mlp_product(M, K, N, seed=k, device="cuda")
    idx = torch.randperm(K, generator=torch.Generator().manual_seed(M))[:k].sort().values.int().cuda()
    Y = rmm.rmm_reduced_gemm(A, B, idx, out_dtype=torch.float32)
    i = idx.long()
    want = A[:, i].double() @ B[i].double()
    # fp32 sums of k products of either sign: 2^-24 per step of a slice's eight interleaved chains
    assert (Y.double() - want).norm() <= k * 2.0 ** -24 * want.norm()
    bad = idx.clone()
    bad[k // 2] = K                                            # an index out of range is reported and contributes nothing
    keep = torch.arange(k, device="cuda") != k // 2
    Y = rmm.rmm_reduced_gemm(A, B, bad, out_dtype=torch.float32)
    assert rmm.rmm_status_read() == rmm.binding.RMM_ERR_BOUNDS
    want = A[:, i[keep]].double() @ B[i[keep]].double()
    assert (Y.double() - want).norm() <= k * 2.0 ** -24 * want.norm()
