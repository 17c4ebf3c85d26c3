"""Selection whose keys share the threshold's first digit: few of them (finished from a list in the front end) or many (select.cuh)."""
import numpy as np
import pytest
import torch

import paper_2608_13426_b200 as rmm

pytestmark = pytest.mark.gpu


def clustered(K, same, seed):
    """`same` keys within 2^-12 of each other, ties among them, the others spread over six powers of two."""
    g = torch.Generator().manual_seed(seed)
    x = 64.0 ** torch.rand(K, generator=g) * 0.1
    x[torch.randperm(K, generator=g)[:same]] = 1.0 + torch.randint(0, 300, (same,), generator=g) * 2.0 ** -21
    return x


@pytest.mark.parametrize("K", [129, 255, 1023, 1024, 1025, 4095, 4096, 4097, 8191, 8192])
@pytest.mark.parametrize("same", [1, 31, 256, 1000, 1024, 1025, 4000])
def test_keys_that_share_the_first_digit(oracle, K, same):
    same = min(same, K)
    keys = clustered(K, same, K + same)
    above = int((keys > 1.001).sum())
    for k in sorted({1, K, max(1, above), min(K, above + 1), above + (same + 1) // 2, above + same}):
        got, kept = rmm.rmm_select(keys.cuda(), k=k, want_retained=True)
        want, _ = oracle.select(keys.double().numpy(), k)
        assert np.array_equal(got.cpu().numpy(), want), k
        frac = float(keys.double()[want].sum() / keys.double().sum())
        assert abs(float(kept) - frac) <= 2e-7       # fp64 sums, rounded once to fp32


@pytest.mark.parametrize("M, K, N", [(64, 4096, 4096), (300, 8192, 512), (40, 2048, 1024), (128, 8192, 2048)])
@pytest.mark.parametrize("same", [3, 900, 2000])
def test_a_product_keeps_the_columns_that_the_selection_keeps(oracle, M, K, N, same):
    """Two entries a column whose squares and their sum are exact in fp32, so the energies do not depend on any order."""
    same = min(same, K)
    g = torch.Generator().manual_seed(M + same)
    one, two = 8.0 ** torch.rand(K, generator=g), torch.zeros(K)
    near = torch.randperm(K, generator=g)[:same]
    one[near], two[near] = 1.0, torch.randint(0, 128, (same,), generator=g) * 2.0 ** -11
    one = one.bfloat16().float()
    A, col = torch.zeros(M, K), torch.arange(K)
    A[col % M, col], A[(col + 7) % M, col] = one, two
    energy = one.double() ** 2 + two.double() ** 2
    assert torch.equal(energy, energy.float().double())
    k = int((energy > 1.01).sum()) + (same + 1) // 2
    B = torch.randint(-3, 4, (K, N), generator=g).float()
    Y, idx = rmm.rmm_product(A.cuda().bfloat16(), B.cuda().bfloat16(), k=k)
    want, _ = oracle.select(energy.numpy(), k)
    assert np.array_equal(idx.cpu().numpy(), want)
    exact = A[:, want].double() @ B[want].double()
    assert float((Y.double().cpu() - exact).abs().max()) <= float(exact.abs().max()) * 2.0 ** -8   # one rounding to bf16
