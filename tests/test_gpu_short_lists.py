"""Selection of at most 128 keys by comparing all pairs (select.cuh)."""
import numpy as np
import pytest
import torch

import paper_2608_13426_b200 as rmm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [1, 2, 3, 15, 16, 17, 31, 32, 33, 64, 96, 127, 128, 129])
def test_short_lists_against_the_oracle(oracle, K):
    g = torch.Generator().manual_seed(K)
    keys = torch.randint(0, max(2, K // 3), (5, K), generator=g).float()     # ties across the threshold
    keys[1] = torch.rand(K, generator=g)
    keys[2] = 0.0
    if K > 4:
        keys[3, 1], keys[3, 3], keys[3, K - 1] = float("inf"), -float("inf"), torch.finfo(torch.float32).min
    keys[4] = -torch.rand(K, generator=g)
    for k in sorted({1, (K + 1) // 2, max(1, K - 1), K}):
        idx, kept = rmm.rmm_select(keys.cuda(), k=k, want_retained=True)
        for b in range(5):
            assert np.array_equal(idx[b].cpu().numpy(), oracle.select(keys[b].double().numpy(), k)[0]), (b, k)
        assert abs(float(kept[1]) - float(keys[1][idx[1].cpu().long()].double().sum() / keys[1].double().sum())) <= 2e-7
