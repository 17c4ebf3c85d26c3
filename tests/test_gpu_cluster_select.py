"""Selection of more keys than one block holds (select_cluster_kernel)."""
import numpy as np
import pytest
import torch

import paper_2608_13426_b200 as rmm

pytestmark = pytest.mark.gpu


def keys_of(kind, K, seed):
    g = torch.Generator().manual_seed(seed)
    if kind == "uniform":
        return torch.rand(K, generator=g)
    if kind == "concentrated":              # column energies: nearly equal, with a few far larger ones
        x = 1.0 + 0.01 * torch.randn(K, generator=g)
        x[torch.randperm(K, generator=g)[: K // 100]] *= 300.0
        return x
    if kind == "ties":
        return torch.randint(0, 7, (K,), generator=g).float()
    if kind == "equal":
        return torch.full((K,), 2.5)
    x = torch.randn(K, generator=g) * 1e30   # signs, zeros, infinities and the lowest value
    x[::97], x[5::1013], x[7::2011], x[9::3001] = 0.0, float("inf"), -float("inf"), torch.finfo(torch.float32).min
    return x


@pytest.mark.parametrize("K", [8193, 8200, 14336, 16383, 16384, 16385, 28672, 32768, 32771, 65536, 65537])
@pytest.mark.parametrize("kind", ["uniform", "concentrated", "ties", "equal", "wild"])
def test_many_keys_match_the_oracle(oracle, K, kind):
    keys = keys_of(kind, K, K)
    for k in (1, 2, K // 3, K // 2, K - 1, K):
        want, _ = oracle.select(keys.double().numpy(), k)
        assert np.array_equal(rmm.rmm_select(keys.cuda(), k=k).cpu().numpy(), want), k


def test_many_keys_batches_retained_and_alignment(oracle):
    K = 10001                                # rows of the batch start off 16 bytes
    keys = torch.stack([keys_of("concentrated", K, s) for s in range(20)])
    idx, kept = rmm.rmm_select(keys.cuda(), rho=0.4, want_retained=True)
    for b in range(20):
        want, _ = oracle.select(keys[b].double().numpy(), idx.shape[1])
        frac = float(keys[b].double()[want].sum() / keys[b].double().sum())
        assert np.array_equal(idx[b].cpu().numpy(), want)
        assert abs(float(kept[b]) - frac) <= 2e-7      # fp64 sums, rounded once to fp32


@pytest.mark.parametrize("batch, K", [(79, 8201), (130, 14336), (120, 28672), (149, 9000), (300, 16385), (150, 49152), (140, 49153)])
def test_many_lists_at_once_match_one_at_a_time(batch, K):
    """A block per list or a cluster per list, whichever the rule takes: the sets and fractions are the same."""
    keys = torch.stack([keys_of(("uniform", "concentrated", "ties", "wild")[b % 4], K, b) for b in range(batch)]).cuda()
    keys[3::4] = keys[3::4].clamp(min=0.0, max=1e30)                       # (fractions of what is finite)
    idx, kept = rmm.rmm_select(keys, rho=0.3, want_retained=True)
    for b in range(0, batch, 7):
        one, frac = rmm.rmm_select(keys[b].contiguous(), rho=0.3, want_retained=True)
        assert torch.equal(idx[b], one), b
        assert abs(float(kept[b]) - float(frac)) <= 2.0 ** -23
    assert rmm.rmm_status_read() == 0
