"""Attention whose K or V holds less than the call would read is refused before anything is launched; more is fine."""
import pytest
import torch

import paper_2608_13426_b200 as rmm
from paper_2608_13426_b200 import binding, synth

Q_SHAPE, KV_SHAPE = (2, 4, 3, 16), (2, 2, 40, 16)
SMALLER = [((1, 2, 40, 16), KV_SHAPE), ((2, 2, 40, 8), KV_SHAPE),                       # K: a sequence, columns short
           (KV_SHAPE, (1, 2, 40, 16)), (KV_SHAPE, (2, 1, 40, 16)), (KV_SHAPE, (2, 2, 39, 16)), (KV_SHAPE, (2, 2, 40, 8))]


class OnDevice:
    """A tensor of the CPU that says it is on a GPU; nothing but its description can be had."""

    def __init__(self, *shape):
        t = torch.empty(shape, dtype=torch.bfloat16)
        self.shape, self.dtype, self.is_cuda, self.dim, self.stride = t.shape, t.dtype, True, t.dim, t.stride


@pytest.mark.parametrize("k, v", SMALLER)
def test_refused_by_its_description(k, v):
    with pytest.raises(binding.RmmError) as e:
        rmm.rmm_reduced_attn(OnDevice(*Q_SHAPE), OnDevice(*k), OnDevice(*v), True, 0.5)
    assert e.value.code == binding.RMM_ERR_INVALID_ARG


@pytest.mark.gpu
@pytest.mark.parametrize("k, v", SMALLER)
def test_refused_by_both_ways_of_marshalling(k, v):
    Q, K, V = (torch.zeros(s, dtype=torch.bfloat16, device="cuda") for s in (Q_SHAPE, k, v))
    assert binding._native().attn(Q, K, V, True, 0.5, 1.0) is None
    launched = rmm.rmm_launch_count()
    for more in ({}, {"want_idx": True}):
        with pytest.raises(binding.RmmError) as e:
            rmm.rmm_reduced_attn(Q, K, V, True, 0.5, **more)
        assert e.value.code == binding.RMM_ERR_INVALID_ARG
    assert rmm.rmm_launch_count() == launched


@pytest.mark.gpu
@pytest.mark.parametrize("Lq, rho_t", [(1, 1.0), (70, 1.0), (70, 0.5)])
def test_caches_longer_and_wider_than_the_call(Lq, rho_t):
    Q, K, V = synth.attention_qkv(1, 4, 2, Lq, 200, 64, seed=3, device="cuda")
    want = rmm.rmm_reduced_attn(Q, K[:, :, :150].contiguous(), V[:, :, :150].contiguous(), True, 0.5, rho_t)
    wide = torch.zeros(3, 2, 200, 72, dtype=torch.bfloat16, device="cuda")
    wide[:1, ..., :64] = K
    assert torch.equal(rmm.rmm_reduced_attn(Q, wide[:, :, :150], V, True, 0.5, rho_t), want)
