"""The quantising gather (quant.cu) shown by products with unit weights: every output is one code times its row's step."""
import numpy as np
import pytest
import torch

import paper_2608_13426_b200 as rmm
from paper_2608_13426_b200 import synth

pytestmark = pytest.mark.gpu


def shown(A, idx, N):
    """Dequantised A[:, idx[:N]] from the library: row n of B holds a one at its n-th kept column."""
    K, pitch = A.shape[1], (A.shape[1] + 15) // 16 * 16           # rows start on 16 bytes
    W = torch.zeros(N, pitch, dtype=torch.uint8)
    W[torch.arange(N), idx[:N].long()] = 0x38                      # the code of 1.0
    W = W.view(torch.float8_e4m3fn).cuda()[:, :K]
    wide = torch.full((A.shape[0], pitch), float("nan"), dtype=torch.bfloat16, device="cuda")   # what lies between rows is not used
    wide[:, :K] = A.cuda()
    Y, step = rmm.rmm_reduced_gemm_q8(wide[:, :K], W, 1.0, idx.int().cuda(), out_dtype=torch.float32, want_scales=True)
    assert rmm.rmm_status_read() == 0
    return Y.cpu().numpy(), step.cpu().numpy()


@pytest.mark.parametrize("M,K,k", [
    (1, 16, 16), (147, 4096, 4096), (300, 4096, 2048),     # a row or two per block
    (1200, 1000, 333),                                     # K off 16, k off 4: the zero pad stands for missing columns
    (700, 9000, 8200), (400, 20000, 12300), (160, 30008, 20000),   # four, two and one rows at a time
    (90, 56000, 2000),                                     # rows just short of the limit
    (20, 60000, 700),                                      # beyond it: one block per row
])
def test_codes_and_steps_match_the_definition(oracle, M, K, k):
    A = synth.heavy_tailed_activations(M, K, seed=K)
    idx = torch.randperm(K, generator=torch.Generator().manual_seed(k))[:k].sort().values
    N = min(k, 2048) // 16 * 16 or k
    got, step = shown(A, idx, N)
    codes, steps = oracle.quantize_rows_e4m3(A[:, idx].float().numpy())
    assert np.array_equal(step, steps.astype(np.float32))
    want = (codes[:, :N].astype(np.float32) * steps[:, None].astype(np.float32))
    assert np.array_equal(got, want)


def test_codes_at_ties_zeros_and_extremes(oracle):
    """Rows whose quotients sit on, just above and just below the points where codes change, tiny rows and zero rows."""
    g = torch.Generator().manual_seed(3)
    rows = []
    for e in (-120, -20, 0, 30, 100):
        for top in (448.0, 447.0, 300.0, 257.0):
            x = torch.rand(512, generator=g) * top
            x[:200] = torch.arange(1, 201).float() * 2.0 ** -10 * top / 448.0          # the smallest codes and what rounds to zero
            x[200:400] = (torch.randint(8, 16, (200,), generator=g) + 0.5) * 2.0 ** torch.randint(-8, 4, (200,), generator=g).float()
            x[400] = top
            rows.append(x.clamp(max=top) * 2.0 ** e * torch.where(torch.rand(512, generator=g) < 0.5, -1.0, 1.0))
    rows += [torch.zeros(512), torch.full((512,), 1e-40), torch.full((512,), -3e38)]
    A = torch.stack(rows).to(torch.bfloat16).repeat(20, 1)
    idx = torch.arange(512)
    got, step = shown(A, idx, 512)
    codes, steps = oracle.quantize_rows_e4m3(A.float().numpy())
    assert np.array_equal(step, steps.astype(np.float32))
    assert np.array_equal(got, codes.astype(np.float32) * steps[:, None].astype(np.float32))


@pytest.mark.parametrize("M,K,k", [
    (149, 4096, 2048), (149, 4096, 2049),                   # the last count that rows take on their own, the first that streams
    (500, 4104, 4097), (310, 16400, 12288),                 # an output in a second group of 4096; three groups, full
    (200, 30000, 24570), (150, 32000, 28000), (150, 40000, 32768),   # six, seven and eight groups, a row at a time
])
def test_every_number_of_output_groups(oracle, M, K, k):
    test_codes_and_steps_match_the_definition(oracle, M, K, k)
