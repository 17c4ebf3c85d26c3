"""2^x on the FMA pipe (ex2_fma in sm100_ptx.cuh) by itself, against 64 bits."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2608_13426_b200 import build as rmm_build

pytestmark = pytest.mark.gpu

SOURCE = """
#include <cuda_bf16.h>
#include "sm100_ptx.cuh"
__global__ void both(const float *x, float *y, long pairs)
{
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < pairs) rmm::ptx::ex2_fma(x[2 * i], x[2 * i + 1], y[2 * i], y[2 * i + 1]);
}
extern "C" int run(const float *x, float *y, long pairs)
{
    both<<<(unsigned)((pairs + 255) / 256), 256>>>(x, y, pairs);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def ex2_fma(tmp_path_factory):
    at = tmp_path_factory.mktemp("ex2_fma")
    (at / "t.cu").write_text(SOURCE)
    subprocess.run([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), *rmm_build.NVCC_FLAGS, "-shared", "-I", os.path.join(rmm_build.ROOT, "include"),
                    "-I", rmm_build.CSRC, "-o", str(at / "t.so"), str(at / "t.cu")], check=True)
    run = ctypes.CDLL(str(at / "t.so")).run
    run.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_long]

    def f(x):
        x = torch.from_numpy(np.resize(x, (len(x) + 1) // 2 * 2)).cuda()
        y = torch.full_like(x, float("nan"))
        torch.cuda.synchronize()
        assert run(x.data_ptr(), y.data_ptr(), len(x) // 2) == 0
        return y.cpu().numpy()

    return f


def test_against_64_bits(ex2_fma):
    halves = np.arange(-280, 81, dtype=np.float32) / 2            # where x changes its integer
    x = np.concatenate([halves, np.nextafter(halves, np.float32(-999)), np.nextafter(halves, np.float32(999)),
                        np.random.default_rng(0).uniform(-140, 40, 4_000_000).astype(np.float32),
                        np.linspace(-1, 1, 2_000_001, dtype=np.float32)])
    y = ex2_fma(x)[:len(x)].astype(np.float64)
    want = np.exp2(x.astype(np.float64))
    normal = x >= -126
    # the polynomial with fp32 coefficients 1.09e-7 (its error over [-1/2, 1/2] in 64 bits), and the last rounding, 2^-24
    assert (np.abs(y - want) <= 1.7e-7 * want)[normal].all()
    # subnormal results: off by at most a rounding more, or zero once x rounds to -127
    low = ~normal & (x > -126.5)
    assert (np.abs(y - want) <= 1.7e-7 * want + 2.0 ** -149)[low].all()
    assert (y[x < -126.5] == 0).all()


def test_special_values(ex2_fma):
    y = ex2_fma(np.array([-np.inf, np.nan, -3e38, 0, -0.0, 1, np.nan, 5], dtype=np.float32))
    assert y[0] == 0 and np.isnan(y[1]) and y[2] == 0 and y[3] == 1 and y[4] == 1 and y[5] == 2 and np.isnan(y[6]) and y[7] == 32
