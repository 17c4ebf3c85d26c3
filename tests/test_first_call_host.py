"""Several threads at a kernel's first use (common.cuh, PerDeviceOnce), against a runtime of two fake calls: a thread that comes
while another is still setting the shared-memory attribute must not go on to its launch before the attribute is set."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

FAKES = r"""
#include <atomic>
#include <thread>
std::atomic<int> calls{0};
std::atomic<bool> set{false}, second_back{false};
extern "C" void **__cudaRegisterFatBinary(void *) { return nullptr; }   // (what the compiler's start-up code refers to)
extern "C" void __cudaRegisterFatBinaryEnd(void **) {}
extern "C" void __cudaUnregisterFatBinary(void **) {}
extern "C" char __cudaInitModule(void **) { return 0; }
extern "C" int cudaGetDevice(int *d) { *d = 3; return 0; }
extern "C" int cudaFuncSetAttribute(const void *, int, int)
{
    if (calls.fetch_add(1) == 0)
        while (!second_back) std::this_thread::yield();   // the first thread is held inside the call
    set = true;
    return 0;
}
"""

HARNESS = r"""
#include <cstdio>
#include <thread>
#include "common.cuh"
extern std::atomic<int> calls;
extern std::atomic<bool> set, second_back;
void kernel(int) {}
int main()
{
    static rmm::PerDeviceOnce once;
    std::thread first([] { once.smem(65536, kernel); });
    while (calls.load() == 0) std::this_thread::yield();
    const bool ok = once.smem(65536, kernel) == cudaSuccess && set;   // set although the first thread is not back
    second_back = true;
    first.join();
    const int after = calls;
    const bool kept = once.smem(65536, kernel) == cudaSuccess && calls == after;   // and no more calls from then on
    printf("%d %d\n", ok, kept);
    return ok && kept ? 0 : 1;
}
"""


@pytest.mark.skipif(not os.path.exists(NVCC), reason="needs nvcc")
def test_nobody_goes_on_before_the_attribute_is_set(tmp_path):
    src, fakes, exe = tmp_path / "once.cu", tmp_path / "fakes.cpp", tmp_path / "once"
    src.write_text(HARNESS)
    fakes.write_text(FAKES)
    inc = [os.path.join(ROOT, "include"), os.path.join(ROOT, "paper_2608_13426_b200", "csrc")]
    subprocess.run([NVCC, "-std=c++17", "-cudart", "none", "--expt-relaxed-constexpr", *[a for i in inc for a in ("-I", i)], "-o", str(exe), str(src), str(fakes),
                    "-lpthread"], check=True, capture_output=True, text=True, timeout=300)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
