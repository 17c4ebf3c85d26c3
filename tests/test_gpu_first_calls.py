"""Threads that use a kernel for the first time at the same moment: nobody may launch before the kernel's shared-memory
attribute is set (a launch without it is refused by the runtime with an error code; nothing runs)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import threading, torch
import paper_2608_13426_b200 as rmm
from paper_2608_13426_b200 import synth
N = 12
Q, K, V = (x.cuda() for x in synth.attention_qkv(1, 2, 2, 300, 300, 128, seed=1))
A, B = (x.cuda() for x in synth.mlp_product(2048, 1024, 512, seed=2))
W = (synth.weight(512, 1024, seed=3, dtype=torch.float32) * 64).to(torch.float8_e4m3fn).cuda()
idx = torch.arange(0, 1024, 2, dtype=torch.int32, device="cuda")
calls = [
    lambda ws: rmm.rmm_reduced_attn(Q[:, :, :1], K, V, True, 0.5, ws=ws),
    lambda ws: rmm.rmm_reduced_attn(Q, K, V, True, 0.5, ws=ws),
    lambda ws: rmm.rmm_reduced_gemm(A[:8], B, idx, ws=ws),
    lambda ws: rmm.rmm_reduced_gemm(A[:100], B, idx, ws=ws),
    lambda ws: rmm.rmm_reduced_gemm(A, B, idx, ws=ws),
    lambda ws: rmm.rmm_reduced_gemm_q8(A, W, 1.0 / 64, idx, ws=ws),
    lambda ws: rmm.rmm_score_select(A, rho=0.5, ws=ws)[0],
    lambda ws: rmm.rmm_score_select(A[:, 1:], rho=0.5, ws=ws)[0],
]
workspaces = [torch.zeros(64 << 20, dtype=torch.uint8, device="cuda") for _ in range(N)]
streams = [torch.cuda.Stream() for _ in range(N)]
torch.cuda.synchronize()
start, errors, results = threading.Barrier(N), [], [[None] * N for _ in calls]
def work(t):
    with torch.cuda.stream(streams[t]):
        for c, call in enumerate(calls):
            start.wait()
            try:
                results[c][t] = call(workspaces[t])
            except Exception as e:
                errors.append((c, t, str(e)))
threads = [threading.Thread(target=work, args=(t,)) for t in range(N)]
[t.start() for t in threads]
[t.join() for t in threads]
torch.cuda.synchronize()
assert not errors, errors
for c in range(len(calls)):
    assert all(torch.equal(results[c][0], r) for r in results[c]), c
assert all(rmm.rmm_status_read(ws=ws) == 0 for ws in workspaces)
"""


def test_threads_may_share_a_kernel_s_first_call():
    env = dict(os.environ, PYTHONPATH=ROOT + os.pathsep + os.environ.get("PYTHONPATH", ""))
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-1000:] + r.stderr[-3000:]
