"""On a device whose flags ask for blocking waits (cudaDeviceScheduleBlockingSync)
a solve leaves the processor while it waits.  Run in a process of its own: the
flags belong to the process's context.

Bar: at most a quarter of the solve's wall time in the calling thread.  The
launches are some 4 per update of about 0.3 ms (3% of it); a thread that spins
through step 1, the only step here, takes more than half."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = """
import ctypes, time
cu = ctypes.CDLL("libcuda.so.1")
assert cu.cuInit(0) == 0 and cu.cuDevicePrimaryCtxSetFlags_v2(0, 4) == 0  # blocking sync
import torch
import paper_2406_03468_gb300 as lsq
m, n = 400000, 500
g = torch.Generator(device="cuda")
g.manual_seed(1)
A = torch.randn(m, n, generator=g, dtype=torch.float64, device="cuda")
b = torch.randn(m, generator=g, dtype=torch.float64, device="cuda")
x = torch.empty(n, dtype=torch.float64, device="cuda")
plan = lsq.Plan(m, n, seed=1, max_refine=1)
for _ in range(2):
    st, info = plan.solve(A, b, x)
assert st == 0 and info["iters"][0] > 10
torch.cuda.synchronize()
w, c = time.perf_counter(), time.thread_time()
for _ in range(10):
    plan.solve(A, b, x)
print("share", (time.thread_time() - c) / (time.perf_counter() - w))
plan.close()
"""


def test_blocking_device_is_waited_for_without_spinning():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD], capture_output=True, text=True, cwd=root,
                       timeout=300, env=dict(os.environ, PYTHONPATH=root))
    assert r.returncode == 0, r.stderr[-2000:]
    share = float(r.stdout.split("share")[1])
    assert share <= 0.25, share
