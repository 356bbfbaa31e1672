"""A run's waits for the GPU leave the core where the process has asked the CUDA runtime for blocking waits."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# The flags of the device's context (cudaDeviceScheduleBlockingSync = 4) before anything has run on it, then PageRank on a
# graph whose iteration keeps the GPU busy for over a millisecond: of the waits' time a blocking wait takes the wake-ups
# only, some hundredths; a spin takes all of it.
PROGRAM = """
import ctypes, sys, time
import torch
cuda = ctypes.CDLL("libcuda.so.1")
assert cuda.cuInit(0) == 0 and cuda.cuDevicePrimaryCtxSetFlags_v2(0, int(sys.argv[1])) == 0
import paper_1806_08092_gb300 as gp
n, d = 1 << 23, 12
gen = torch.Generator(device="cuda"); gen.manual_seed(1)
col = torch.randint(n, (n * d,), device="cuda", generator=gen).to(torch.int32).view(torch.uint32)
row_ptr = (torch.arange(n + 1, device="cuda") * d).view(torch.uint64)
G = gp.Graph.from_csr(row_ptr, col)
G.run("pagerank", max_iters=3)
t0, c0 = time.perf_counter(), time.thread_time()
r = G.run("pagerank", max_iters=600)
t1, c1 = time.perf_counter(), time.thread_time()
print("share", (c1 - c0) / (t1 - t0), r.stats["iterations"])
"""


@pytest.mark.parametrize("flags", [4])
def test_blocking_waits_are_honoured(flags):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1806_08092_gb300 as gp
    gp.build()
    out = subprocess.run([sys.executable, "-c", PROGRAM, str(flags)], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr[-2000:]
    share, iterations = [x.split()[1:] for x in out.stdout.splitlines() if x.startswith("share")][0]
    assert int(iterations) == 600
    assert float(share) < 0.5, share
