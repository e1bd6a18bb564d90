"""What a process pays for its first handle, and kernels that are first used while a graph is being captured.  Each in a process of its
own: kernels are loaded once per process."""

import subprocess
import sys
from pathlib import Path

import pytest

pytestmark = pytest.mark.gpu

ROOT = Path(__file__).resolve().parent.parent

CREATE = """
import ctypes, sys, time
cuda, ctx = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p()
assert cuda.cuInit(0) == 0 and cuda.cuDevicePrimaryCtxRetain(ctypes.byref(ctx), 0) == 0 and cuda.cuCtxSetCurrent(ctx) == 0
lib, h = ctypes.CDLL(sys.argv[1]), ctypes.c_void_p()
start = time.perf_counter()
assert lib.slaq_create(8, 20, ctypes.byref(h)) == 0
print((time.perf_counter() - start) * 1e3)
lib.slaq_destroy(h)
"""

CAPTURE = """
import sys
sys.path.insert(0, sys.argv[1]); sys.path.insert(0, sys.argv[1] + "/tests")
import numpy as np, torch
import paper_1802_04819_b200 as slaq
from gpu_common import make_scheduler
from workloads import make_workload
wl = make_workload(2, n_jobs=int(sys.argv[2]))
a, stream = make_scheduler(wl), torch.cuda.Stream()
a.set_stream(stream)
out = torch.zeros(wl.n_jobs, dtype=torch.int32, device="cuda")
a.schedule_device(wl.epoch_seconds, wl.total_cores, out)
a.set_param(slaq.binding.P_WARM_START, 1)   # other kernels than the epoch before took
graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph, stream=stream):
    a.schedule_device(wl.epoch_seconds, wl.total_cores, out)
with torch.cuda.stream(stream):
    graph.replay()
stream.synchronize()
b = make_scheduler(wl)
b.schedule(wl.epoch_seconds, wl.total_cores)
b.set_param(slaq.binding.P_WARM_START, 1)
ref, _ = b.schedule(wl.epoch_seconds, wl.total_cores)
np.testing.assert_array_equal(out.cpu().numpy(), ref)
"""


def test_the_first_handle_of_a_process():
    """21 ms while there were 12 fit kernels; 29 with the 26 of three block sizes, all set up and their code unpacked from compressed
    form."""
    import paper_1802_04819_b200 as slaq
    slaq.build()
    lib = ROOT / "paper_1802_04819_b200" / "libslaq.so"
    ms = [float(subprocess.run([sys.executable, "-c", CREATE, str(lib)], check=True, capture_output=True, text=True,
                               timeout=120).stdout) for _ in range(4)]
    assert min(ms) < 20.0, ms


@pytest.mark.parametrize("jobs", [100, 4000, 20000])
def test_a_kernel_may_be_used_first_under_capture(jobs):
    subprocess.run([sys.executable, "-c", CAPTURE, str(ROOT), str(jobs)], check=True, timeout=300)
