"""The library's plans (slaq_fit_plan.cuh, slaq_select_plan.cuh), compiled for the host."""

import ctypes
import functools
import subprocess
import tempfile
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_1802_04819_b200" / "csrc"

SOURCE = r"""
#include "slaq_fit_plan.cuh"
#include "slaq_select_plan.cuh"
extern "C" void plan(int max_hist, long long jobs, int sm_count, long long slice_bytes, int* out) {
    const slaq::FitPlan p = slaq::fit_plan(max_hist, jobs, sm_count, (size_t)slice_bytes);
    const slaq::FitClasses c = slaq::fit_classes(max_hist, p);
    out[0] = slaq::kFitWarps[p.kind], out[1] = p.lanes, out[2] = c.n, out[3] = c.slice;
    for (int i = 0; i < slaq::kMaxFitClasses; ++i) out[4 + 3 * i] = c.h_lo[i], out[5 + 3 * i] = c.h_hi[i], out[6 + 3 * i] = c.L[i];
}
extern "C" int bounded(long long jobs, int cap, long long want, int sm_count) {
    return slaq::select_bounded(jobs, cap, want, sm_count, sm_count);
}
"""


@functools.lru_cache(maxsize=1)
def _library():
    with tempfile.TemporaryDirectory(prefix="fit_plan") as where:
        source, so = Path(where) / "plan.cpp", Path(where) / "plan.so"
        source.write_text(SOURCE)
        subprocess.run(["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-I", str(CSRC), "-o", str(so), str(source)], check=True)
        return ctypes.CDLL(str(so))


def fit_plan(max_hist, jobs, sm_count=148, slice_bytes=13824):
    """(warps of a block, least lanes, classes as (lanes, windows longer than, up to), doubles of a warp's slice)."""
    out = (ctypes.c_int * 28)()
    _library().plan(int(max_hist), ctypes.c_longlong(int(jobs)), int(sm_count), ctypes.c_longlong(int(slice_bytes)), out)
    classes = [(out[6 + 3 * i], out[4 + 3 * i], out[5 + 3 * i]) for i in range(out[2])]
    return out[0], out[1], classes, out[3]


def select_bounded(jobs, cap, cores, sm_count=148):
    """Whether a selection of so many rows, all of them active, predicts them down to a bound from a sample."""
    want = min(int(cores), jobs * cap) - (jobs if cores >= jobs else 0)
    return bool(_library().bounded(ctypes.c_longlong(jobs), int(cap), ctypes.c_longlong(want), int(sm_count)))
