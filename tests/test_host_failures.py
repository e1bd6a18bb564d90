"""Host code of the library where something fails: built against a CUDA runtime that only pretends (host_fakes/), so that launches
and allocations fail when a test says so and no GPU is needed."""

import ctypes
import shutil
import subprocess
from ctypes import byref, c_double, c_int, c_int32, c_int64, c_long, c_size_t, c_void_p
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parent.parent
CSRC = ROOT / "paper_1802_04819_b200" / "csrc"


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    where = tmp_path_factory.mktemp("fake")
    inc = ["-I", str(ROOT / "include"), "-I", str(CSRC), "-I", str(Path(shutil.which("nvcc")).resolve().parent.parent / "include")]
    fakes = ROOT / "tests" / "host_fakes"
    objects = []
    for source in (CSRC / "slaq_api.cu", CSRC / "slaq_pipe.cu", fakes / "fake_launches.cu", fakes / "fake_cuda.cpp"):
        objects.append(str(where / (source.stem + ".o")))
        cuda = ["nvcc", "-gencode", "arch=compute_100a,code=sm_100a", "-cudart", "none", "-Xcompiler"]
        compiler = cuda if source.suffix == ".cu" else ["g++"]
        subprocess.run([*compiler, "-fPIC", "-O1", "-std=c++17", *inc, "-c", str(source), "-o", objects[-1]], check=True)
    so = where / "libfake.so"
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", str(so), *objects, "-lpthread"], check=True)
    return ctypes.CDLL(str(so))


def _handle(lib, jobs=8):
    h = c_void_p()
    assert lib.slaq_create_in(None, c_size_t(0), c_int32(jobs), c_int32(16), c_int32(4), byref(h)) == 0
    return h


def _clears(lib):
    return c_size_t.in_dll(lib, "fake_clears").value


def _epoch(lib, h):
    return lib.slaq_schedule_device(h, c_double(1.0), c_int64(8), None)


def test_the_epoch_after_one_that_could_not_be_launched_clears_its_scratch(lib):
    h = _handle(lib)
    before = _clears(lib)
    assert _epoch(lib, h) == 2 and _clears(lib) == before          # no active jobs: underfilled; nothing to clear
    c_int.in_dll(lib, "fake_fail_select").value = 1
    assert _epoch(lib, h) == -5                                    # the fit was queued, the selection was not
    assert _epoch(lib, h) == 2
    assert _clears(lib) == before + 1
    assert _epoch(lib, h) == 2 and _clears(lib) == before + 1
    lib.slaq_destroy(h)


@pytest.mark.parametrize("failure", ["launch", "report"])
def test_every_handle_of_a_group_that_failed_clears_its_scratch(lib, failure):
    hs = [_handle(lib) for _ in range(3)]
    rows = [(c_int32 * 8)() for _ in hs]
    handles, out = (c_void_p * 3)(*[h.value for h in hs]), (c_void_p * 3)(*[ctypes.addressof(r) for r in rows])

    def group():
        return lib.slaq_schedule_group(handles, c_int32(3), c_double(1.0), c_int64(24), out)

    assert group() == 2
    before = _clears(lib)
    assert group() == 2 and _clears(lib) == before
    if failure == "launch":
        c_int.in_dll(lib, "fake_fail_select").value = 1
    else:
        c_int.in_dll(lib, "fake_err_word").value = 1               # the launch ran, and some block found an inconsistency
    assert group() == -5
    before = _clears(lib)
    for h in hs:                                                   # each member's next epoch, alone
        assert _epoch(lib, h) == 2
    assert _clears(lib) == before + 3
    for h in hs:
        lib.slaq_destroy(h)


def test_a_bulk_copy_without_memory_for_its_lists_is_an_error(lib):
    """No C entry throws: every allocation of a load and of its copies (threads among them) is let fail in turn."""
    jobs, points = 8, 9_000_000                                    # enough for the page-locked buffers of the copies
    h = c_void_p()
    assert lib.slaq_create_in(None, c_size_t(0), c_int32(jobs), c_int32(16), c_int32(4), byref(h)) == 0
    losses = (c_double * points)()
    ids, k_last = (c_int32 * jobs)(*range(jobs)), (c_int64 * jobs)(*[points // jobs] * jobs)
    offsets = (c_int64 * (jobs + 1))(*[points // jobs * j for j in range(jobs + 1)])
    fails = c_long.in_dll(lib, "fake_new_fails_in")
    kernels = c_int.in_dll(lib, "fake_device_kernels")
    results = set()
    for at in range(1, 25):
        fails.value = at
        before = kernels.value
        rc = lib.slaq_load_histories(h, c_int32(jobs), ids, offsets, losses, k_last, None)
        left, fails.value = fails.value, 0
        results.add((rc, left > 0))
        # the fake runs no kernel, so a load that got that far reports that its own did not come to an end
        assert rc == (-5 if kernels.value > before else -4)
    assert (-4, False) in results and (-5, False) in results and (-5, True) in results
    lib.slaq_result_take.restype = c_void_p
    for at in range(1, 12):
        fails.value = 1
        block = lib.slaq_result_take(c_size_t(70000 + 131072 * at))
        assert block is None
    fails.value = 0
    lib.slaq_destroy(h)
