"""What is read back after an epoch belongs to that epoch, also where its launches wrote the gain table only as far as the
selection needed it (more than 2,048 gains per SM) and the handle's state has changed since."""

import numpy as np
import pytest

from gpu_common import make_scheduler
from workloads import make_workload

pytestmark = pytest.mark.gpu

JOBS = 6000      # x 64 cores: a streamed table


def _change(slaq, sched, wl, how):
    J = wl.n_jobs
    ids = np.arange(J, dtype=np.int32)
    last = wl.losses[wl.offsets[1:] - 1]
    if how == "append":
        for c in (1, 3):
            sched.append_losses(ids, 0.9 * last, 3.0 * (wl.s + wl.w / c), np.full(J, c, np.int32))
    elif how == "time law":
        sched.set_time_model(ids[::2], 2.0 * wl.s[::2], 0.5 * wl.w[::2])
    elif how == "target":
        sched.set_target_loss(ids[::2], last[::2])
    elif how == "envelope":
        sched.set_param(slaq.binding.P_GAIN_ENVELOPE, 1)
    elif how == "remove":
        sched.remove_jobs(ids[1::3])
    elif how == "load":
        sched.load_histories(ids, wl.offsets, wl.losses[::-1].copy(), wl.k_last, wl.m_seen)
    elif how == "fit state":
        st = sched.get_fit_state()
        sched.set_fit_state(dict(st, span=np.where(st["valid"] > 0, 2.0 * st["span"], st["span"])))


@pytest.mark.parametrize("law", ["fixed", "samples"])
@pytest.mark.parametrize("how", ["nothing", "append", "time law", "target", "envelope", "remove", "load", "fit state"])
def test_gain_rows_are_those_of_the_epoch(how, law):
    import paper_1802_04819_b200 as slaq
    slaq.build()
    wl = make_workload(4, n_jobs=JOBS)
    J, C = wl.n_jobs, 3 * JOBS
    ids = np.arange(J, dtype=np.int32)

    def one():
        s = make_scheduler(wl) if law == "fixed" else slaq.Scheduler(J, wl.max_hist, wl.max_cores_per_job)
        if law == "samples":     # a tenth of the jobs has no iteration times: they predict nothing
            s.load_histories(ids, wl.offsets, wl.losses, wl.k_last, wl.m_seen)
            last = wl.losses[wl.offsets[1:] - 1]
            some = ids[ids % 10 != 0]
            for c in (1, 4):
                s.append_losses(some, last[some], (wl.s + wl.w / c)[some], np.full(some.size, c, np.int32))
        return s, s.schedule(wl.epoch_seconds, C)[0]

    a, alloc = one()
    b, alloc_b = one()
    np.testing.assert_array_equal(alloc, alloc_b)
    want = a.get_predictions()
    np.testing.assert_array_equal(want["gain"], a.get_predictions()["gain"])
    taken = np.arange(wl.max_cores_per_job)[None, :] < alloc[:, None]
    np.testing.assert_allclose(np.where(taken, want["gain"], 0.0).sum(1), want["R"], rtol=1e-12)
    _change(slaq, a, wl, how)
    _change(slaq, b, wl, how)
    rest_a, got = a.get_predictions(want_gain=False), b.get_predictions()
    np.testing.assert_array_equal(got["gain"], want["gain"])
    for key in ("R", "status", "family", "params", "S", "evals", "M"):      # reading rows changes nothing else
        np.testing.assert_array_equal(got[key], rest_a[key])
    a.close()
    b.close()


def test_gain_rows_after_a_captured_epoch():
    """The caller's own graph: every replay is an epoch the host knows nothing of, its rows are read back all the same."""
    import torch
    import paper_1802_04819_b200 as slaq
    slaq.build()
    wl = make_workload(4, n_jobs=JOBS)
    J, C = wl.n_jobs, 3 * JOBS
    last = wl.losses[wl.offsets[1:] - 1]
    ids = np.arange(J, dtype=np.int32)
    stream = torch.cuda.Stream()
    a, b = make_scheduler(wl), make_scheduler(wl)
    a.set_stream(stream)
    out = torch.zeros(J, dtype=torch.int32, device="cuda")
    a.schedule_device(wl.epoch_seconds, C, out)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        a.schedule_device(wl.epoch_seconds, C, out)
    for step in range(3):
        for s in (a, b):
            s.append_losses(ids, (0.97 - 0.01 * step) * last, 2.0 * wl.s, np.ones(J, np.int32))
        with torch.cuda.stream(stream):
            graph.replay()
        stream.synchronize()
        ref, _ = b.schedule(wl.epoch_seconds, C)
        np.testing.assert_array_equal(out.cpu().numpy(), ref)
        got, want = a.get_predictions(), b.get_predictions()
        for key in ("gain", "R", "params", "status"):
            np.testing.assert_array_equal(got[key], want[key])
    # a table the caller sets afterwards is the table
    gain = np.sort(np.random.default_rng(1).random((J, wl.max_cores_per_job)), 1)[:, ::-1].copy()
    a.set_gains(gain)
    np.testing.assert_array_equal(a.get_predictions()["gain"], gain)
    a.close()
    b.close()


def _definition(gain, C):
    J, cap = gain.shape
    floor = 1 if C >= J else 0
    want = min(C, J * cap) - floor * J
    order = np.argsort(-gain[:, floor:].ravel(), kind="stable")[:want]
    return (floor + np.bincount(order // (cap - floor), minlength=J)).astype(np.int32)


@pytest.mark.parametrize("change", [False, True])
def test_allocate_only_reads_the_whole_rows_of_the_epoch(change):
    import paper_1802_04819_b200 as slaq
    slaq.build()
    wl = make_workload(4, n_jobs=JOBS)
    twin, s = make_scheduler(wl), make_scheduler(wl)
    for h in (twin, s):
        h.schedule(wl.epoch_seconds, 2 * JOBS)
    gain = twin.get_predictions()["gain"]
    if change:
        _change(slaq, s, wl, "time law")
    for C in (20 * JOBS, 40 * JOBS, 2 * JOBS, JOBS // 2):
        alloc, _ = s.allocate_only(C)
        np.testing.assert_array_equal(alloc, _definition(gain, C))
    np.testing.assert_array_equal(s.get_predictions()["gain"], gain)
    twin.close()
    s.close()


def test_rows_the_caller_sets_stay_after_an_epoch():
    import paper_1802_04819_b200 as slaq
    slaq.build()
    wl = make_workload(4, n_jobs=JOBS)
    gain = np.sort(np.random.default_rng(7).random((JOBS, wl.max_cores_per_job)), 1)[:, ::-1].copy()
    s = make_scheduler(wl)
    s.schedule(wl.epoch_seconds, 2 * JOBS)
    s.set_gains(gain)
    np.testing.assert_array_equal(s.get_predictions()["gain"], gain)
    for C in (3 * JOBS, 30 * JOBS):
        np.testing.assert_array_equal(s.allocate_only(C)[0], _definition(gain, C))
    s.close()
