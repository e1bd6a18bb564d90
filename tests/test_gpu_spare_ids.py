"""Handles with ids to spare: a job's fit depends on its history and on the cluster's active jobs, not on how many ids the
handle was made for, so a cluster in shards equals the undivided one bit for bit whatever their capacities are."""

import numpy as np
import pytest

from workloads import make_workload

pytestmark = pytest.mark.gpu


def _handle(slaq, wl, lo, hi, capacity, spread, window=None):
    s = slaq.Scheduler(capacity, window or wl.max_hist, wl.max_cores_per_job)
    ids = (np.arange(hi - lo, dtype=np.int32) * spread).astype(np.int32)
    s.load_histories(ids, wl.offsets[lo:hi + 1] - wl.offsets[lo], wl.losses[wl.offsets[lo]:wl.offsets[hi]], wl.k_last[lo:hi],
                     wl.m_seen[lo:hi])
    s.set_time_model(ids, wl.s[lo:hi], wl.w[lo:hi])
    return s, ids


# Teams of one warp per family (windows of up to 512) and of several, windows that fit a part of a warp; capacities from the
# first at which a block per id is not taken, over a list made by one block, to more ids than one block sorts.
@pytest.mark.parametrize("jobs,longest,capacity,window", [
    (400, 60, 1000, 60), (160, 40, 4000, 300), (580, 16, 600, 16), (12, 5, 2000, 5), (30, 900, 3000, 1000), (140, 700, 593, 1000),
    (8, 33, 20000, 1000), (8, 33, 20000, 33), (1, 4, 593, 4)])
def test_shards_equal_the_whole_at_any_capacity(jobs, longest, capacity, window):
    import paper_1802_04819_b200 as slaq
    from paper_1802_04819_b200.binding import P_WARM_START
    slaq.build()

    class Steps(slaq.LocalExchange):   # not the class itself: schedule_sharded goes through the steps
        pass

    rng = np.random.default_rng(jobs)
    lengths = rng.integers(3, longest + 1, size=jobs)
    lengths[0] = longest
    wl = make_workload(3, hist_lengths=[int(v) for v in lengths])
    C, cut = 3 * jobs + 1, (jobs + 1) // 2
    whole, ids = _handle(slaq, wl, 0, jobs, capacity, capacity // jobs, window)
    full, _ = _handle(slaq, wl, 0, jobs, jobs, 1, window)
    parts = [_handle(slaq, wl, lo, hi, n, 1, window)
             for lo, hi, n in ((0, cut, max(cut, 300)), (cut, jobs, max(jobs - cut, capacity // 2))) if hi > lo]
    for warm in (0, 1):
        for s in [whole, full] + [p for p, _ in parts]:
            s.set_param(P_WARM_START, warm)
        alloc, _ = whole.schedule(wl.epoch_seconds, C)
        ref = whole.get_predictions()
        assert alloc.sum() == min(C, jobs * wl.max_cores_per_job) and whole.get_stats().points == int(lengths.sum())
        alloc_full, _ = full.schedule(wl.epoch_seconds, C)
        got = full.get_predictions()
        np.testing.assert_array_equal(alloc_full, alloc[ids])
        for key in ("params", "S", "gain", "R", "status", "evals"):
            np.testing.assert_array_equal(got[key], ref[key][ids])
        for exchange in (Steps(), slaq.LocalExchange()):
            allocs = slaq.schedule_sharded([p for p, _ in parts], exchange, wl.epoch_seconds, C)
            at = 0
            for (p, mine), al in zip(parts, allocs):
                there = ids[at: at + mine.size]
                at += mine.size
                np.testing.assert_array_equal(al[mine], alloc[there])
                got = p.get_predictions()
                for key in ("params", "S", "gain", "R", "status", "evals"):
                    np.testing.assert_array_equal(got[key][mine], ref[key][there])
        last = wl.losses[wl.offsets[1:] - 1]
        whole.append_losses(ids, 0.9 * last)
        full.append_losses(np.arange(jobs), 0.9 * last)
        at = 0
        for p, mine in parts:
            p.append_losses(mine, 0.9 * last[at: at + mine.size])
            at += mine.size
        lengths = np.minimum(lengths + 1, window)
    for s in [whole, full] + [p for p, _ in parts]:
        s.close()


@pytest.mark.parametrize("window", [200, 1000])
def test_jobs_that_arrive_after_a_capture_are_fitted(window):
    """The launches of a captured epoch cover every id of the handle, not the jobs there were."""
    import torch
    import paper_1802_04819_b200 as slaq
    slaq.build()
    wl = make_workload(2, n_jobs=300)
    stream = torch.cuda.Stream()
    s, ids = _handle(slaq, wl, 0, 20, 5000, 1, window)
    s.set_stream(stream)
    out = torch.zeros(5000, dtype=torch.int32, device="cuda")
    s.schedule_device(3.0, 5000, out)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        s.schedule_device(3.0, 5000, out)
    more = np.arange(20, 300, dtype=np.int32)
    s.load_histories(more, wl.offsets[20:] - wl.offsets[20], wl.losses[wl.offsets[20]:], wl.k_last[20:], wl.m_seen[20:])
    s.set_time_model(more, wl.s[20:], wl.w[20:])
    with torch.cuda.stream(stream):
        graph.replay()
    stream.synchronize()
    pred = s.get_predictions(want_gain=False)
    assert (pred["status"][:300] >= 0).all() and (pred["status"][300:] == -1).all()
    assert s.get_stats().points == int(wl.offsets[-1])
    s.close()
