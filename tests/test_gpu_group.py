"""Several handles of one GPU scheduled together (slaq_schedule_group), step by step, and one handle holding all jobs: the
same allocation, reductions and tie order from all three.  Integer work and identical sums, so bit for bit."""

import numpy as np
import pytest

from workloads import make_workload

pytestmark = pytest.mark.gpu


def _handle(slaq, wl, lo, hi):
    ids = np.arange(hi - lo, dtype=np.int32)
    s = slaq.Scheduler(hi - lo, wl.max_hist, wl.max_cores_per_job)
    s.load_histories(ids, wl.offsets[lo:hi + 1] - wl.offsets[lo], wl.losses[wl.offsets[lo]:wl.offsets[hi]], wl.k_last[lo:hi],
                     wl.m_seen[lo:hi])
    s.set_time_model(ids, wl.s[lo:hi], wl.w[lo:hi])
    return s


# rows resident in shared memory; a streamed table cut unevenly; the most handles one call takes, and one more
@pytest.mark.parametrize("cfg,n_jobs,cuts", [
    (1, None, [0, 1, 160]), (2, 3000, [0, 17, 2999, 3000]), (4, 9000, [0, 4000, 9000]), (4, 40000, [0, 39000, 39001, 40000]),
    (2, 1600, list(range(0, 1601, 200))), (1, None, [0, 3, 20, 40, 60, 80, 100, 120, 140, 160])])
def test_handles_of_one_gpu(cfg, n_jobs, cuts):
    import paper_1802_04819_b200 as slaq
    slaq.build()

    class Steps(slaq.LocalExchange):   # not the class itself: schedule_sharded goes through the steps
        pass

    wl = make_workload(cfg, n_jobs=n_jobs)
    J, cap = wl.n_jobs, wl.max_cores_per_job
    whole = _handle(slaq, wl, 0, J)
    shards = [_handle(slaq, wl, lo, hi) for lo, hi in zip(cuts[:-1], cuts[1:])]
    for C in (wl.total_cores, 0, J - 1, J, J * cap // 2, J * cap + 1):
        ref, _ = whole.schedule(wl.epoch_seconds, C)
        R = whole.get_predictions(want_gain=False)["R"]
        for exchange in (slaq.LocalExchange(), Steps(), slaq.LocalExchange()):
            parts = slaq.schedule_sharded(shards, exchange, wl.epoch_seconds, C)
            np.testing.assert_array_equal(np.concatenate(parts), ref)
            got = np.concatenate([s.get_predictions(want_gain=False)["R"] for s in shards])
            np.testing.assert_array_equal(got, R)
            stats = [s.get_stats() for s in shards]
            assert sum(t.cores_handed_out for t in stats) == min(C, J * cap)
    for s in shards:       # a member of a group schedules alone afterwards
        s.set_param(slaq.binding.P_FIT_CLUSTER_JOBS, 0)
        alloc, _ = s.schedule(wl.epoch_seconds, 2 * s.max_jobs)
        assert alloc.sum() == min(2, cap) * s.max_jobs


# rows that end at and beside a multiple of the gains in flight together, and at the largest cap
@pytest.mark.parametrize("cap,per_job", [(33, 30), (48, 44), (49, 47), (1024, 300), (1024, 900)])
def test_steps_add_long_rows_as_one_handle_does(cap, per_job):
    import paper_1802_04819_b200 as slaq
    slaq.build()

    class Steps(slaq.LocalExchange):
        pass

    wl = make_workload(4, n_jobs=700)
    J = wl.n_jobs

    def handle(lo, hi):
        ids = np.arange(hi - lo, dtype=np.int32)
        s = slaq.Scheduler(hi - lo, wl.max_hist, cap)
        s.load_histories(ids, wl.offsets[lo:hi + 1] - wl.offsets[lo], wl.losses[wl.offsets[lo]:wl.offsets[hi]], wl.k_last[lo:hi],
                         wl.m_seen[lo:hi])
        s.set_time_model(ids, wl.s[lo:hi], wl.w[lo:hi])
        return s

    whole, shards = handle(0, J), [handle(0, 257), handle(257, J)]
    for C in (per_job * J, J * cap - 1, J * cap):
        ref, _ = whole.schedule(wl.epoch_seconds, C)
        parts = slaq.schedule_sharded(shards, Steps(), wl.epoch_seconds, C)
        np.testing.assert_array_equal(np.concatenate(parts), ref)
        assert ref.max() > 32
        got = np.concatenate([s.get_predictions(want_gain=False)["R"] for s in shards])
        np.testing.assert_array_equal(got, whole.get_predictions(want_gain=False)["R"])


def test_a_group_refuses_what_it_cannot_do():
    import paper_1802_04819_b200 as slaq
    from paper_1802_04819_b200.binding import P_GAIN_ENVELOPE, schedule_group
    wl = make_workload(1)
    a, b = _handle(slaq, wl, 0, 80), _handle(slaq, wl, 80, 160)
    with pytest.raises(slaq.SlaqError):
        schedule_group([a, a], 1.0, 100)
    with pytest.raises(slaq.SlaqError):
        schedule_group([a, b], 0.0, 100)
    b.set_param(P_GAIN_ENVELOPE, 1)
    assert schedule_group([a, b], 1.0, 100) is None
