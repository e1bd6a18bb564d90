"""Windows on both sides of the limits of the fit's lane classes (118, 260 and 544 points at twelve warps): in the bounds build, and where no
curve can be started."""

import numpy as np
import pytest

from fit_plan import fit_plan
from gpu_common import compare_epoch
from test_gpu_bounds_build import _epoch, slaq  # noqa: F401  (fixture: the library and its bounds build)
from workloads import make_unfittable_histories, make_workload

pytestmark = pytest.mark.gpu

EDGES = [4, 5, 33, 64, 117, 118, 119, 259, 260, 261, 543, 544, 545, 1000]


@pytest.mark.parametrize("cluster_jobs", [0, 10_000_000])
def test_no_index_leaves_its_extent(slaq, cluster_jobs):
    assert [high for _, _, high in fit_plan(1000, 10_000_000)[2]] == [1000, 544, 260, 118]
    wl = make_workload(3, hist_lengths=EDGES * 50)
    params = ((slaq.binding.P_FIT_CLUSTER_JOBS, cluster_jobs),)
    checked, plain = _epoch(slaq, wl, "bounds", True, params), _epoch(slaq, wl, None, True, params)
    np.testing.assert_array_equal(checked[0], plain[0])
    for key in ("gain", "params", "S", "R", "status", "M"):
        np.testing.assert_array_equal(checked[1][key], plain[1][key])


@pytest.mark.parametrize("cluster_jobs", [0, 10_000_000])
def test_windows_without_a_usable_start(slaq, oracle_mod, cluster_jobs):
    """The windows between ordinary ones, every class among them: predicted from their mean change, as the oracle does."""
    offsets, losses, m_seen, _ = make_unfittable_histories(EDGES, "staircase", seed=1)
    wl = make_workload(3, hist_lengths=[7, 40, 90, 300, 600, 950] * 12)
    half, bad = wl.n_jobs // 2, len(EDGES)
    pieces = [(wl.offsets[:half + 1], wl.losses[:wl.offsets[half]], wl.m_seen[:half]), (offsets, losses, m_seen),
              (wl.offsets[half:] - wl.offsets[half], wl.losses[wl.offsets[half]:], wl.m_seen[half:])]
    H = np.concatenate([np.diff(o) for o, _, _ in pieces])
    offsets = np.concatenate([[0], np.cumsum(H)]).astype(np.int64)
    losses, m_seen = (np.concatenate([p[i] for p in pieces]) for i in (1, 2))
    J, cap = H.size, 16
    rng = np.random.default_rng(5)
    s, w = rng.uniform(0.05, 0.5, J), rng.uniform(1.0, 100.0, J)
    sched, ids = slaq.Scheduler(J, 1000, cap), np.arange(J, dtype=np.int32)
    sched.load_histories(ids, offsets, losses, H.astype(np.int64) - 1, m_seen, packed=True)
    sched.set_time_model(ids, s, w)
    sched.set_param(slaq.binding.P_FIT_CLUSTER_JOBS, cluster_jobs)
    alloc, _ = sched.schedule(1.0, 4 * J)
    pred = sched.get_predictions()
    compare_epoch(alloc, pred, oracle_mod.schedule(offsets, losses, m_seen, s, w, 1.0, 4 * J, cap), 4 * J, cap)
    failed = (ids >= half) & (ids < half + bad)
    np.testing.assert_array_equal(pred["status"], np.where(failed, slaq.JOB_FIT_FAILED, slaq.JOB_FITTED))


@pytest.mark.parametrize("capacity", [700, 17_000])
def test_the_work_list_at_the_longest_windows(slaq, capacity):
    """One block sorts, or a block per 2,048 ids, with bins for 6,000 lengths: the results are those of the unsorted fit."""
    wl = make_workload(3, hist_lengths=[6000, 5999, 3001, 1000, 400, 100, 20, 4])
    ref = slaq.Scheduler(wl.n_jobs, 6000, wl.max_cores_per_job)
    listed = slaq.Scheduler(capacity, 6000, wl.max_cores_per_job)
    ids = np.arange(wl.n_jobs, dtype=np.int32)
    for sched in (ref, listed):
        sched.load_histories(ids, wl.offsets, wl.losses, wl.k_last, wl.m_seen)
        sched.set_time_model(ids, wl.s, wl.w)
    want, _ = ref.schedule(wl.epoch_seconds, wl.total_cores)
    alloc, _ = listed.schedule(wl.epoch_seconds, wl.total_cores)
    np.testing.assert_array_equal(alloc[ids], want)
    assert alloc[wl.n_jobs:].sum() == 0
    for key in ("params", "S", "gain", "R", "status"):
        np.testing.assert_array_equal(listed.get_predictions()[key][ids], ref.get_predictions()[key])
