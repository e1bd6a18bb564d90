"""Selection over rows predicted down to a bound that a sample of them gives: each case says whether the sample is taken (the rule is the
library's own, compiled for the host) and whether it misleads, for one handle and for a group of shards."""

import numpy as np
import pytest

from fit_plan import select_bounded

pytestmark = pytest.mark.gpu

JOBS = 61_000      # the kernel samples from 60,000 rows on


def _sampled_rows(jobs, sm_count, cuts=None):
    """The rows the kernel's blocks look at first (predict_to_bound in slaq_select.cu), of one handle or of several cut at `cuts`."""
    cuts = cuts or [0, jobs]
    shards = list(zip(cuts[:-1], cuts[1:]))
    rows = -(-jobs // sm_count)
    while sum(-(-(hi - lo) // rows) for lo, hi in shards) > sm_count:
        rows += 1
    out, block = [], 0
    for lo, hi in shards:
        for j0 in range(lo, hi, rows):
            n = min(rows, hi - j0)
            k = min(n, max(32, n // 64))
            r = np.arange(k, dtype=np.int64)
            mix = ((r * 2654435761 + block * 40503) & 0xffffffff) % n
            out.append(j0 + (r * n + mix) // k)
            block += 1
    return np.concatenate(out)


def _misled(gain, active, rows, cores):
    """Whether that sample's bound (64 bins per power of two) leaves fewer gains than are wanted."""
    J, cap = gain.shape
    floor = 1 if cores >= active.sum() else 0
    want = min(cores, int(active.sum()) * cap) - floor * int(active.sum())
    keys = np.ascontiguousarray(gain).view(np.int64) >> 46
    least = (1023 - 31) * 64 + 1                            # the first bin keeps what is smaller
    seen = keys[rows][active[rows] > 0][:, floor:].ravel()
    seen = np.sort(seen[seen >= least])[::-1]
    rank = want * (rows.size / J)
    rank = int(rank + 5.0 * np.sqrt(cap * rank) + 8.0)
    bound = min(seen[rank - 1], least + 32 * 64 - 2) if rank <= seen.size else 0
    return int((keys[active > 0][:, floor:] >= bound).sum()) < want


def _losses(rng, jobs, rows, who_falls):
    falls = np.zeros(jobs, bool)
    if who_falls == "some":
        falls[rng.choice(jobs, jobs // 10, replace=False)] = True
    elif who_falls == "the sample":
        falls[rows] = True
    elif who_falls == "all but the sample":
        falls[:] = True
        falls[rows] = False
    H = 6
    k = np.arange(H)
    rate = rng.uniform(0.05, 0.5, jobs)[:, None]
    steep = np.exp(-rate * k) * np.exp(0.01 * rng.standard_normal((jobs, H)))
    flat = 0.3 * (1.0 + 1e-6 * rng.standard_normal((jobs, H)))       # has converged: next to nothing to gain
    losses = np.where(falls[:, None], steep, flat)
    losses[::7, 0] = losses[::7, 1]                                  # and some windows alike
    losses[7::7] = losses[:-7:7][: losses[7::7].shape[0]] if who_falls == "nobody" else losses[7::7]
    return losses


def _handle(slaq, losses, w, cap, variant=None):
    jobs, H = losses.shape
    s = slaq.Scheduler(jobs, H, cap, variant=variant)
    ids = np.arange(jobs, dtype=np.int32)
    s.load_histories(ids, np.arange(jobs + 1, dtype=np.int64) * H, losses.ravel(), np.full(jobs, 50, np.int64), np.ones(jobs))
    s.set_time_model(ids, np.full(jobs, 0.05), w)
    return s


@pytest.mark.parametrize("who_falls", ["some", "the sample", "all but the sample", "nobody"])
@pytest.mark.parametrize("cap,cores_per_job,jobs,bounded", [
    (17, 3.0, JOBS, True), (64, 4.0, JOBS, True), (64, 0.5, JOBS, True), (64, 63.9, JOBS, False), (33, 1.0, JOBS, True),
    (128, 1.02, JOBS, False), (128, 1.02, 100_000, True), (128, 25.0, JOBS, True)])
def test_allocation_is_the_greedy_loops(oracle_mod, who_falls, cap, cores_per_job, jobs, bounded):
    import torch
    import paper_1802_04819_b200 as slaq
    sm_count = torch.cuda.get_device_properties(0).multi_processor_count
    cores = int(cores_per_job * jobs)
    assert select_bounded(jobs, cap, cores, sm_count) == bounded
    rng = np.random.default_rng(5)
    rows = _sampled_rows(jobs, sm_count)
    losses = _losses(rng, jobs, rows, who_falls)
    s = _handle(slaq, losses, rng.uniform(0.5, 20.0, jobs), cap)
    ids = np.arange(jobs, dtype=np.int32)
    s.remove_jobs(ids[5::911])
    for _ in range(2):                                               # the launch leaves its scratch as it found it
        alloc, _ = s.schedule(1.0, cores)
    p = s.get_predictions(want_gain=True)
    active = np.ones(jobs, np.uint8)
    active[5::911] = 0
    want = oracle_mod.allocate(p["gain"], active, cores)
    np.testing.assert_array_equal(alloc, want)
    direct = np.where(np.arange(cap)[None, :] < alloc[:, None], p["gain"], 0.0).sum(axis=1)
    np.testing.assert_allclose(p["R"], direct, rtol=1e-12, atol=1e-15)   # sums of up to 128 terms in another order
    assert s.get_stats().cores_handed_out == alloc.sum()
    if bounded:
        # where the jobs' floor leaves a few dozen cores the margin is wider than what is wanted
        assert _misled(p["gain"], active, rows, cores) == (who_falls == "the sample" and cores_per_job != 1.0)


@pytest.mark.parametrize("variant", [None, "bounds"])
@pytest.mark.parametrize("who_falls", ["some", "the sample"])
def test_a_group_is_allocated_as_one_handle(who_falls, variant):
    """Shards of one GPU, one of them shorter than a block's rows; the bounds build checks every index."""
    import torch
    import paper_1802_04819_b200 as slaq
    from paper_1802_04819_b200.build import build_variant
    if variant:
        build_variant(variant)
    sm_count = torch.cuda.get_device_properties(0).multi_processor_count
    cap, cores, cuts = 33, 3 * JOBS, [0, 40_000, 40_100, JOBS]
    assert select_bounded(JOBS, cap, cores, sm_count)
    rng = np.random.default_rng(6)
    rows = _sampled_rows(JOBS, sm_count, cuts)
    losses, w = _losses(rng, JOBS, rows, who_falls), rng.uniform(0.5, 20.0, JOBS)
    whole = _handle(slaq, losses, w, cap, variant)
    shards = [_handle(slaq, losses[lo:hi], w[lo:hi], cap, variant) for lo, hi in zip(cuts[:-1], cuts[1:])]
    ref, _ = whole.schedule(1.0, cores)
    p = whole.get_predictions(want_gain=True)
    assert _misled(p["gain"], np.ones(JOBS, np.uint8), rows, cores) == (who_falls == "the sample")
    for _ in range(2):
        parts = slaq.schedule_sharded(shards, slaq.LocalExchange(), 1.0, cores)
        np.testing.assert_array_equal(np.concatenate(parts), ref)
    np.testing.assert_array_equal(np.concatenate([s.get_predictions(want_gain=False)["R"] for s in shards]), p["R"])
    assert sum(s.get_stats().cores_handed_out for s in shards) == cores
