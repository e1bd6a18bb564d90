"""Selection over rows predicted down to a bound that a sample of them gives: the allocation is the literal greedy loop's over the gains
of the same epoch, bit for bit, also where the sample misleads."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

JOBS = 61_000      # the kernel samples from 60,000 rows on


def _sampled_rows(jobs, sm_count):
    """The rows the kernel's blocks look at first (predict_to_bound in slaq_select.cu)."""
    rows = -(-jobs // sm_count)
    out = []
    for block, j0 in enumerate(range(0, jobs, rows)):
        n = min(rows, jobs - j0)
        k = min(n, max(32, n // 64))
        r = np.arange(k, dtype=np.int64)
        mix = ((r * 2654435761 + block * 40503) & 0xffffffff) % n
        out.append(j0 + (r * n + mix) // k)
    return np.concatenate(out)


@pytest.mark.parametrize("who_falls", ["some", "the sample", "all but the sample", "nobody"])
@pytest.mark.parametrize("cap,cores_per_job", [(17, 3.0), (64, 4.0), (64, 0.5), (64, 63.9), (33, 1.0), (128, 1.02)])
def test_allocation_is_the_greedy_loops(oracle_mod, who_falls, cap, cores_per_job):
    import torch
    import paper_1802_04819_b200 as slaq
    rng = np.random.default_rng(5)
    rows = _sampled_rows(JOBS, torch.cuda.get_device_properties(0).multi_processor_count)
    falls = np.zeros(JOBS, bool)
    if who_falls == "some":
        falls[rng.choice(JOBS, JOBS // 10, replace=False)] = True
    elif who_falls == "the sample":
        falls[rows] = True
    elif who_falls == "all but the sample":
        falls[:] = True
        falls[rows] = False
    H = 6
    k = np.arange(H)
    rate = rng.uniform(0.05, 0.5, JOBS)[:, None]
    steep = np.exp(-rate * k) * np.exp(0.01 * rng.standard_normal((JOBS, H)))
    flat = 0.3 * (1.0 + 1e-6 * rng.standard_normal((JOBS, H)))       # has converged: next to nothing to gain
    losses = np.where(falls[:, None], steep, flat)
    losses[::7, 0] = losses[::7, 1]                                  # and some windows alike
    losses[7::7] = losses[:-7:7][: losses[7::7].shape[0]] if who_falls == "nobody" else losses[7::7]
    s = slaq.Scheduler(JOBS, H, cap)
    ids = np.arange(JOBS, dtype=np.int32)
    s.load_histories(ids, np.arange(JOBS + 1, dtype=np.int64) * H, losses.ravel(), np.full(JOBS, 50, np.int64), np.ones(JOBS))
    s.set_time_model(ids, np.full(JOBS, 0.05), rng.uniform(0.5, 20.0, JOBS))
    s.remove_jobs(ids[5::911])
    cores = int(cores_per_job * JOBS)
    for _ in range(2):                                               # the launch leaves its scratch as it found it
        alloc, _ = s.schedule(1.0, cores)
    p = s.get_predictions(want_gain=True)
    active = np.ones(JOBS, np.uint8)
    active[5::911] = 0
    want = oracle_mod.allocate(p["gain"], active, cores)
    np.testing.assert_array_equal(alloc, want)
    direct = np.where(np.arange(cap)[None, :] < alloc[:, None], p["gain"], 0.0).sum(axis=1)
    np.testing.assert_allclose(p["R"], direct, rtol=1e-12, atol=1e-15)   # sums of up to 128 terms in another order
    assert s.get_stats().cores_handed_out == alloc.sum()
