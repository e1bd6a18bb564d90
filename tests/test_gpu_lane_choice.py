"""Lanes per job and slots per SM of the fit over its range of cluster sizes, against the oracle."""

import numpy as np
import pytest

from gpu_common import compare_epoch, make_scheduler, oracle_epoch
from workloads import make_workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def slaq():
    import paper_1802_04819_b200 as s
    s.build()
    return s


# Cluster sizes around one warp per SM (148), one per sub-partition (592), one slot per warp of the GPU (2368), and
# windows that make the rule take 32, 16, 8, 4 and 2 lanes, in one length class or in several.
@pytest.mark.parametrize("jobs, longest", [(1, 20), (149, 33), (593, 17), (1200, 5), (2369, 40), (2500, 300), (5000, 12),
                                           (9000, 41), (18000, 12)])
def test_every_choice_of_lanes_matches_the_oracle(slaq, oracle_mod, jobs, longest):
    rng = np.random.default_rng(jobs)
    lengths = rng.integers(3, longest + 1, size=jobs)
    lengths[0] = longest
    wl = make_workload(3, hist_lengths=[int(v) for v in lengths])
    sched = make_scheduler(wl)
    alloc, _ = sched.schedule(wl.epoch_seconds, wl.total_cores)
    counts = compare_epoch(alloc, sched.get_predictions(), oracle_epoch(oracle_mod, wl), wl.total_cores,
                           wl.max_cores_per_job)
    assert counts["jobs"] == jobs
