"""The fit with a block per job, over the sizes at which its teams of warps change, against the oracle."""

import numpy as np
import pytest

from gpu_common import compare_epoch, make_scheduler, oracle_epoch
from workloads import make_workload

pytestmark = pytest.mark.gpu


# one, two and four warps per family; windows that end a row, a part's rows, or leave lanes and parts without any
@pytest.mark.parametrize("jobs, longest", [(1, 4), (2, 32), (5, 33), (40, 128), (40, 129), (74, 257), (75, 258), (148, 513),
                                           (149, 768), (296, 385), (297, 512), (592, 65), (7, 6000)])
def test_teams_match_the_oracle(oracle_mod, jobs, longest):
    import paper_1802_04819_b200 as slaq
    slaq.build()
    rng = np.random.default_rng(100 * jobs + longest)
    lengths = rng.integers(3, longest + 1, size=jobs)
    lengths[0] = longest
    wl = make_workload(3, hist_lengths=[int(v) for v in lengths])
    sched = make_scheduler(wl, packed=jobs % 2 == 0)
    alloc, _ = sched.schedule(wl.epoch_seconds, wl.total_cores)
    compare_epoch(alloc, sched.get_predictions(), oracle_epoch(oracle_mod, wl), wl.total_cores, wl.max_cores_per_job)
    stats = sched.get_stats()
    assert stats.points == int(lengths.sum())
