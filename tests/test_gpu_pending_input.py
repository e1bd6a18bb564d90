"""An entry that slaq_append_losses_device skipped is reported by the next slaq_schedule, whatever is called in between."""

import numpy as np
import pytest

from gpu_common import make_scheduler
from workloads import make_workload

pytestmark = pytest.mark.gpu


def test_allocate_only_leaves_the_report_to_the_next_epoch():
    import torch
    import paper_1802_04819_b200 as slaq
    slaq.build()
    wl = make_workload(1)
    s = make_scheduler(wl)
    gain = np.sort(np.random.default_rng(0).random((wl.n_jobs, wl.max_cores_per_job)), 1)[:, ::-1].copy()
    bad = torch.tensor([0, wl.n_jobs + 5], dtype=torch.int32, device="cuda")
    s.append_losses_device(bad, torch.ones(2, dtype=torch.float64, device="cuda"))
    s.set_gains(gain)
    alloc, rc = s.allocate_only(wl.total_cores)
    assert rc == 0 and alloc.sum() == wl.total_cores
    with pytest.raises(slaq.SlaqError) as e:
        s.schedule(wl.epoch_seconds, wl.total_cores)
    assert e.value.code == -5 and "slaq_append_losses_device" in str(e.value)
    assert s.schedule(wl.epoch_seconds, wl.total_cores)[1] == 0       # reported once
    s.close()
