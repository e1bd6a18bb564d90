"""Calls on a handle whose stream the caller captures into a graph of its own."""

import numpy as np
import pytest

from gpu_common import make_scheduler
from workloads import make_workload

pytestmark = pytest.mark.gpu


# one block sorts the windows and the queue hands out more slots than the GPU has warps; the counting sort of many jobs
@pytest.mark.parametrize("cfg,jobs", [(3, 6000), (4, 60000)])
def test_a_captured_epoch_clears_its_scratch_itself(cfg, jobs):
    """Between two replays the handle makes calls that leave the scratch of an epoch as they used it."""
    import torch
    import paper_1802_04819_b200 as slaq
    slaq.build()
    wl = make_workload(cfg, n_jobs=jobs)
    J, C = wl.n_jobs, wl.total_cores
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
        a.shard_predict(wl.epoch_seconds, True)
        for s in (a, b):
            s.append_losses(ids, (0.96 - 0.02 * step) * last)
        with torch.cuda.stream(stream):
            graph.replay()
        stream.synchronize()
        ref, _ = b.schedule(wl.epoch_seconds, C)
        np.testing.assert_array_equal(out.cpu().numpy(), ref)
        mine, theirs = a.get_stats(), b.get_stats()       # the statistics are the replay's
        for key in ("points", "model_sweeps", "fitted_jobs", "cores_handed_out", "tie_units", "threshold"):
            assert getattr(mine, key) == getattr(theirs, key)
        assert mine.ms_total > 0.0 and mine.ms_fit > 0.0
    a.close()
    b.close()


@pytest.mark.parametrize("jobs", [8, 5000])
def test_an_append_from_host_arrays_is_refused_under_capture(jobs):
    """It would be applied by the replays and not by the call, from arrays the caller may reuse."""
    import torch
    import paper_1802_04819_b200 as slaq
    slaq.build()
    wl = make_workload(2, n_jobs=jobs)
    ids = np.arange(jobs, dtype=np.int32)
    last = wl.losses[wl.offsets[1:] - 1]
    stream = torch.cuda.Stream()
    a, b = make_scheduler(wl), make_scheduler(wl)
    a.set_stream(stream)
    graph = torch.cuda.CUDAGraph()
    refused = None
    try:
        with torch.cuda.graph(graph, stream=stream):
            try:
                a.append_losses(ids, 0.5 * last)
            except slaq.SlaqError as e:
                refused = e.code
    except RuntimeError:
        pass                      # the refused call may have ended the capture
    assert refused == -5
    torch.cuda.synchronize()
    np.testing.assert_array_equal(a.schedule(wl.epoch_seconds, 2 * jobs)[0], b.schedule(wl.epoch_seconds, 2 * jobs)[0])
    for s in (a, b):              # and the next one is taken
        s.append_losses(ids, 0.9 * last)
    np.testing.assert_array_equal(a.schedule(wl.epoch_seconds, 2 * jobs)[0], b.schedule(wl.epoch_seconds, 2 * jobs)[0])
    assert a.export_state().tobytes() == b.export_state().tobytes()
    a.close()
    b.close()
