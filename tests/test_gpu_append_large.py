"""Appends above the mailbox's size are checked on the device: accepted or refused as a whole, with the host's messages."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N = 33000     # more entries than pass through the mailbox


@pytest.mark.parametrize("n", [N, N + 257])
def test_large_appends_are_taken_or_refused_whole(n):
    import paper_1802_04819_b200 as slaq
    slaq.build()
    rng = np.random.default_rng(n)
    ids, loss = np.arange(n, dtype=np.int32), rng.uniform(1.0, 2.0, n)
    times, cores = rng.uniform(0.1, 1.0, n), rng.integers(1, 9, n).astype(np.int32)
    order = rng.permutation(n)
    with slaq.Scheduler(n, 8, 4) as a, slaq.Scheduler(n, 8, 4) as b:
        a.append_losses(ids, loss, times, cores)
        b.append_losses(ids[order], loss[order], times[order], cores[order])     # ids that do not rise are fine
        assert a.export_state().tobytes() == b.export_state().tobytes()
        before = a.export_state().tobytes()

        def spoiled(v, at, x):
            w = v.copy()
            w[at] = x
            return w

        for bad in ((ids, spoiled(loss, n - 1, np.nan), times, cores), (ids, spoiled(loss, 7, np.inf), times, cores),
                    (ids, loss, spoiled(times, 255, -np.inf), cores), (ids, loss, times, spoiled(cores, n // 2, 0)),
                    (spoiled(ids, 5, 4), loss, times, cores), (spoiled(ids, n - 1, n), loss, times, cores),
                    (spoiled(ids, 0, -1), loss, times, cores)):
            with pytest.raises(slaq.SlaqError):
                a.append_losses(*bad)
            assert a.export_state().tobytes() == before
        a.append_losses(ids, loss * 0.9, times, cores)                           # and the next good one is taken
        b.append_losses(ids, loss * 0.9, times, cores)
        assert a.export_state().tobytes() == b.export_state().tobytes() != before
