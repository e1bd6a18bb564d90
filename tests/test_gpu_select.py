"""The selection launch at the sizes where its paths change, against the definition: the C' largest gains beyond the
floor, ties to the lowest job id.  Integer results, so bit for bit."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _rows(kind, J, cap, rng):
    if kind == "spread":      # many orders of magnitude, some rows nothing
        g = np.exp(rng.uniform(-60, 2, (J, 1))) * np.sort(rng.random((J, cap)), 1)[:, ::-1]
        g[rng.random(J) < 0.1] = 0.0
    elif kind == "one bin":   # every gain inside one bin of the first histogram: all blocks narrow
        g = 0.25 * (1.0 + 0.004 * np.sort(rng.random((J, cap)), 1)[:, ::-1])
    elif kind == "equal":     # one value everywhere: handed out in job order over the blocks
        g = np.full((J, cap), 0.37)
    elif kind == "levels":    # a few values, thousands of ties each, zero among them
        g = np.sort(rng.integers(0, 4, (J, cap)), 1)[:, ::-1] * 2.0 ** -33
    else:                     # "deep": few rows hold nearly everything, so they are continued far beyond the others
        g = np.where(np.arange(J)[:, None] % 97 == 0, 1.0, 1e-6) * np.sort(rng.random((J, cap)), 1)[:, ::-1]
    return np.ascontiguousarray(g, dtype=np.float64)


def _expected(gain, C):
    J, cap = gain.shape
    floor = 1 if C >= J else 0
    want = min(C, J * cap) - floor * J
    tail = gain[:, floor:]
    key = tail.ravel()
    order = np.argsort(-key, kind="stable")[:want]          # stable: (job id, n) among equal gains
    alloc = floor + np.bincount(order // max(1, cap - floor), minlength=J) if want else np.full(J, floor)
    return alloc.astype(np.int32)


# one block; the last resident table and the first streamed one (2048 gains x 148 SMs); more tiles than one per block
@pytest.mark.parametrize("J,cap", [(1, 1), (3, 1024), (33, 31), (4736, 64), (4737, 64), (2368, 128), (90000, 17), (151600, 2)])
@pytest.mark.parametrize("kind", ["spread", "one bin", "equal", "levels", "deep"])
def test_selection_equals_the_definition(J, cap, kind):
    import paper_1802_04819_b200 as slaq
    slaq.build()
    rng = np.random.default_rng(J + cap)
    gain = _rows(kind, J, cap, rng)
    with slaq.Scheduler(J, 4, cap) as sched:
        sched.append_losses(np.arange(J), np.ones(J))
        sched.set_gains(gain)
        for C in sorted({0, J - 1, J, J + 1, J + J * (cap - 1) // 7, J * cap - 1, J * cap, J * cap + 5}):
            alloc, _ = sched.allocate_only(C)
            want = _expected(gain, C)
            np.testing.assert_array_equal(alloc, want)
            R = sched.get_predictions(want_gain=False)["R"]
            ref = np.concatenate([np.zeros((J, 1)), np.cumsum(gain, 1)], 1)[np.arange(J), want]
            np.testing.assert_array_equal(R, ref)           # the same additions in the same order


def test_rows_that_only_some_blocks_continue():
    """A streamed table whose long rows lie in a tenth of the blocks: those are still counting while the others have long
    reached the second barrier.  The same table over and over, as the blocks meet differently each time."""
    import paper_1802_04819_b200 as slaq
    slaq.build()
    J, cap = 30000, 64
    rng = np.random.default_rng(5)
    gain = np.exp(rng.uniform(-30, -10, (J, 1))) * np.sort(rng.random((J, cap)), 1)[:, ::-1]
    gain[J // 2: J // 2 + J // 10] *= np.exp(25.0)            # whole rows above everything else
    with slaq.Scheduler(J, 4, cap) as sched:
        sched.append_losses(np.arange(J), np.ones(J))
        sched.set_gains(gain)
        for C in (J + 1000, 3 * J, J + J // 10 * (cap - 1) - 1):
            want = _expected(gain, C)
            for _ in range(60):
                alloc, _ = sched.allocate_only(C)
                np.testing.assert_array_equal(alloc, want)
