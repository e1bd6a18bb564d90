"""Levels are the losses divided by the largest reduction, correctly rounded, on both ways the kernel takes: by a reciprocal and
corrections where all magnitudes lie within 2^-400 .. 2^400, by divisions elsewhere."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _windows(rng, H):
    one = rng.uniform(0.5, 2.0, H)
    yield one, 1.0
    yield one, np.nextafter(1.0, 0.0)                       # all bits of the mantissa set
    yield one * 2.0 ** rng.integers(-300, 300), 3.0 * 2.0 ** 299
    for e in (-401, -400, -399, 399, 400, 401):             # on either side of both limits
        yield one * 2.0 ** e, 1.7
        yield one, 1.3 * 2.0 ** e
    z = one.copy()
    z[::3] = 0.0
    yield z, 0.7
    yield -one, 0.9
    yield one * 1e-310, 1.1                                 # subnormal
    yield one * 1e300, 1e-5                                 # levels near the end of the range


@pytest.mark.parametrize("H", [2, 5, 33, 200])
def test_levels_are_correctly_rounded_quotients(H):
    import paper_1802_04819_b200 as slaq
    rng = np.random.default_rng(H)
    rows = list(_windows(rng, H))
    J = len(rows)
    s = slaq.Scheduler(J, 200, 8)
    off = np.arange(J + 1, dtype=np.int64) * H
    ids = np.arange(J, dtype=np.int32)
    losses = np.concatenate([h for h, _ in rows])
    s.load_histories(ids, off, losses, np.full(J, 500, np.int64), np.array([m for _, m in rows]))
    at, _, got, _ = s.get_normalised(ids)
    for j, (h, seen) in enumerate(rows):
        M = max(seen, float(np.max(h[:-1] - h[1:])))
        levels = got[at[j]: at[j + 1]]
        with np.errstate(over="ignore"):
            np.testing.assert_array_equal(levels, h / M)
