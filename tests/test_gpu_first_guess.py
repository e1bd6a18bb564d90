"""The fits' starting points (no trials at all) against the oracle's: the logarithm by table and the sign of family I's quadratic read off
its lowest point are used nowhere else.  The second number of jobs is beyond what teams fit."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _windows():
    """(window, largest reduction seen before it) by kind and length."""
    rng = np.random.default_rng(11)
    out = []
    for H in (4, 5, 31, 33, 64, 200):
        m = np.arange(H)
        for scale in (1.0, 1e-12, 3e15):                     # every bin of the logarithm, far from 1 and close to it
            out.append((scale * (0.9 ** m + 0.05) * np.exp(0.01 * rng.standard_normal(H)), -np.inf))
            out.append((scale / (1.0 + 0.3 * m) * np.exp(0.01 * rng.standard_normal(H)), -np.inf))
        # 1 / (loss - d0) falls and rises again: the quadratic's lowest point lies inside the window, at a point or between two, above
        # zero or below
        for turn in (0.2, 0.5, 0.5 + 0.5 / H, 0.93):
            for low in (0.9, 0.3, 0.05):
                z = low + (m / (H - 1.0) - turn) ** 2 * 4.0
                out.append((1.0 / z, 1.0))
        out.append((2.0 - 1e-5 * m, -np.inf))                # levels far above their differences
        out.append((1.0 + rng.random(H), 1e250))             # levels of 1e-250: the spread is normal, its bottom part is not squared
        out.append(((1.0 + rng.random(H)) * 1e-60, 1e250))   # subnormal levels
        out.append((np.linspace(1.0, 2.0, H), 1e-308))       # rising under a tiny M: levels near the end of the range
    return out


@pytest.mark.parametrize("warm,copies", [(0, 1), (1, 1), (0, 8)])
def test_first_guesses_match_the_oracle(oracle_mod, warm, copies):
    import paper_1802_04819_b200 as slaq
    rows = _windows()
    n, J = len(rows), len(rows) * copies
    rows = rows * copies
    sched = slaq.Scheduler(J, 200, 16)
    sched.set_param(slaq.binding.P_LM_TRIALS, 0)
    sched.set_param(slaq.binding.P_WARM_START, warm)
    off = np.zeros(J + 1, np.int64)
    np.cumsum([h.size for h, _ in rows], out=off[1:])
    ids = np.arange(J, dtype=np.int32)
    sched.load_histories(ids, off, np.concatenate([h for h, _ in rows]), np.full(J, 1000, np.int64),
                         np.array([m for _, m in rows]))
    sched.set_time_model(ids, np.full(J, 0.1), np.full(J, 2.0))
    sched.schedule(1.0, 4 * J)
    st = sched.get_fit_state()
    lines = 0
    for k in range(1, copies):
        same = st["valid"][:n] != 0
        np.testing.assert_array_equal(st["valid"][k * n: (k + 1) * n], st["valid"][:n])
        np.testing.assert_array_equal(st["p"][k * n: (k + 1) * n][same], st["p"][:n][same])
    for j, (h, m_seen) in enumerate(rows[:n]):
        for fam in (0, 1):
            ref = oracle_mod.fit_family(fam, h, m_seen, trials=0)
            got, p0 = st["p"][j, 4 * fam: 4 * fam + 4], ref["p0"]
            assert bool(st["valid"][j] >> fam & 1) == bool(np.isfinite(ref["S"])), (j, fam)
            if not np.isfinite(ref["S"]):
                continue
            if fam == 0:
                assert (got[0] == 0.0) == (p0[0] == 0.0), (j, got, p0)     # the line through two points, or the parabola
                lines += p0[0] == 0.0
            # weighted normal equations in x, x^2, 1 of up to 200 points: conditions up to some 1e6 times a few ulp
            np.testing.assert_allclose(got[:3 + (fam == 0)], p0[:3 + (fam == 0)], rtol=1e-7, atol=1e-9 * np.abs(p0).max())
    assert 0 < lines < n
