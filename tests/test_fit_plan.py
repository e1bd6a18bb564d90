"""The plan of a fit - which block size, lanes and length classes a cluster gets - and of a selection."""

import random

import pytest

from fit_plan import fit_plan, select_bounded

SMS = 148


@pytest.mark.parametrize("lanes,jobs", [(4, 148 * 8 * 8), (2, 148 * 8 * 16)])
def test_a_few_slots_more_than_one_wave_are_a_second_one(lanes, jobs):
    """Eight warps per SM hold 1,184 slots: a few jobs more and a second wave of as long a chain follows (19,000 full windows of 32: 146 us,
    106 at twelve warps)."""
    for H in (24, 32, 48, 64):
        for more in (1, 8, 24, 56):
            warps, least, classes, _ = fit_plan(H, jobs + more)
            slots = -(-(jobs + more) * least // 32)
            assert len(classes) == 1
            assert slots <= SMS * warps or slots > 1.1 * SMS * warps, (H, more, warps, least)


def test_every_plan_is_one_that_has_a_kernel():
    """Eight and sixteen warps have kernels for one class only, sixteen for two lanes only; the classes cover all lengths, and the windows of
    each have room in a warp's slice."""
    rng = random.Random(3)
    seen = set()
    for _ in range(4000):
        jobs = int(2 ** rng.uniform(0, 21))
        H = int(2 ** rng.uniform(2, 14))
        given = rng.choice([13824, 13824, rng.randrange(8192, 204801)])
        warps, least, classes, slice_doubles = fit_plan(H, jobs, SMS, given)
        seen.add((warps, least, len(classes)))
        if warps != 12:
            assert len(classes) == 1 and classes[0][0] == least
        if warps == 16:
            assert least == 2
            assert 8 * (H + 16 * slice_doubles) <= 226 * 1024 or given == 13824
        above = H
        for lanes, low, high in classes:
            assert high == above and low < high
            above = low
            rows = -(-high // lanes)
            assert 12 * (64 // lanes) + 32 * (rows + 1) <= slice_doubles      # parked sums, the rows, one spare
        assert above == 0
    assert {w for w, _, _ in seen} == {8, 12, 16} and {n for _, _, n in seen} >= {1, 2, 3, 4}


def test_a_slice_of_the_callers_runs_sixteen_warps_at_two_lanes_where_they_have_room():
    assert fit_plan(64, 150_000, SMS, 12288)[:2] == (16, 2)
    assert fit_plan(64, 150_000, SMS, 16384)[:2] == (12, 2)      # sixteen of those do not fit


def test_a_sample_is_small_beside_the_first_gains_of_all_rows():
    """60,000 rows of 256: 28 us from the first 16 gains of each, 37 from a sample of 32 rows per block."""
    assert not select_bounded(60_000, 256, 120_000) and not select_bounded(60_000, 128, 120_000)
    assert select_bounded(60_000, 64, 240_000) and select_bounded(100_000, 64, 400_000) and select_bounded(1_000_000, 128, 4_000_000)
    assert not select_bounded(33_000, 64, 132_000)
    for jobs in (60_000, 80_000, 150_000, 500_000):
        for cap in (17, 40, 64, 100, 128, 256, 1024):
            for per in (0.3, 1.5, 4.0, 16.0):
                want = int(per * jobs) - (jobs if per >= 1 else 0)
                depth = min(cap, max(16, -(-4 * (-(-want // jobs) + 1) // 16) * 16))
                if select_bounded(jobs, cap, int(per * jobs)):
                    assert depth < cap and depth * jobs >= 2.5 * 32 * SMS * cap
