"""The selection of small tables, which one block does, at the sizes where that begins and ends, against the definition."""

import numpy as np
import pytest

from test_gpu_select import _expected, _rows

pytestmark = pytest.mark.gpu


# up to 256 rows and 6144 gains take one block; more than 256 candidates that are all equal go out in job order
@pytest.mark.parametrize("J,cap", [(8, 16), (31, 5), (32, 33), (6, 1024), (7, 1024), (192, 32), (193, 32), (256, 24), (257, 23)])
@pytest.mark.parametrize("kind", ["spread", "one bin", "equal", "levels", "deep"])
def test_small_tables_equal_the_definition(J, cap, kind):
    import torch
    import paper_1802_04819_b200 as slaq
    slaq.build()
    gain = _rows(kind, J, cap, np.random.default_rng(7 * J + cap))
    d_gain = torch.from_numpy(gain).cuda()
    d_alloc = torch.zeros(J, dtype=torch.int32, device="cuda")
    d_R = torch.zeros(J, dtype=torch.float64, device="cuda")
    for C in sorted({0, J - 1, J, J + 1, J + J * (cap - 1) // 7, J * cap - 1, J * cap, J * cap + 5}):
        slaq.allocate_static(d_gain, C, d_alloc, d_R)
        want = _expected(gain, C)
        np.testing.assert_array_equal(d_alloc.cpu().numpy(), want)
        ref = np.concatenate([np.zeros((J, 1)), np.cumsum(gain, 1)], 1)[np.arange(J), want]
        np.testing.assert_array_equal(d_R.cpu().numpy(), ref)           # the same additions in the same order
