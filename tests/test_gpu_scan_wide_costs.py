"""The scan of int32 costs of fewer than 256 centers (and of 256 to 512) where a
difference needs all 32 bits: costs from 50,000 up, and 1 and 2^31 - 1 in one
matrix, so that differences reach both ends, +-(2^31 - 2), next to the value
that marks an empty entry.  Few distinct costs, so that ties cross row ranges."""
from types import SimpleNamespace

import numpy as np
import pytest

from test_gpu_best_transfer import gpu_table, ref_table

pytestmark = pytest.mark.gpu

TOP = 2**31 - 1
COSTS = {"above 16 bits": [50_000, 50_001, 82_769, 115_535, 131_072],
         "both ends": [1, 2, TOP - 1, TOP],
         "ends and middle": [1, 40_000, 1 << 30, TOP]}


# one cluster, one table in column slices, several tables and a merge, more
# than one row range per cluster; the row-order path of 256 centers and more
@pytest.mark.parametrize("n,k", [(5, 3), (3000, 20), (6000, 64), (900, 200), (9001, 126),
                                 (50001, 126), (20011, 255), (30000, 256)])
@pytest.mark.parametrize("costs", list(COSTS))
def test_wide_differences(gpu_lib, costs, n, k):
    rng = np.random.default_rng(n + k)
    cm = rng.choice(np.array(COSTS[costs], np.int32), (n, k))
    assign = rng.integers(-1, k, n).astype(np.int32)
    assign[assign == k // 2] = -1          # an empty center
    inst = SimpleNamespace(n=n, k=k, cm=cm)
    tc, td = gpu_table(gpu_lib, inst, assign, "i32")
    rtc, rtd = ref_table(inst, assign)
    if costs == "both ends" and n > 1000:
        assert rtc.min() == 2 - 2**31
        assert (rtc == TOP).any() and (rtd[rtc == TOP] == -1).all()
    assert np.array_equal(tc, rtc) and np.array_equal(td, rtd)


def test_largest_difference(gpu_lib):
    """Every transfer out of center 0 costs 2^31 - 2: one below an empty entry."""
    n, k = 4000, 40
    cm = np.full((n, k), TOP, np.int32)
    cm[:, 0] = 1
    assign = np.zeros(n, np.int32)
    assign[::3] = -1
    inst = SimpleNamespace(n=n, k=k, cm=cm)
    tc, td = gpu_table(gpu_lib, inst, assign, "i32")
    assert (tc[0, 1:] == TOP - 1).all() and (td[0, 1:] == 1).all()
    assert (tc[1:] == TOP).all() and (td[1:] == -1).all()
