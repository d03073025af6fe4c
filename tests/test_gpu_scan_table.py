"""The row-order table scan of fewer than 256 centers against the oracle:
one vector per row and ragged rows, one cluster and many, one column slice
and several, 32- and 64-bit keys, ties across row ranges, and entries of the
allotment that name no center."""
from types import SimpleNamespace

import numpy as np
import pytest

import oracle
from test_gpu_best_transfer import gpu_table, ref_table

pytestmark = pytest.mark.gpu


def instance(n, k, seed, cm_max):
    rng = np.random.default_rng(seed)
    cm = rng.integers(1, cm_max + 1, (n, k), dtype=np.int32)
    assign = rng.integers(0, k, n).astype(np.int32)
    odd = rng.random(n) < 0.05
    assign[odd] = rng.choice([-1, k, k + 7, 2**31 - 1, -2**31], int(odd.sum()))
    return SimpleNamespace(n=n, k=k, cm=cm), assign


# (n, k): around 8 and 4 columns per vector, 1 MB and 4 MB of costs, the
# slice limits (221 to 255 int16, 159 to 255 int32), one row
SIZES = [(1, 1), (1, 255), (2, 9), (37, 8), (3000, 3), (2047, 20), (2049, 21), (9001, 126),
         (40000, 17), (30000, 64), (50001, 126), (20011, 158), (20011, 159), (17000, 220),
         (17000, 221), (15013, 255)]


@pytest.mark.parametrize("dtype", ["i16", "i32"])
@pytest.mark.parametrize("case", range(len(SIZES)))
def test_table_scan_matches_oracle(gpu_lib, dtype, case):
    n, k = SIZES[case]
    inst, assign = instance(n, k, 900 + case, (3, 200, 32767)[case % 3])
    tc, td = gpu_table(gpu_lib, inst, assign, dtype)
    ref = np.where((assign >= 0) & (assign < k), assign, -1).astype(np.int32)
    rtc, rtd = ref_table(inst, ref)
    assert np.array_equal(tc, rtc) and np.array_equal(td, rtd)


def test_table_scan_long_ranges_use_wide_keys(gpu_lib):
    """More than 65,536 rows per range: int16 costs with 64-bit keys."""
    inst, assign = instance(11_000_000, 2, 950, 9)
    tc, td = gpu_table(gpu_lib, inst, assign, "i16")
    ref = np.where((assign >= 0) & (assign < 2), assign, -1).astype(np.int32)
    rtc, rtd = ref_table(inst, ref)
    assert np.array_equal(tc, rtc) and np.array_equal(td, rtd)
