"""The row-order scan of 256 to 512 centers with int16 costs takes column slices
of 32 or 64 columns by the waves that the row ranges make: sizes on both sides,
with ragged last slices, against the oracle."""
from types import SimpleNamespace

import numpy as np
import pytest

from test_gpu_best_transfer import gpu_table, ref_table

pytestmark = pytest.mark.gpu


# 64 columns: ranges past one wave (600,000 x 500; 449 = 7 x 64 + 1), one wave
# that 64 columns fill better (420,000 x 512); 32 columns: the same rows with a
# center count that 32 columns suit (600,000 x 300), few rows (7,001 x 449)
@pytest.mark.parametrize("n,k", [(600_000, 500), (660_001, 449), (420_000, 512), (600_000, 300),
                                 (7_001, 449)])
def test_slices(gpu_lib, n, k):
    rng = np.random.default_rng(n + k)
    cm = rng.integers(1, 40, (n, k), dtype=np.int16)
    cm[:: n // 7] += np.int16(32700)           # differences near both ends of 16 bits
    assign = rng.integers(-1, k, n).astype(np.int32)
    assign[assign == 5] = -1
    inst = SimpleNamespace(n=n, k=k, cm=cm.astype(np.int32))
    tc, td = gpu_table(gpu_lib, inst, assign, "i16")
    rtc, rtd = ref_table(inst, assign)
    assert np.array_equal(tc, rtc) and np.array_equal(td, rtd)
