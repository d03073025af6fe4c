"""Scans of fewer than 256 centers by the room for packed tables: a workspace
of the size that the grouped scan needed is enough, and the sizes where one
cluster ends."""
import numpy as np
import pytest

import lbdd_inputs as L
import oracle
from test_gpu_best_transfer import ref_table

pytestmark = pytest.mark.gpu

# (n, k, bytes): what the seven-launch scan's workspace took at these sizes
SIZES = [(50001, 126, 375296), (20011, 255, 676608), (9001, 126, 200960), (30000, 64, 178688),
         (9000, 200, 414208), (5000, 255, 612864)]


# around 64 centers and 393,216 entries, and calls of one table and several
EDGES = [(6144, 64), (6145, 64), (6049, 65), (90, 65), (16384, 24), (16385, 24), (49152, 8),
         (49153, 8), (80, 200), (1300, 200), (2000, 100), (3, 255)]


@pytest.mark.parametrize("dtype", ["i16", "i32"])
@pytest.mark.parametrize("n,k", EDGES)
def test_scan_where_one_cluster_ends(gpu_lib, dtype, n, k):
    run(gpu_lib, dtype, n, k, gpu_lib.best_transfer_workspace(n, k))


@pytest.mark.parametrize("dtype", ["i16", "i32"])
@pytest.mark.parametrize("n,k,size", SIZES)
def test_scan_with_the_smaller_workspace(gpu_lib, dtype, n, k, size):
    run(gpu_lib, dtype, n, k, size)


def run(gpu_lib, dtype, n, k, size):
    import torch
    inst = L.random_small(9300 + k, n=n, k=k, cm_max=90)
    assign = np.random.default_rng(k).integers(-1, k, n).astype(np.int32)
    dt, tdt = (gpu_lib.CM_I16, torch.int16) if dtype == "i16" else (gpu_lib.CM_I32, torch.int32)
    ld = gpu_lib.cm_pitch(k, dt)
    buf = torch.zeros(n * ld + 128, dtype=tdt, device="cuda")
    buf[: n * ld].view(n, ld)[:, :k] = torch.from_numpy(inst.cm).cuda().to(tdt)
    a = torch.from_numpy(assign).cuda()
    tc = torch.empty(k * k, dtype=torch.int32, device="cuda")
    td = torch.empty_like(tc)
    ws = torch.full((size + 4096,), 0x5a, dtype=torch.uint8, device="cuda")
    gpu_lib.best_transfer(n, k, buf, dt, ld, a, tc, td, ws, size)
    rtc, rtd = ref_table(inst, assign)
    assert np.array_equal(tc.cpu().numpy().reshape(k, k), rtc)
    assert np.array_equal(td.cpu().numpy().reshape(k, k), rtd)
    assert bool((ws[size:] == 0x5a).all())
    with pytest.raises(gpu_lib.LbddError):
        gpu_lib.best_transfer(n, k, buf, dt, ld, a, tc, td, ws, 1024)
