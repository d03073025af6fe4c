"""Long tables of int32 costs with 64 to 255 centers: the row-order scan from
64 MB of costs on, the grouped scan or the table scan where the workspace has no
room for its row ranges."""
import numpy as np
import pytest

from test_gpu_best_transfer import ref_table

pytestmark = pytest.mark.gpu


def rows(k, mb):
    return -(-(mb << 20) // (4 * k))


# both sides of 64 centers and of 64 MB, ragged last slices of 32 columns
CASES = [(rows(64, 64), 64), (rows(64, 64) - 1, 64), (rows(63, 70), 63), (rows(65, 70), 65),
         (rows(100, 64), 100), (rows(128, 66), 128), (rows(201, 100), 201), (rows(255, 64), 255)]


@pytest.mark.parametrize("room", ["asked", "least"])
@pytest.mark.parametrize("n,k", CASES)
def test_long_tables(gpu_lib, n, k, room):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    ld = gpu_lib.cm_pitch(k, gpu_lib.CM_I32)
    buf = torch.randint(1, 90, (n * ld + 128,), generator=g, device="cuda", dtype=torch.int32)
    cm = buf[: n * ld].view(n, ld)[:, :k]
    cm[:: n // 11] += 2**31 - 100          # differences near both ends of 32 bits
    assign = np.random.default_rng(k).integers(-1, k, n).astype(np.int32)
    assign[assign == 3] = -1
    assign[::1009] = k + 5                 # no center
    a = torch.from_numpy(assign).cuda()
    tc = torch.empty(k * k, dtype=torch.int32, device="cuda")
    td = torch.empty_like(tc)
    size = gpu_lib.best_transfer_workspace(n, k)
    if room == "least":
        size = min(size, 4 * n + n // 4 + 8 * k * k + 276 * k + 2048)
    ws = torch.full((size + 4096,), 0x5a, dtype=torch.uint8, device="cuda")
    gpu_lib.best_transfer(n, k, buf, gpu_lib.CM_I32, ld, a, tc, td, ws, size)
    from types import SimpleNamespace
    inst = SimpleNamespace(n=n, k=k, cm=np.ascontiguousarray(cm.cpu().numpy()))
    rtc, rtd = ref_table(inst, np.where(assign < k, assign, -1).astype(np.int32))
    assert np.array_equal(tc.cpu().numpy().reshape(k, k), rtc)
    assert np.array_equal(td.cpu().numpy().reshape(k, k), rtd)
    assert bool((ws[size:] == 0x5a).all())
