"""What the request server charges for a request, and requests that the budget
admits only without the guided rounds' mirror."""
import numpy as np
import pytest

import lbdd_inputs as L
import oracle

pytestmark = pytest.mark.gpu


def serve(lb, budget, cm, inst):
    with lb.Server(budget_bytes=budget) as srv:
        info, a = srv.result(srv.submit(cm, inst.cap, inst.pen), 300_000)
        return info, a, srv.stats().peak_bytes


def test_wide_costs_are_charged_their_own_mirror(gpu_lib):
    n, k = 100, 600
    inst = L.random_small(9400, n=n, k=k, cm_max=50, cap_frac=0.5, pen=(5, 60))
    wide = inst.cm + np.int32(40000)
    _, _, narrow_bytes = serve(gpu_lib, 8 << 30, inst.cm.astype(np.int16), inst)
    info, a, wide_bytes = serve(gpu_lib, 8 << 30, wide, inst)
    ref = oracle.asral(wide, inst.cap, inst.pen)
    assert info.objective == ref.delta and np.array_equal(a, ref.assign)
    # 4 bytes instead of 2 per cost and per entry of the mirror
    assert wide_bytes - narrow_bytes >= 2 * n * k + 2 * k * k


def test_request_that_fits_without_the_mirror(gpu_lib):
    inst = L.random_small(9401, n=400, k=300, cm_max=50, cap_frac=0.5, pen=(5, 60))
    cm = inst.cm.astype(np.int16)
    ref = oracle.asral(inst.cm, inst.cap, inst.pen)
    info, a, full = serve(gpu_lib, 8 << 30, cm, inst)
    assert info.objective == ref.delta and np.array_equal(a, ref.assign)
    info, a, less = serve(gpu_lib, full - 1, cm, inst)
    assert info.state == gpu_lib.REQ_DONE and less < full
    assert info.objective == ref.delta and np.array_equal(a, ref.assign)
