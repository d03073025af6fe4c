"""Batch plans of solvers that run the guided rounds next to solvers that run
the full Bellman-Fords: the tuning table keeps the two apart, and the limit on
a batch's groups counts them once."""
import numpy as np
import pytest

import lbdd_inputs as L
import oracle

pytestmark = pytest.mark.gpu


def plan(lb, s):
    b = lb.Batch([s])
    try:
        return b.plan()[0]
    finally:
        b.close()


@pytest.mark.parametrize("full", ["ncyc_skip", "npath_reuse", "large penalty"])
def test_tuning_of_one_kind_leaves_plans_of_the_other(gpu_lib, full):
    """Times measured on one kind of rounds do not plan the other: its plan is
    the one without measurements."""
    inst = L.random_small(9900, n=700, k=300, cm_max=60, cap_frac=0.7, pen=(5, 90))
    pen = inst.pen.copy()
    kw = {}
    if full == "large penalty":
        pen[3] = 1 << 30
    else:
        kw[full] = False
    gpu_lib.tune_clear()
    try:
        with gpu_lib.Solver(inst.cm, inst.cap, inst.pen) as g, \
                gpu_lib.Solver(inst.cm, inst.cap, pen, **kw) as f:
            plan_g, plan_f = plan(gpu_lib, g), plan(gpu_lib, f)
            assert plan_g == [1] and plan_f == [4]   # 128 columns per CTA
            gpu_lib.autotune([g], probe_rounds=500)
            assert plan(gpu_lib, f) == plan_f
            gpu_lib.tune_clear()
            gpu_lib.autotune([f], probe_rounds=500)
            assert plan(gpu_lib, g) == plan_g
    finally:
        gpu_lib.tune_clear()


def test_sixteen_option_sets_with_both_kinds(gpu_lib):
    """Sixteen combinations of options form sixteen groups, the most a batch
    takes; a penalty past the guided limit in four of them adds none."""
    combos = [(a, b, c, d) for a in (0, 1) for b in (0, 1) for c in (0, 1) for d in (0, 1)]
    solvers, refs = [], []
    try:
        for i, (ncyc, npath, tc, timers) in enumerate(combos + [x for x in combos if x[0] and x[1]]):
            inst = L.random_small(9950 + i, n=90, k=7, cm_max=30, cap_frac=0.6, pen=(3, 40))
            pen = inst.pen.copy()
            if i >= len(combos):
                pen[0] = 1 << 30
            refs.append(oracle.asral(inst.cm, inst.cap, pen))
            solvers.append(gpu_lib.Solver(inst.cm, inst.cap, pen, ncyc_skip=bool(ncyc),
                                          npath_reuse=bool(npath), tc_smem=bool(tc),
                                          phase_timers=bool(timers)))
        gpu_lib.solve_batch([s.h for s in solvers], cluster_size=1)
        for s, ref in zip(solvers, refs):
            assert s.objective == ref.delta and np.array_equal(s.assignment(), ref.assign)
    finally:
        for s in solvers:
            s.close()
