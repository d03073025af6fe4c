"""The price-guided one-CTA rounds against the oracle, at the sizes where
their layout changes: one column per lane (31 to 33 centers: one warp, then
several), 512 columns per pass (511 to 513), the cost table in shared memory
or in its global mirror (about 290 centers with int16 costs, 200 with int32),
member lists over several pages, penalty tables, and prices rebuilt after
rounds that kept none."""
import numpy as np
import pytest

import lbdd_inputs as L
import oracle

pytestmark = pytest.mark.gpu

TINF = 2**31 - 1


def check(s, ref, cm):
    assert s.objective == ref.delta
    assert np.array_equal(s.assignment(), ref.assign)
    assert np.array_equal(s.loads().astype(np.int64), ref.load)
    st = s.stats()
    for f in ("cycles_applied", "paths_applied", "moves"):
        assert getattr(st, f) == ref.stats[f], f
    tc, td = s.table()
    rtc, rtd = oracle.best_transfer(cm, ref.assign)
    assert np.array_equal(tc, np.where(rtc >= oracle.INF, TINF, rtc)) and np.array_equal(td, rtd)


CASES = [  # (n, k, cm_max, cap_frac, pen, added to every cost)
    (900, 2, 60, 0.5, (1, 40), 0),        # lists of several pages
    (1500, 5, 300, 0.4, (20, 900), 0),
    (300, 31, 25, 0.5, (1, 30), 0),
    (300, 32, 25, 0.5, (1, 30), 0),
    (300, 33, 25, 0.5, (1, 30), 0),
    (260, 33, 25, 0.5, (1, 30), 40000),
    (500, 129, 40, 0.6, (5, 60), 0),
    (450, 210, 90, 0.4, (5, 90), 40000),
    (500, 280, 30, 0.4, (5, 60), 0),
    (500, 300, 30, 0.4, (5, 60), 0),
    (560, 511, 40, 0.9, (5, 60), 0),
    (560, 513, 40, 0.9, (5, 60), 0),
    (200, 40, 30000, 0.5, (1, 1 << 29), 0),
    (200, 40, 30000, 0.5, (1 << 30, 2**31 - 1), 0),   # past the guided limit: unguided rounds
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_guided_matches_oracle(gpu_lib, case):
    n, k, cm_max, cap_frac, pen, add = CASES[case]
    inst = L.random_small(7700 + case, n=n, k=k, cm_max=cm_max, cap_frac=cap_frac, pen=pen)
    cm = inst.cm + np.int32(add)
    ref = oracle.asral(cm, inst.cap, inst.pen)
    assert ref.rc == 0 and ref.stats["moves"] > 0
    for tc_smem in (True, False):
        with gpu_lib.Solver(cm, inst.cap, inst.pen, tc_smem=tc_smem) as s:
            s.solve()
            check(s, ref, cm)


@pytest.mark.parametrize("seed", range(3))
def test_guided_penalty_table(gpu_lib, seed):
    k = (7, 33, 90)[seed]
    inst = L.random_small(7800 + seed, n=400, k=k, cm_max=30, cap_frac=0.4)
    qtab = L.penalty_table(7800 + seed, k, 6, base=(1, 20), step=(0, 15))
    ref = oracle.asral_q(inst.cm, inst.cap, qtab)
    assert ref.rc == 0 and ref.stats["paths_applied"] > 0
    with gpu_lib.Solver(inst.cm, inst.cap, inst.pen, qtab=qtab) as s:
        s.solve()
        check(s, ref, inst.cm)


@pytest.mark.parametrize("strict", [False, True])
@pytest.mark.parametrize("k,cluster", [(9, 2), (48, 4)])
def test_prices_are_rebuilt_after_unguided_rounds(gpu_lib, k, cluster, strict):
    """Slices of guided rounds, rounds that keep no prices (Alg. 1 never
    skipped) and rounds with the costs out of shared memory, on one CTA and on
    a cluster."""
    inst = L.random_small(7900 + k, n=420, k=k, cm_max=30, cap_frac=0.5, pen=(5, 60))
    with gpu_lib.Solver(inst.cm, inst.cap, inst.pen, strict=strict) as s:
        for i, rounds in enumerate((150, 60, 40, 50, 30, -1)):
            gpu_lib.set_option(s.h, gpu_lib.OPT_NCYC_SKIP, 0 if i in (1, 4) else 1)
            gpu_lib.set_option(s.h, gpu_lib.OPT_TC_SMEM, 0 if i in (2, 5) else 1)
            gpu_lib.set_option(s.h, gpu_lib.OPT_CLUSTER, cluster if i in (3, 4) else 0)
            s.solve(rounds)
        if strict:
            rc, assign, cost, _ = oracle.strict(inst.cm, inst.cap)
            assert rc == 0 and s.objective == cost and np.array_equal(s.assignment(), assign)
        else:
            ref = oracle.asral(inst.cm, inst.cap, inst.pen)
            check(s, ref, inst.cm)


@pytest.mark.parametrize("case", range(6))
def test_guided_strict(gpu_lib, case):
    """Alg. 5 guided: one and several columns' warps, int16 and int32 costs,
    capacity short (dummy center), equal to n, and ample."""
    n, k, cm_max, frac, add = [(300, 31, 40, 0.8, 0), (300, 33, 40, 1.0, 0), (420, 33, 9, 1.3, 0),
                               (260, 64, 300, 0.9, 40000), (700, 3, 90, 0.9, 0),
                               (400, 140, 60, 1.1, 0)][case]
    inst = L.random_small(8000 + case, n=n, k=k, cm_max=cm_max, cap_frac=frac)
    cm = inst.cm + np.int32(add)
    rc, assign, cost, ref = oracle.strict(cm, inst.cap)
    assert rc == 0
    for tc_smem in (True, False):
        with gpu_lib.Solver(cm, inst.cap, None, strict=True, tc_smem=tc_smem) as s:
            s.solve()
            st = s.stats()
            assert s.objective == cost and np.array_equal(s.assignment(), assign)
            assert st.cycles_applied == ref["cycles_applied"] and st.moves == ref["moves"]
