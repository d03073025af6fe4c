"""The full Bellman-Ford rounds (asral_cluster_kernel), which run where the
guided ones do not: a shortcut switched off, penalties of 2^30 and more, more
centers than the guided layout holds.  Each case checks which kernel ran
(lbdd_guided_rounds) and compares everything with the oracle."""
import numpy as np
import pytest

import lbdd_inputs as L
import oracle
from test_gpu_paths import GLOBAL_CASES, INT32_CASES, _check_golden, _golden, check, clusters_for

pytestmark = pytest.mark.gpu


def run(lb, cm, inst, cluster, rounds=-1, **kw):
    """test_gpu_paths.solve's tuple and the rounds that ran guided."""
    with lb.Solver(cm, inst.cap, inst.pen, cluster=cluster, **kw) as s:
        s.solve(rounds)
        return (s.assignment(), s.objective, s.loads(), s.stats(), s.table()), s.guided_rounds


@pytest.mark.parametrize("case", range(len(GLOBAL_CASES)))
def test_slice_in_global_memory(gpu_lib, case):
    n, k, cm_max, cap_frac, pen = GLOBAL_CASES[case]
    inst = L.random_small(7300 + case, n=n, k=k, cm_max=cm_max, cap_frac=cap_frac, pen=pen)
    ref = oracle.asral(inst.cm, inst.cap, inst.pen)
    for cluster in clusters_for(k, (1, 2, 4, 16)):
        for off in ("npath_reuse", "ncyc_skip"):
            out, guided = run(gpu_lib, inst.cm, inst, cluster, tc_smem=False, **{off: False})
            assert guided == 0 and out[3].cost_slice_in_smem == 0
            check(out, ref, inst.cm)


@pytest.mark.parametrize("case", range(len(INT32_CASES)))
def test_int32_clusters(gpu_lib, case):
    n, k, cm_max, off, cap_frac, pen = INT32_CASES[case]
    inst = L.random_small(7400 + case, n=n, k=k, cm_max=cm_max, cap_frac=cap_frac, pen=pen)
    cm = inst.cm + np.int32(off)
    ref = oracle.asral(cm, inst.cap, inst.pen)
    assert ref.rc == 0 and ref.stats["moves"] > 0
    for cluster in clusters_for(k, (1, 2, 4, 16)):
        for tc_smem in (True, False):
            out, guided = run(gpu_lib, cm, inst, cluster, tc_smem=tc_smem, npath_reuse=False)
            assert guided == 0 and out[3].cm_elem_bytes == 4
            check(out, ref, cm)


@pytest.mark.parametrize("cluster", [16, 8])
def test_wide_prefix_matches_golden(gpu_lib, cluster):
    """20,000 x 2,000, 1,000 rounds with cycles and paths, slices in global memory."""
    gold = _golden("wide_r1000_oracle.json")
    inst = L.make_named("wide", dtype="i16")
    out, guided = run(gpu_lib, inst.cm, inst, cluster, rounds=gold["rounds"], npath_reuse=False)
    assert guided == 0 and out[3].cost_slice_in_smem == 0 and out[3].cluster_size == cluster
    _check_golden(out, gold)


# around the most centers of the guided layout (2,680 with int16 costs, 1,954
# with int32 costs) and far past it.  The oracle takes minutes at these sizes:
# the two kernels are compared with each other, the table with the oracle's for
# the same allotment, the objective with Eq. (1).
@pytest.mark.parametrize("k,add,kind", [(2680, 0, "guided"), (2681, 0, "full"), (1954, 40000, "guided"),
                                        (1955, 40000, "full"), (4000, 0, "full")])
def test_limit_of_the_guided_layout(gpu_lib, k, add, kind):
    n = 900
    inst = L.random_small(7600 + k, n=n, k=k, cm_max=20, cap_frac=0.5, pen=(1, 9))
    inst.cap = np.ones(k, np.int32)
    cm = inst.cm + np.int32(add)
    cm[:, 12:] += 60   # few centers are near, so that they overflow
    (assign, delta, loads, st, (tc, td)), guided = run(gpu_lib, cm, inst, 0)
    assert guided == (n if kind == "guided" else 0)
    assert st.cycles_applied > 0 and st.paths_applied > 0
    other, guided = run(gpu_lib, cm, inst, 0, npath_reuse=False, ncyc_skip=False)
    assert guided == 0
    assert np.array_equal(assign, other[0]) and delta == other[1]
    assert np.array_equal(loads, other[2]) and st.moves == other[3].moves
    assert np.array_equal(tc, other[4][0]) and np.array_equal(td, other[4][1])
    load = np.bincount(assign, minlength=k)
    assert delta == (int(cm[np.arange(n), assign].astype(np.int64).sum()) +
                     int((np.maximum(0, load - inst.cap) * inst.pen.astype(np.int64)).sum()))
    rtc, rtd = oracle.best_transfer(cm, assign)
    assert np.array_equal(tc, np.where(rtc >= oracle.INF, 2**31 - 1, rtc))
    assert np.array_equal(td, rtd)


def test_default_rounds_are_guided(gpu_lib):
    inst = L.random_small(7650, n=300, k=40, cm_max=30, cap_frac=0.5, pen=(1, 30))
    for pen, guided in ((inst.pen, 300), (np.full(40, 1 << 30, np.int32), 0)):
        with gpu_lib.Solver(inst.cm, inst.cap, pen) as s:
            s.solve(100)
            gpu_lib.set_option(s.h, gpu_lib.OPT_PHASE_TIMERS, 1)
            s.solve()
            assert s.guided_rounds == guided and s.rounds == 300
            s.reset()
            assert s.guided_rounds == 0
