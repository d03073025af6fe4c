"""Guided rounds that scan long member lists for many entries end early and the
next stretch of rounds runs on the full Bellman-Ford kernel: the results are
those of a solver that runs the full form throughout, whatever launches the
rounds (whole and sliced solves, batches, the server)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def one_center(n, k, kind, dtype=np.int16, add=0):
    """Center 0 is the nearest of every unit and takes half of them.  `equal`: a
    unit costs the same at every other center (every entry of row 0 has the same
    best unit); `near`: it does not."""
    rng = np.random.default_rng(n + k)
    if kind == "equal":
        cm = np.tile(rng.integers(2000, 9000, (n, 1)), (1, k))
        cm[:, 0] = 1000
    else:
        cm = rng.integers(5000, 9000, (n, k))
        cm[:, 0] = rng.integers(1, 2000, n)
    cm = (cm + add).astype(dtype)
    cap = np.full(k, max(1, n // (4 * k)), np.int32)
    cap[0] = n // 2
    return cm, cap, np.full(k, 9000 + add, np.int32)


def state(s):
    return s.objective, s.assignment(), s.loads(), *s.table()


def same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


# the last one stays below the limit
CASES = [("equal", 12000, 300, np.int16, 0, True), ("equal", 9000, 300, np.int32, 40000, True),
         ("near", 30000, 500, np.int16, 0, True), ("equal", 3000, 100, np.int16, 0, False)]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_stretches_of_full_rounds(gpu_lib, case):
    kind, n, k, dtype, add, trips = CASES[case]
    cm, cap, pen = one_center(n, k, kind, dtype, add)
    with gpu_lib.Solver(cm, cap, pen, npath_reuse=False) as s:
        s.solve()
        assert s.guided_rounds == 0
        ref = state(s)
    with gpu_lib.Solver(cm, cap, pen) as s:
        s.solve()
        assert s.rounds == n and same(state(s), ref)
        assert n // 3 < s.guided_rounds < n if trips else s.guided_rounds == n
        s.reset()
        for r in (n // 2, 1, 1, 150, 700, 900, 1, -1):
            before = s.rounds
            s.solve(r)
            assert s.rounds == (n if r < 0 else min(n, before + r))
        assert same(state(s), ref)
    if kind == "near":
        return
    with gpu_lib.Solver(cm, cap, pen, cluster=1) as s:
        s.solve()
        assert s.stats().cluster_size == 1 and same(state(s), ref)


def test_in_batches_and_on_the_server(gpu_lib):
    kinds = [("equal", 12000, 300), ("near", 3000, 40), ("equal", 9000, 260), ("equal", 500, 20)]
    insts = [one_center(n, k, kind) for kind, n, k in kinds]
    refs = []
    for cm, cap, pen in insts:
        with gpu_lib.Solver(cm, cap, pen, npath_reuse=False) as s:
            s.solve()
            refs.append(state(s))
    solvers = [gpu_lib.Solver(*x) for x in insts]
    try:
        b = gpu_lib.Batch(solvers)
        for steps in ((-1,), (6400, 50, 50, 700, 1, 1400, -1)):
            for r in steps:
                want = [s.n if r < 0 else min(s.n, s.rounds + r) for s in solvers]
                b.run(r)
                assert [s.rounds for s in solvers] == want
            for s, ref in zip(solvers, refs):
                assert same(state(s), ref)
            assert solvers[0].guided_rounds < solvers[0].n
            for s in solvers:
                s.reset()
        b.close()
        gpu_lib.solve_batch([s.h for s in solvers], cluster_size=2)
        for s, ref in zip(solvers, refs):
            assert same(state(s), ref)
    finally:
        for s in solvers:
            s.close()
    with gpu_lib.Server(budget_bytes=4 << 30, quantum_us=20000) as srv:
        tickets = [srv.submit(*x) for x in insts]
        for t, ref in zip(tickets, refs):
            info, a = srv.result(t, 300_000)
            assert info.objective == ref[0] and np.array_equal(a, ref[1])


def test_strict_and_inserted_units(gpu_lib):
    cm, cap, pen = one_center(12000, 300, "equal")
    with gpu_lib.Solver(cm, cap, None, strict=True, ncyc_skip=False) as s:
        s.solve()
        ref = s.objective, s.assignment()
    with gpu_lib.Solver(cm, cap, None, strict=True) as s:
        s.solve()
        assert s.objective == ref[0] and np.array_equal(s.assignment(), ref[1])
    got = []
    for kw in ({}, {"npath_reuse": False}):
        with gpu_lib.Solver(cm[:8000], cap, pen, **kw) as s:
            s.solve()
            for row in cm[8000:8040]:
                s.insert(row)
                s.solve()
            got.append(state(s))
    assert same(*got)
