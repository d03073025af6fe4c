"""Short first calls: the prologue of many units runs on a cluster of its own
before the rounds on one CTA, in lone solves, batches and served passes."""
import numpy as np
import pytest

import lbdd_inputs as L
import oracle

pytestmark = pytest.mark.gpu


def check(s, ref):
    assert s.objective == ref.delta and np.array_equal(s.assignment(), ref.assign)
    assert np.array_equal(s.loads().astype(np.int64), ref.load)


# (n, k, added to every cost): around the size from which it has its own launch
CASES = [(2990, 30, 0), (3000, 30, 0), (4100, 40, 0), (4100, 40, 40000), (900, 500, 0)]


@pytest.mark.parametrize("n,k,add", CASES)
def test_short_calls_match_oracle(gpu_lib, n, k, add):
    inst = L.random_small(8800 + n + k, n=n, k=k, cm_max=60, cap_frac=0.6, pen=(5, 90))
    cm = inst.cm + np.int32(add)
    ref = oracle.asral(cm, inst.cap, inst.pen)
    with gpu_lib.Solver(cm, inst.cap, inst.pen) as s:
        for first in (0, 1, n // 16 - 1, n // 16, -1):   # the last two leave it to the rounds' CTA
            s.reset()
            s.solve(first)
            assert s.rounds == (n if first < 0 else first)
            assert s.stats().cluster_size == 1
            s.solve()
            check(s, ref)


def test_short_batch_and_served_passes_match_oracle(gpu_lib):
    insts = [L.random_small(8900 + i, n=n, k=k, cm_max=60, cap_frac=0.6, pen=(5, 90))
             for i, (n, k) in enumerate([(4500, 40), (300, 12), (6000, 25), (5000, 33), (700, 450)])]
    refs = [oracle.asral(x.cm, x.cap, x.pen) for x in insts]
    solvers = [gpu_lib.Solver(x.cm, x.cap, x.pen) for x in insts]
    try:
        b = gpu_lib.Batch(solvers)
        for again in range(2):
            b.run(3)
            assert [s.rounds for s in solvers] == [3] * len(solvers)
            b.run(5)
            b.run()
            for s, ref in zip(solvers, refs):
                check(s, ref)
                s.reset()
        b.close()
    finally:
        for s in solvers:
            s.close()
    with gpu_lib.Server(budget_bytes=4 << 30, quantum_us=150) as srv:   # below four prologues
        tickets = [srv.submit(x.cm, x.cap, x.pen) for x in insts]
        for t, ref in zip(tickets, refs):
            info, a = srv.result(t, 300_000)
            assert info.objective == ref.delta and np.array_equal(a, ref.assign)


@pytest.mark.parametrize("how", ["solve", "batch"])
def test_prologue_of_a_short_call_is_shared(gpu_lib, how):
    """100,000 x 300: one CTA's prologue takes about four times as long as
    eight CTAs'."""
    import torch
    n, k = 100_000, 300
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    cm = torch.randint(1, 20000, (n, k), generator=g, device="cuda", dtype=torch.int16)
    cap, pen = np.full(k, n // k, np.int32), np.full(k, 500, np.int32)
    took = []
    for cluster in (0, 1):
        with gpu_lib.Solver(cm, cap, pen, cluster=cluster) as s:
            best = 1 << 62
            for _ in range(3):
                s.reset()
                if how == "solve" or cluster == 1:
                    s.solve(4)
                else:
                    gpu_lib.Batch([s]).run(4)
                best = min(best, s.stats().prologue_ns)
            took.append(best)
    assert 2 * took[0] < took[1]
