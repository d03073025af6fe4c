"""Road graphs that leave the grid's shape, against the oracle's Dijkstra:
nodes of more than 8 roads, frontiers past the shared-memory lists, lengths
spread over four decades, one-way roads, and a graph whose bitmaps do not fit
shared memory."""
from types import SimpleNamespace

import numpy as np
import pytest

import oracle
from test_gpu_road import gpu_cm

pytestmark = pytest.mark.gpu


def csr(V, src, dst, w, k, seed):
    o = np.lexsort((dst, src))
    row_ptr = np.zeros(V + 1, np.int32)
    row_ptr[1:] = np.cumsum(np.bincount(src, minlength=V))
    rng = np.random.default_rng(seed)
    centers = np.sort(rng.permutation(V)[:k]).astype(np.int32)
    demand = np.setdiff1d(np.arange(V, dtype=np.int32), centers)
    return SimpleNamespace(V=V, row_ptr=row_ptr, col=dst[o].astype(np.int32),
                           w=w[o].astype(np.int32), centers=centers, demand=demand)


def both(a, b, w):
    return np.concatenate([a, b]), np.concatenate([b, a]), np.concatenate([w, w])


def hubs():
    """Two hubs of 6,000 spokes each, joined: 6,000-node frontiers."""
    m = 6000
    a = np.concatenate([np.zeros(m, int), np.full(m, 1), [0]])
    b = np.concatenate([2 + np.arange(m), 2 + m + np.arange(m), [1]])
    w = 1 + (np.arange(len(a)) * 7919) % 500
    return csr(2 + 2 * m, *both(a, b, w), 5, 1)


def random_graph(seed, V, deg, wmax):
    """A ring (so that every node is reached) plus random one-way roads, a few
    nodes with most of them."""
    rng = np.random.default_rng(seed)
    ring = np.arange(V)
    E = V * deg
    a = np.concatenate([ring, np.where(rng.random(E) < 0.1, rng.integers(0, 5, E),
                                       rng.integers(0, V, E))])
    b = np.concatenate([np.roll(ring, -1), rng.integers(0, V, E)])
    w = np.maximum(1, np.exp(rng.random(len(a)) * np.log(wmax))).astype(np.int64)
    return csr(V, a, b, w, 9, seed)


def grid(W, H, k):
    idx = np.arange(W * H).reshape(H, W)
    a = np.concatenate([idx[:, :-1].ravel(), idx[:-1].ravel()])
    b = np.concatenate([idx[:, 1:].ravel(), idx[1:].ravel()])
    w = 50 + (np.arange(len(a)) * 2654435761) % 200
    return csr(W * H, *both(a, b, w), k, 3)


@pytest.mark.parametrize("name", ["hubs", "random3", "random9", "line", "large"])
def test_road_graph_matches_dijkstra(gpu_lib, name):
    g = {"hubs": hubs, "random3": lambda: random_graph(5, 3000, 3, 10000),
         "random9": lambda: random_graph(6, 2000, 9, 300), "line": lambda: grid(900, 1, 3),
         "large": lambda: grid(700, 600, 2)}[name]()
    rc, ref = oracle.road_cm(g.row_ptr, g.col, g.w, g.centers, g.demand)
    assert rc == 0
    assert np.array_equal(gpu_cm(gpu_lib, g), ref)


def test_longest_accepted_lengths(gpu_lib):
    """Roads back from a node whose distance is close to 2^31: the sum one road
    further passes 2^31 and must not lower a label."""
    t = lambda *a: np.array(a, np.int32)
    x = 700_000_000
    ring = SimpleNamespace(V=4, row_ptr=t(0, 1, 2, 3, 4), col=t(1, 2, 3, 0), w=t(x, x, x, x),
                           centers=t(0), demand=t(1, 2, 3))
    y = 1_000_000_000
    line = SimpleNamespace(V=3, row_ptr=t(0, 1, 3, 4), col=t(1, 0, 2, 1), w=t(y, y, y, y),
                           centers=t(0, 2), demand=t(1))
    z = 2**31 - 2
    pair = SimpleNamespace(V=2, row_ptr=t(0, 1, 2), col=t(1, 0), w=t(z, z), centers=t(0),
                           demand=t(1))
    # a node of 9 roads: the last ones are read from its CSR row
    m = 200_000_000
    hub = both(np.zeros(9, int), 1 + np.arange(9), np.full(9, m))
    star = csr(10, *hub, 1, 2)
    for g in (ring, line, pair, star):
        rc, ref = oracle.road_cm(g.row_ptr, g.col, g.w, g.centers, g.demand)
        assert rc == 0
        assert np.array_equal(gpu_cm(gpu_lib, g), ref)
