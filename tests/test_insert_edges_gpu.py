"""Insertion at the edges of its warps, CTAs and grid: edge counts around a warp,
two CTAs' 1,024 edges and two passes of the whole grid; endpoints that repeat
along an edge list (a hub as every source, as every target, in runs that cross
warps, scattered), which share one atomic per run; and a bad edge anywhere, after
which the graph is as before.  The packed CSR must equal a host sort of the edges
inserted, the exploited costs Dijkstra's."""
import numpy as np
import pytest

import oracle as O
import paper_2003_04920_gb300 as P
from paper_2003_04920_gb300 import workloads as W
from tests.gpu_util import assert_parity
from tests.test_parity_gpu import _csr_matches

pytestmark = pytest.mark.gpu


def _edges(rng, kind, n, m):
    i = np.arange(m)
    if kind == "hub source":
        u, v = np.zeros(m, np.int64), 1 + i % (n - 1)
    elif kind == "hub target":
        u, v = 1 + i % (n - 1), np.zeros(m, np.int64)
    elif kind == "runs":  # 1 .. 70 edges in a row from one vertex
        u = np.repeat(rng.integers(0, n, m), rng.integers(1, 71, m))[:m]
        v = (u + 1 + rng.integers(0, n - 1, m)) % n
    else:
        u = rng.integers(0, n, m)
        v = (u + 1 + rng.integers(0, n - 1, m)) % n
    return u.astype(np.int32), v.astype(np.int32)


def _check(D, n, us, vs, cs):
    u, v, c = np.concatenate(us), np.concatenate(vs), np.concatenate(cs)
    off, col, cost = D.get_adjacency()
    _csr_matches(off, col, cost, u, v, c, n)
    D.exploit()
    rm = W.Roadmap("edges", np.zeros((n, 2)), u, v, c, np.zeros(n + 1, np.int64), n)
    d, _ = O.dijkstra(n, u, v, c.astype(np.float64))
    assert_parity(rm, D.get_costs(), D.get_parents(), d)


@pytest.mark.parametrize("kind", ["hub source", "hub target", "runs", "scattered"])
@pytest.mark.parametrize("m", [1, 31, 33, 1023, 1025, 304 * 1024 + 7])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_edge_counts_and_runs(kind, m, dtype):
    rng = np.random.default_rng(m)
    n = 40 if m < 100 else 900
    with P.Graph(n, 3 * m, 0, dtype) as D:
        us, vs, cs = [], [], []
        for b in range(3):  # the first block brings the vertices, the others old rows only
            u, v = _edges(rng, kind, n, m)
            c = rng.uniform(1.0, 3.0, m).astype(dtype)
            D.insert_batch(n if b == 0 else 0, u, v, c)
            us.append(u), vs.append(v), cs.append(c)
        _check(D, n, us, vs, cs)


@pytest.mark.parametrize("at", [0, 31, 32, 4999])
def test_a_bad_edge_leaves_the_graph_as_it_was(at):
    rng = np.random.default_rng(3)
    n, m = 500, 5000
    with P.Graph(n + 10, 4 * m, 0, np.float32) as D:
        u, v = _edges(rng, "runs", n, m)
        c = rng.uniform(1.0, 3.0, m).astype(np.float32)
        D.insert_batch(n, u, v, c)
        D.exploit()
        for dst, cost in ((n + 10, 1.0), (-1, 1.0), (u[at], 1.0), (v[at], np.nan), (v[at], 0.0)):
            vb, cb = v.copy(), c.copy()
            vb[at], cb[at] = dst, cost
            with pytest.raises(P.PirrtError):
                D.insert_batch(10, u, vb, cb)
            assert D.n == n and D.m == 2 * m
        u2, v2 = _edges(rng, "scattered", n, m)
        c2 = rng.uniform(1.0, 3.0, m).astype(np.float32)
        D.insert_batch(0, u2, v2, c2)
        _check(D, n, [u, u2], [v, v2], [c, c2])
