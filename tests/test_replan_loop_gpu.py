"""The one-launch Replan loop against the host-driven loop of separate kernels
and the oracle's shortest paths, at the sizes where its staging can go wrong:
rows longer than one pass, more lowered children than a CTA stages, more listed
vertices than it stages, parallel edges, chains deeper than the rounds summed
from the root, single vertices, and every grid size in between."""
import numpy as np
import pytest

import oracle as O
import paper_2003_04920_gb300 as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P.load_library()


def _graph(kind, rng):
    """(n, u, v, cost, initial parents, late edges): the late edges arrive after
    the first exploit and lower whole subtrees."""
    if kind == "star":  # one vertex with 3000 children, two leaves below each
        k = 3000
        hub, kids = 1, np.arange(2, 2 + k)
        leaf = np.arange(2 + k, 2 + 3 * k)
        u = np.r_[0, np.full(k, hub), np.repeat(kids, 2)]
        v = np.r_[hub, kids, leaf]
        par = np.full(2 + 3 * k, -1)
        par[v] = u
    elif kind == "chain":  # 150 levels, 40 side edges that never win
        u, v = np.arange(149), np.arange(1, 150)
        par = np.r_[-1, np.arange(149)]
    elif kind == "double":  # every edge of a random tree three times
        n = 700
        v = np.arange(1, n)
        u = (v * rng.random(n - 1) ** 0.5).astype(np.int64)
        par = np.r_[-1, u]
        u, v = np.tile(u, 3), np.tile(v, 3)
    else:  # "mesh": a tree of 4000 with many cross edges, rows of up to ~100
        n = 4000
        v = np.arange(1, n)
        u = (v * rng.random(n - 1)).astype(np.int64)
        par = np.r_[-1, u]
        a, b = rng.integers(0, n, (2, 60_000))
        keep = a != b
        u, v = np.r_[u, a[keep]], np.r_[v, b[keep]]
    n = len(par)
    c = rng.uniform(0.5, 1.0, len(u))
    late = (np.array([0, n]), np.array([n, 1]), np.array([1e-3, 1e-3]))
    return n, u.astype(np.int32), v.astype(np.int32), c, par.astype(np.int32), late


def _run(g, dtype, **kw):
    n, u, v, c, par, (lu, lv, lc) = g
    with P.Graph(n + 1, len(u) + 2, 0, dtype) as G:
        G.insert_batch(n, u, v, c.astype(dtype))
        G.set_policy(par)
        s0 = G.exploit(**kw)
        G.insert_batch(1, lu.astype(np.int32), lv.astype(np.int32), lc.astype(dtype))
        s1 = G.exploit(**kw)
        return G.get_costs(), G.get_parents(), (s0, s1)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("evaluate", ["auto", "wave", "jump"])
@pytest.mark.parametrize("kind", ["star", "chain", "double", "mesh"])
def test_loop_equals_host_loop_and_dijkstra(kind, evaluate, dtype):
    g = _graph(kind, np.random.default_rng(7))
    gc, pc, sc = _run(g, dtype, evaluate=evaluate)
    gh, ph, sh = _run(g, dtype, evaluate=evaluate, host_loop=True)
    assert [s["graph_launch"] for s in sc] == [1, 1] and [s["graph_launch"] for s in sh] == [0, 0]
    assert [s["iterations"] for s in sc] == [s["iterations"] for s in sh]
    assert [s["switches"] for s in sc] == [s["switches"] for s in sh]
    np.testing.assert_array_equal(pc, ph)
    n, u, v, c, _, (lu, lv, lc) = g
    d, _ = O.dijkstra(n + 1, np.r_[u, lu].astype(np.int32), np.r_[v, lv].astype(np.int32),
                      np.r_[c, lc].astype(dtype))
    # the wave's sums are the host-driven wave's, bit for bit.  FP32 costs of one
    # binade and a half sum exactly; FP64 sums by pointer jumping (set_policy
    # evaluates so) are reassociated, which over a path of at most 150 edges moves
    # a cost by less than 150 ulp
    if evaluate == "wave":
        np.testing.assert_array_equal(gc, gh)
    if dtype == np.float32:
        np.testing.assert_array_equal(gc, d)
    else:
        np.testing.assert_allclose(gc, d, rtol=150 * 2.0 ** -52, atol=0)


@pytest.mark.parametrize("n", [1, 2, 31, 33, 127, 129, 1025, 19_456, 19_457])
def test_every_grid_size(n):
    """A path with shortcuts, so that lists of every length occur."""
    rng = np.random.default_rng(n)
    u, v = np.arange(n - 1), np.arange(1, n)
    m = 3 * n if n > 2 else 0
    a, b = rng.integers(0, n, (2, m))
    keep = a != b
    u, v = np.r_[u, a[keep]].astype(np.int32), np.r_[v, b[keep]].astype(np.int32)
    c = rng.uniform(0.5, 1.0, len(u)).astype(np.float32)
    for evaluate in ("auto", "wave"):
        with P.Graph(n, max(len(u), 1), 0, np.float32) as G:
            G.insert_batch(n, u, v, c)
            st = G.exploit(evaluate=evaluate)
            gc = G.get_costs()
        assert st["converged"] == 1
        d, _ = O.dijkstra(n, u, v, c)
        np.testing.assert_array_equal(gc, d)
