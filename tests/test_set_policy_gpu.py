"""set_policy at the edges of its launch: the fewest vertices, one row more than a
warp's four and a CTA's share, rows shorter and longer than the eight lanes that
read them, parallel edges (the cheapest counts), vertices without a parent; and a
bad entry at the first, middle or last vertex, which leaves the graph as it was.

g is a sum of non-negative terms: a round adds four links in pairs and the last
round one value more, so after r rounds (r <= 7 below 4^7 vertices) the error is at
most (2 r + 1) u = 15 u of the exact sum."""
import numpy as np
import pytest

import paper_2003_04920_gb300 as P

pytestmark = pytest.mark.gpu
RTOL = 15 * 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P.load_library()


def _case(n, rng):
    order = np.r_[0, 1 + rng.permutation(n - 1)] if n > 1 else np.zeros(1, np.int64)
    i = np.arange(1, n)
    par = np.full(n, -1)
    par[order[i]] = order[np.minimum((i * rng.random(n - 1) ** 0.3).astype(np.int64), i - 1)]
    u, v = par[order[i]], order[i]
    hub = np.full(min(n - 1, 300), 0), np.arange(1, min(n, 301))  # one long row
    u, v = np.r_[u, u, hub[0]], np.r_[v, v, hub[1]]  # every tree edge twice
    return par.astype(np.int32), order, u.astype(np.int32), v.astype(np.int32), \
        rng.uniform(0.5, 2.0, len(u))


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n", [1, 2, 5, 63, 65, 513, 9729, 16_383])
def test_costs_of_a_policy(n, dtype):
    rng = np.random.default_rng(n)
    par, order, u, v, c = _case(n, rng)
    c = c.astype(dtype)
    if n > 5:
        par[rng.integers(1, n, 3)] = -1  # subtrees without a root
    best = {}
    for a, b, w in zip(u.tolist(), v.tolist(), c.astype(np.longdouble)):
        k = (min(a, b), max(a, b))
        best[k] = min(w, best.get(k, np.inf))
    want = [np.longdouble(np.inf)] * n
    want[0] = np.longdouble(0)
    for x in order[1:].tolist():
        if par[x] >= 0:
            want[x] = want[par[x]] + best[(min(x, par[x]), max(x, par[x]))]
    want = np.array(want)
    with P.Graph(n, max(len(u), 1), 0, dtype) as G:
        G.insert_batch(n, u, v, c)
        for _ in range(2):
            G.set_policy(par)
            g, p = G.get_costs(), G.get_parents()
            np.testing.assert_array_equal(p, par)
            np.testing.assert_array_equal(np.isinf(g), np.isinf(want))
            fin = np.isfinite(want)
            assert np.all(np.abs(g[fin] - want[fin]) <= RTOL * want[fin])
        assert G.exploit()["converged"] == 1


@pytest.mark.parametrize("at", [1, 700, 1499])
def test_a_bad_entry_leaves_the_policy(at):
    rng = np.random.default_rng(at)
    n = 1500
    par, _, u, v, c = _case(n, rng)
    with P.Graph(n, len(u), 0, np.float32) as G:
        G.insert_batch(n, u, v, c.astype(np.float32))
        G.set_policy(par)
        g, p = G.get_costs(), G.get_parents()
        for wrong in (n, -2, at):  # out of range twice, and no edge to itself
            bad = par.copy()
            bad[at] = wrong
            with pytest.raises(P.PirrtError):
                G.set_policy(bad)
            np.testing.assert_array_equal(G.get_costs(), g)
            np.testing.assert_array_equal(G.get_parents(), p)
        bad = par.copy()
        bad[0] = 1  # a root with a parent
        with pytest.raises(P.PirrtError):
            G.set_policy(bad)
        G.set_policy(par)
        np.testing.assert_array_equal(G.get_costs(), g)
