"""A policy that the walk in shared memory gives up on: a bushy tree that fills the
graph's capacity with one chain around the 96 links it keeps, all of it lowered by
one late edge.  Every vertex is listed once: the marking that follows goes over the
entries of the listed vertices' rows, so `offers` counts them, and a list longer
than the graph would exceed a dense limit of all vertices.

A cost is a sum of at most depth + 1 terms, each addition rounding once."""
import numpy as np
import pytest

import paper_2003_04920_gb300 as P

pytestmark = pytest.mark.gpu
N = 9728  # the largest policy with FP64 costs that is walked


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P.load_library()


def _policy(n, depth, rng):
    """Parents of vertex 1 below the root, a random tree below it, and a chain whose
    last vertex is `depth` links from the root; costs of the links."""
    m = n - (depth - 1)
    i = np.arange(2, m)
    par = np.full(n, -1)
    par[1] = 0
    par[i] = 1 + ((i - 1) * (1.0 - 0.4 * rng.random(m - 2))).astype(np.int64).clip(0, i - 2)
    par[m] = 1
    par[m + 1:] = np.arange(m, n - 1)
    return par.astype(np.int32), rng.uniform(0.5, 1.0, n)


@pytest.mark.parametrize("goal", [False, True])
@pytest.mark.parametrize("depth", [95, 96, 97, 98, 400])
def test_every_changed_vertex_is_listed_once(depth, goal):
    rng = np.random.default_rng(depth)
    par, c = _policy(N, depth, rng)
    kw = dict(evaluate="auto" if goal else "jump", dense_fraction=1.0)
    with P.Graph(N, N, 0, np.float64) as G:
        if goal:
            G.set_goal(N - 1)
        G.insert_batch(N, par[1:], np.arange(1, N, dtype=np.int32), c[1:])
        G.set_policy(par)
        assert G.exploit(**kw)["switches"] == 0
        c[1] = 0.25
        G.insert_batch(0, [0], [1], c[1:2])
        st = G.exploit(**kw)
        entries = G.m
        got, parents = G.get_costs(), G.get_parents()
    np.testing.assert_array_equal(parents, par)
    assert st["switches"] == 1 and st["dense_sweeps"] == 0
    if not goal:
        assert st["offers"] == entries - 2  # every row but the root's, of two entries
    want = np.zeros(N, np.longdouble)
    links = np.zeros(N, np.int64)
    for v in range(1, N):
        want[v] = want[par[v]] + np.longdouble(c[v])
        links[v] = links[par[v]] + 1
    assert links[N - 1] == depth
    assert np.all(np.abs(got - want) <= (links + 1) * 2.0 ** -53 * want)
