"""The walk in shared memory (small policies) at its edges: the fewest vertices,
a CTA's last vertex and the next, the largest policy of each cost type and one
more (which pointer jumping takes), and chains around the 96 links that FP64 costs
keep on the stack.

FP32 costs add without rounding in FP64 here (24-bit costs of similar size, fewer
than 2^20 links), so costs and parents are those of the host-driven loop bit for
bit.  FP64 costs of a chain of at most 97 vertices are the sums from the root down
bit for bit; deeper ones are within one rounding per link of the exact sum."""
import numpy as np
import pytest

import oracle as O
import paper_2003_04920_gb300 as P
from tests.gpu_util import G_RTOL
from tests.test_replan_loop_gpu import _run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P.load_library()


def _tree(n, rng):
    """A random tree on ids in random order, as many cross edges, and a late edge
    that lowers much of it."""
    order = np.r_[0, 1 + rng.permutation(n - 1)] if n > 1 else np.zeros(1, np.int64)
    i = np.arange(1, n)
    par = np.full(n, -1)
    par[order[i]] = order[np.minimum((i * (1.0 - 0.4 * rng.random(n - 1))).astype(np.int64), i - 1)]
    u, v = par[order[i]], order[i]
    a, b = rng.integers(0, n, (2, n if n > 2 else 0))
    keep = a != b
    u, v = np.r_[u, a[keep]], np.r_[v, b[keep]]
    c = rng.uniform(0.5, 1.0, len(u))
    late = (np.array([0, n]), np.array([n, n - 1]), np.array([1e-3, 1e-3])) if n > 1 else \
        (np.array([0]), np.array([1]), np.array([1e-3]))
    return n, u.astype(np.int32), v.astype(np.int32), c, par.astype(np.int32), late


@pytest.mark.parametrize("n,dtype", [(1, np.float32), (2, np.float64), (5, np.float32),
                                     (511, np.float64), (513, np.float64), (1025, np.float32),
                                     (9727, np.float64), (9728, np.float64), (16383, np.float32),
                                     (16384, np.float32)])
def test_sizes(n, dtype):
    g = _tree(n, np.random.default_rng(n))
    gc, pc, sc = _run(g, dtype, evaluate="jump")
    gh, ph, _ = _run(g, dtype, evaluate="jump", host_loop=True)
    if dtype == np.float32:
        np.testing.assert_array_equal(gc, gh)
        np.testing.assert_array_equal(pc, ph)
    _, u, v, c, _, (lu, lv, lc) = g
    d, _ = O.dijkstra(n + 1, np.r_[u, lu].astype(np.int32), np.r_[v, lv].astype(np.int32),
                      np.r_[c, lc].astype(dtype).astype(np.float64))
    np.testing.assert_allclose(gc, d, rtol=G_RTOL, atol=0)


@pytest.mark.parametrize("depth", [1, 95, 96, 97, 98, 400])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_chains(depth, dtype):
    rng = np.random.default_rng(depth)
    n = depth + 1
    c = rng.uniform(0.5, 1.0, depth).astype(dtype)
    order = np.r_[0, 1 + rng.permutation(depth)].astype(np.int32)
    par = np.full(n, -1, np.int32)
    par[order[1:]] = order[:-1]
    with P.Graph(n, 2 * depth, 0, dtype) as G:
        G.insert_batch(n, order[:-1], order[1:], c)
        G.set_policy(par)
        G.exploit(evaluate="jump")
        # a cheaper parallel edge below the root lowers every vertex
        c[0] = dtype(0.25)
        G.insert_batch(0, order[:1], order[1:2], c[:1])
        G.exploit(evaluate="jump")
        got, parents = G.get_costs()[order], G.get_parents()
    np.testing.assert_array_equal(parents, par)
    want = np.cumsum(np.r_[0.0, c.astype(np.float64)])
    if dtype == np.float32 or depth <= 96:
        np.testing.assert_array_equal(got, want)
    else:
        np.testing.assert_allclose(got, want, rtol=depth * 2.0 ** -52, atol=0)
