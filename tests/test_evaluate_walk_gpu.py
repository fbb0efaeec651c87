"""The allocation-free Evaluate at the edges of its grid and of its rounds:
one vertex, a CTA's last vertex and the next, one vertex per thread of the
chip and one more, several per thread, and policies whose depth sits on either
side of a power of four (a round multiplies the links a record spans by four),
up to a path through every vertex that the static scratch serves.

g is a sum of non-negative terms.  A round adds four links in pairs (two
additions deep) and the finishing round one more, so after r rounds the relative
error is at most (2 r + 1) u with u = 2^-53; nine rounds serve the deepest
policy of 262,144 vertices: 19 u, 2.2e-15, against sums in extended precision.
"""
import numpy as np
import pytest

import paper_2003_04920_gb300 as P

pytestmark = pytest.mark.gpu

RTOL = 19 * 2.0 ** -53
MAX_N = 1 << 18


def _evaluate(parent, cost, root=0):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pt = torch.from_numpy(parent.astype(np.int32)).cuda()
    ct = torch.from_numpy(cost).cuda()
    out = torch.full((len(parent),), -7.0, dtype=torch.float64, device="cuda")
    return P.pirrt_evaluate_noalloc(pt, ct, out, root=root), out.cpu().numpy()


def _check(parent, cost, order, root=0):
    """order: every vertex after its parent."""
    rc, g = _evaluate(parent, cost, root)
    assert rc == P.PIRRT_OK
    want = [np.longdouble(np.inf)] * len(parent)
    want[root] = np.longdouble(0)
    par, c = parent.tolist(), cost.astype(np.longdouble)
    for v in order.tolist():
        if v != root and par[v] >= 0:
            want[v] = want[par[v]] + c[v]
    want = np.array(want)
    np.testing.assert_array_equal(np.isinf(g), np.isinf(want))
    fin = np.isfinite(want)
    assert np.all(np.abs(g[fin] - want[fin]) <= RTOL * want[fin])


@pytest.mark.parametrize("n", [1, 2, 511, 512, 513, 152 * 512, 152 * 512 + 1, 152 * 2048 // 2 + 7,
                               MAX_N - 1, MAX_N])
@pytest.mark.parametrize("share", [0.05, 1.0])
def test_random_trees(n, share):
    rng = np.random.default_rng(n)
    i = np.arange(n)
    perm = rng.permutation(n)
    parent = np.full(n, -1, dtype=np.int64)
    up = np.minimum((i * (1.0 - share * rng.random(n))).astype(np.int64), np.maximum(i - 1, 0))
    parent[perm[1:]] = perm[up[1:]]
    parent[perm[1 + rng.integers(0, max(n - 1, 1), n // 1000)] if n > 1000 else []] = -1
    cost = rng.random(n)
    _check(parent, cost, perm, root=int(perm[0]))


@pytest.mark.parametrize("n", [2, 4, 5, 16, 17, 64, 65, 1024, 1025, 16384, 16385, MAX_N])
def test_paths(n):
    rng = np.random.default_rng(n)
    perm = rng.permutation(n)
    parent = np.full(n, -1, dtype=np.int64)
    parent[perm[1:]] = perm[:-1]
    _check(parent, 1e-3 + rng.random(n), perm, root=int(perm[0]))


def test_a_long_cycle_and_the_next_call():
    n = 40_000
    parent = np.arange(-1, n - 1)
    parent[20_000] = 39_999  # 20,000 .. 39,999 form a cycle
    rc, g = _evaluate(parent, np.ones(n))
    assert rc == P.PIRRT_ERR_BAD_TREE
    np.testing.assert_array_equal(g[:20_000], np.arange(20_000.0))
    assert np.all(np.isinf(g[20_000:]))
    parent[20_000] = 19_999
    rc, g = _evaluate(parent, np.ones(n))
    assert rc == P.PIRRT_OK
    np.testing.assert_array_equal(g, np.arange(float(n)))
