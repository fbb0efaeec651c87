"""A grid step whose list overflows: a hub's late edge lowers its children, each over
sixteen parallel edges in random order, so that the step lowers every child three
times on average (the mean number of running minima of sixteen) and takes more
entries than the graph has vertices.  Neighbours that only a child's new cost
improves are found all the same, by a dense sweep.

The costs are multiples of 2^-10 below 64: every sum is exact."""
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


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("host_loop", [False, True])
def test_children_lost_from_a_step(dtype, host_loop):
    rng = np.random.default_rng(11)
    m, par = 3000, 16
    kids, side = 2 + np.arange(m), 2 + m + np.arange(m)
    n = 2 + 2 * m
    many = np.repeat(kids, par)
    cost = rng.integers(256, 1024, len(many)) / 1024.0
    order = rng.permutation(len(many))
    u = np.r_[0, np.ones(len(many), np.int64), np.zeros(m, np.int64), kids]
    v = np.r_[1, many[order], side, side]
    c = np.r_[20.0, cost[order], np.full(m, 30.0), np.full(m, 12.0)]
    policy = np.r_[-1, 0, np.ones(m, np.int64), np.zeros(m, np.int64)].astype(np.int32)
    with P.Graph(n, len(u) + 1, 0, dtype) as G:
        G.insert_batch(n, u.astype(np.int32), v.astype(np.int32), c.astype(dtype))
        G.set_policy(policy)
        assert G.exploit(evaluate="wave")["switches"] == 0
        G.insert_batch(0, [0], [1], np.array([0.125], dtype))
        st = G.exploit(evaluate="wave", dense_fraction=1.0, host_loop=host_loop)
        got = G.get_costs()
    d, _ = O.dijkstra(n, np.r_[u, 0].astype(np.int32), np.r_[v, 1].astype(np.int32),
                      np.r_[c, 0.125])
    np.testing.assert_array_equal(got, d)
    if not host_loop:
        assert st["jump_evaluates"] == 1 and st["dense_sweeps"] >= 1  # it did overflow
