"""AUTO above 10^6 vertices, FP32 costs: iterations that switch more than an eighth of the
vertices are evaluated by pointer jumping, the others by waves, and jumping by choice
does not make the next exploit take the trees for deep.  Costs are Dijkstra's bit for
bit (sums of multiples of 2^-10)."""
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


@pytest.mark.parametrize("goal", [False, True])
def test_iterations_choose(goal):
    n = 1_000_001
    rng = np.random.default_rng(2)
    i = np.arange(1, n)
    u = np.r_[(i * rng.random(n - 1) ** 3).astype(np.int64),
              (i * rng.random(n - 1) ** 3).astype(np.int64)]  # a few links deep
    v = np.r_[i, i]
    order = np.argsort(v, kind="stable")
    u, v = u[order], v[order]
    c = rng.integers(512, 1024, len(u)) / 1024.0
    late = np.arange(1, 21) * 1000
    lu, lv = np.r_[u, np.zeros(20, np.int64)], np.r_[v, late]
    lc = np.r_[c, np.full(20, 2.0 ** -10)]
    with P.Graph(n, len(lu), 0, np.float32) as G:
        if goal:
            G.set_goal(n - 1)
        for e0, e1, n_new in ((0, len(u), n), (len(u), len(lu), 0)):
            G.insert_batch(n_new, lu[e0:e1].astype(np.int32), lv[e0:e1].astype(np.int32),
                           lc[e0:e1].astype(np.float32))
            st = G.exploit()
            assert st["wave_levels"] > 0 and st["switches"] > 0
            assert (st["jump_evaluates"] > 0) == (n_new > 0 and not goal)
            if not goal:
                d, _ = O.dijkstra(n, lu[:e1].astype(np.int32), lv[:e1].astype(np.int32), lc[:e1])
                np.testing.assert_array_equal(G.get_costs(), d)
