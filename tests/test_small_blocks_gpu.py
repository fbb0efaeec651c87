"""AUTO on a goal-free graph above 2*10^5 vertices: a small block is evaluated by waves,
a large one or a new policy by pointer jumping; up to 2*10^5 every block by jumping.
Costs are those of Dijkstra's algorithm bit for bit (sums of multiples of 2^-10)."""
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


@pytest.mark.parametrize("n,waves", [(200_000, False), (200_001, True)])
def test_the_evaluate_follows_the_block(n, waves):
    rng = np.random.default_rng(n)
    i = np.arange(1, n)
    u = np.r_[(i * rng.random(n - 1)).astype(np.int64), rng.integers(0, n - 1, 2 * n)]
    v = np.r_[i, u[n - 1:] + 1]
    c = rng.integers(512, 1024, len(u)) / 1024.0
    few, many = 40, len(u) // 100
    late = rng.integers(0, n - 1, (2, 2 * few + many))
    late[1] += late[1] >= late[0]
    lc = rng.integers(1, 512, late.shape[1]) / 1024.0
    u, v, c = np.r_[u, late[0]].astype(np.int32), np.r_[v, late[1]].astype(np.int32), np.r_[c, lc]
    at = np.cumsum([0, 3 * n - 1, few, many, few])
    with P.Graph(n, len(u), 0, np.float32) as G:
        for k, by_wave in enumerate((False, waves, False, None)):
            e0, e1 = at[k], at[k + 1]
            G.insert_batch(n if k == 0 else 0, u[e0:e1], v[e0:e1], c[e0:e1].astype(np.float32))
            if by_wave is None:  # a policy handed in is new as a whole
                G.set_policy(p)
                by_wave = False
            st = G.exploit()
            assert st["switches"] > 0
            assert (st["wave_levels"] > 0) == by_wave
            assert (st["jump_evaluates"] > 0) == (not by_wave)
            g, p = G.get_costs(), G.get_parents()
            d, _ = O.dijkstra(n, u[:e1], v[:e1], c[:e1])
            np.testing.assert_array_equal(g, d)
