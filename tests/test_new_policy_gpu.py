"""AUTO above 10^6 vertices: after a policy handed in, FP32 costs are evaluated by
pointer jumping and FP64 costs by waves first (which meet the level cap here, so that
jumping follows); a small block after it, FP32, by waves.
Costs are Dijkstra's bit for bit (sums of multiples of 2^-10)."""
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
def test_the_evaluate_after_a_policy(dtype):
    n = 1_000_001
    rng = np.random.default_rng(1)
    i = np.arange(1, n)
    par = np.r_[-1, (i * rng.random(n - 1) ** 0.5).astype(np.int64)]
    u = np.r_[par[1:], rng.integers(0, n - 1, n)]
    v = np.r_[i, u[n - 1:] + 1]
    c = rng.integers(512, 1024, len(u)) / 1024.0
    late = np.arange(1, 41) * 1000
    with P.Graph(n, len(u) + 40, 0, dtype) as G:
        G.insert_batch(n, u.astype(np.int32), v.astype(np.int32), c.astype(dtype))
        G.set_policy(par.astype(np.int32))
        st = G.exploit()
        assert (st["wave_levels"] == 0) == (dtype == np.float32) and st["switches"] > 0
        d, _ = O.dijkstra(n, u.astype(np.int32), v.astype(np.int32), c)
        np.testing.assert_array_equal(G.get_costs(), d)
        G.insert_batch(0, np.zeros(40, np.int32), late.astype(np.int32), np.full(40, 0.25, dtype))
        st = G.exploit()
        assert st["switches"] > 0
        if dtype == np.float32:
            assert st["wave_levels"] > 0
        d, _ = O.dijkstra(n, np.r_[u, np.zeros(40)].astype(np.int32),
                          np.r_[v, late].astype(np.int32), np.r_[c, np.full(40, 0.25)])
        np.testing.assert_array_equal(G.get_costs(), d)
