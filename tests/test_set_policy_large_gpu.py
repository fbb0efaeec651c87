"""set_policy around the size from which it runs two CTAs per SM: the last policy with
one, the first with two; bad entries at the far end are refused and leave the graph."""
import numpy as np
import pytest

import paper_2003_04920_gb300 as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P.load_library()


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n", [500_000, 500_001, 777_777])
def test_costs_of_a_large_policy(n, dtype):
    rng = np.random.default_rng(n)
    i = np.arange(1, n)
    par = np.r_[-1, (i * rng.random(n - 1) ** 0.3).astype(np.int64)].astype(np.int32)
    u, v = par[1:], i.astype(np.int32)
    cheap = rng.integers(512, 1024, n - 1) / 1024.0  # sums are exact
    with P.Graph(n, 2 * n, 0, dtype) as G:
        G.insert_batch(n, u, v, cheap.astype(dtype))
        G.insert_batch(0, u, v, (cheap + 0.5).astype(dtype))
        par[n // 3] = -1  # a subtree without a root
        G.set_policy(par)
        g, p = G.get_costs(), G.get_parents()
        want = np.full(n, np.inf)
        want[0] = 0.0
        parents, costs = par.tolist(), cheap.tolist()
        for x in range(1, n):
            if parents[x] >= 0:
                want[x] = want[parents[x]] + costs[x - 1]
        np.testing.assert_array_equal(g, want)
        np.testing.assert_array_equal(p, par)
        for at, bad in ((n - 1, n), (n - 1, n - 2 if par[n - 1] != n - 2 else n - 3), (0, 1)):
            wrong = par.copy()
            wrong[at] = bad
            with pytest.raises(P.PirrtError) as e:
                G.set_policy(wrong)
            assert e.value.status == P.PIRRT_ERR_BAD_INPUT
            np.testing.assert_array_equal(G.get_costs(), g)
