"""A sweep in which almost every vertex switches: more switches than a CTA stages, with
one and with two CTAs per SM, by waves and by pointer jumping.  A path as the policy
of a graph with many cross edges; costs are multiples of 2^-10, so sums are exact and
the costs are Dijkstra's bit for bit."""
import numpy as np
import pytest

import oracle as O
import paper_2003_04920_gb300 as P

pytestmark = pytest.mark.gpu
N = 200_000


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P.load_library()


@pytest.fixture(scope="module")
def graph():
    rng = np.random.default_rng(77)
    a = rng.integers(0, N, (2, 3 * N))
    a = a[:, a[0] != a[1]]
    u = np.r_[np.arange(N - 1), a[0]].astype(np.int32)
    v = np.r_[np.arange(1, N), a[1]].astype(np.int32)
    c = rng.integers(512, 1024, len(u)) / 1024.0
    return u, v, c, O.dijkstra(N, u, v, c)[0]


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("evaluate", ["auto", "wave", "jump"])
@pytest.mark.parametrize("ctas", [0, 1, 2])
def test_costs_and_counts(graph, dtype, evaluate, ctas):
    u, v, c, d = graph
    with P.Graph(N, len(u), 0, dtype) as G:
        G.insert_batch(N, u, v, c.astype(dtype))
        G.set_policy(np.r_[np.int32(-1), u[:N - 1]].astype(np.int32))
        st = G.exploit(evaluate=evaluate, wave_ctas=ctas)
        got, p = G.get_costs(), G.get_parents()
    np.testing.assert_array_equal(got, d)
    assert st["switches"] > N and st["dense_sweeps"] > 1
    assert p[0] == -1 and (p[1:] >= 0).all()
