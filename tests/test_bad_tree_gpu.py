"""A cycle in the parents: set_policy reports it, and so does every exploit until a
valid policy or an insertion takes the error away, as a reset does."""
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


def _path(n, dtype):
    """A path 0 - 1 - ... and its policy, with vertices n - 2 and n - 3 each other's
    parent in the second one."""
    u = np.arange(n - 2, dtype=np.int32)
    par = np.r_[-1, u].astype(np.int32)
    loop = par.copy()
    loop[n - 3] = n - 2
    c = np.random.default_rng(n).uniform(0.5, 1.0, n - 2).astype(dtype)
    return u, u + 1, c, par, loop


def _status(call, *a, **kw):
    try:
        call(*a, **kw)
    except P.PirrtError as e:
        return e.status
    return P.PIRRT_OK


# walked in shared memory, and by pointer jumping
@pytest.mark.parametrize("n,dtype", [(60, np.float32), (60, np.float64), (17_000, np.float32),
                                     (10_000, np.float64)])
def test_a_valid_policy_or_an_insertion_recovers(n, dtype):
    u, v, c, par, loop = _path(n, dtype)
    with P.Graph(n, 2 * n, 0, dtype) as G:
        G.insert_batch(n - 1, u, v, c)
        G.set_policy(par)
        G.exploit()
        assert _status(G.set_policy, loop) == P.PIRRT_ERR_BAD_TREE
        # one switch, so that the Evaluate goes over the policy
        G.insert_batch(1, [0], [n - 1], np.array([0.5], dtype))
        assert _status(G.exploit, evaluate="jump") == P.PIRRT_ERR_BAD_TREE
        G.insert_batch(0, [0], [n - 1], np.array([0.25], dtype))
        assert _status(G.exploit, evaluate="wave") == P.PIRRT_OK  # top-down, above the cycle
        G.set_policy(np.r_[par, 0].astype(np.int32))
        assert G.exploit()["converged"] == 1
        got = G.get_costs()
    d, _ = O.dijkstra(n, np.r_[u, 0].astype(np.int32), np.r_[v, n - 1].astype(np.int32),
                      np.r_[c.astype(np.float64), 0.25])
    np.testing.assert_allclose(got, d, rtol=n * 2.0 ** -52, atol=0)


@pytest.mark.parametrize("kw", [{}, dict(evaluate="wave"), dict(evaluate="jump"),
                                dict(host_loop=True)])
def test_an_exploit_over_a_rejected_policy_reports_it(kw):
    n = 60
    u, v, c, par, loop = _path(n, np.float32)
    with P.Graph(n - 1, n, 0, np.float32) as G:
        G.insert_batch(n - 1, u, v, c)
        G.set_policy(par)
        G.exploit()
        want = G.get_costs()
        assert _status(G.set_policy, loop) == P.PIRRT_ERR_BAD_TREE
        for _ in range(2):
            assert _status(G.exploit, **kw) == P.PIRRT_ERR_BAD_TREE
        G.set_policy(par)
        assert G.exploit(**kw)["converged"] == 1
        np.testing.assert_array_equal(G.get_costs(), want)
