"""An insertion whose barrier timed out leaves rows that may name entries never
written: every call that follows rows says so, and a reset or a load ends it."""
import numpy as np
import pytest

import paper_2003_04920_gb300 as P
from paper_2003_04920_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P.load_library()


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_every_call_that_follows_rows_reports_it(dtype, tmp_path):
    rm = W.random_graph(3, 600, 3000, connected=True)
    c = rm.cost.astype(dtype)
    path = str(tmp_path / "graph")
    with P.Graph(rm.n, rm.m + 1, 0, dtype) as G:
        def fill():
            G.insert_batch(rm.n, rm.u, rm.v, c)
            G.exploit()

        fill()
        g, p = G.get_costs(), G.get_parents()
        G.save(path)
        saved = open(path, "rb").read()
        for restore in (lambda: (G.reset(), fill()), lambda: (G.load(path), G.exploit())):
            for call in (G.exploit, lambda: G.exploit(host_loop=True),
                         lambda: G.exploit(evaluate="async"), lambda: G.exploit(tile=2),
                         lambda: G.set_policy(p), G.get_adjacency, lambda: G.save(path),
                         lambda: G.insert_batch(0, rm.u[:1], rm.v[:1], c[:1])):
                G.selftest_insert_timeout()
                with pytest.raises(P.PirrtError) as e:
                    call()
                assert e.value.status == P.PIRRT_ERR_DEVICE_TIMEOUT
            assert open(path, "rb").read() == saved
            restore()
            np.testing.assert_array_equal(G.get_costs(), g)
            np.testing.assert_array_equal(G.get_parents(), p)
            G.get_adjacency()
