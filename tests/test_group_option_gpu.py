"""opts.group selects the lanes per vertex: the default count runs as the one-launch
loop, any other as the kernels of that count (more launches), for both cost types and
with the same costs."""
import numpy as np
import pytest

import oracle as O
import paper_2003_04920_gb300 as P
from paper_2003_04920_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P.load_library()


@pytest.mark.parametrize("dtype,default", [(np.float32, 4), (np.float64, 8)])
@pytest.mark.parametrize("group", [0, 4, 8, 16, 32])
def test_group_selects_its_form(dtype, default, group):
    rm = W.random_graph(21, 700, 4000, connected=True)
    c = (np.round(rm.cost * 1024) / 1024 + 1 / 1024).astype(dtype)  # sums are exact
    with P.Graph(rm.n, rm.m, 0, dtype) as G:
        G.insert_batch(rm.n, rm.u, rm.v, c)
        G.set_profiling(2)
        st = G.exploit(group=group)
        launches = G.get_profile()["launches"]
        got = G.get_costs()
    if group in (0, default):
        assert launches == 1
    else:
        assert launches > st["iterations"]
    d, _ = O.dijkstra(rm.n, rm.u, rm.v, c.astype(np.float64))
    np.testing.assert_array_equal(got, d)
