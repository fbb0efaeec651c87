"""get_costs into device buffers at any address: costs are 8 bytes, the buffer need
not be aligned to them, and nothing beside it is written."""
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


@pytest.mark.parametrize("offset", [0, 1, 4, 8, 12])
def test_costs_at_any_address(offset):
    import torch
    rm = W.random_graph(5, 333, 1500, connected=True)
    lib = P.load_library()
    with P.Graph(rm.n, rm.m, 0, np.float32) as G, P.Batch([rm.n], [rm.m]) as B:
        G.insert_batch(rm.n, rm.u, rm.v, rm.cost.astype(np.float32))
        B.insert(0, rm.u, rm.v, rm.cost.astype(np.float32))
        G.exploit()
        B.exploit()
        want = G.get_costs()
        for read in (lambda p: lib.pirrt_graph_get_costs(G._h, p, rm.n, 1),
                     lambda p: lib.pirrt_batch_get_costs(B._h, 0, p, rm.n, 1)):
            buf = torch.full((8 * rm.n + 32,), 0xA5, dtype=torch.uint8, device="cuda")
            assert read(buf.data_ptr() + offset) == P.PIRRT_OK
            got = buf.cpu().numpy()
            end = offset + 8 * rm.n
            np.testing.assert_array_equal(got[offset:end].copy().view(np.float64), want)
            assert (got[:offset] == 0xA5).all() and (got[end:] == 0xA5).all()
