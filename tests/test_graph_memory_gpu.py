"""The device memory of a graph, and the block of it that insertions, every loop form,
set_policy and the read-backs use in turn: one graph goes through all of them,
block after block, and ends with the costs of Dijkstra's."""
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


def test_bytes_per_vertex():
    """FP32 costs: 16 B of row extent, four pool entries of 8 B, a block of 96 B and 80 B
    of arrays that last; 16 allocations rounded up to 2 MB each."""
    import torch
    n = 16_000_000
    P.Graph(16, 16, 0, np.float32).close()  # whatever the first graph loads
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    with P.Graph(n, 1, 0, np.float32):
        used = free - torch.cuda.mem_get_info()[0]
    assert used <= 224 * n + 24 * (2 << 20)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_uses_in_turn(dtype, tmp_path):
    rm = W.random_graph(31, 4000, 30_000, connected=True)
    c = (np.floor(rm.cost * 512) / 512 + 1 / 512).astype(dtype)  # sums are exact
    path = str(tmp_path / "g")
    forms = [{}, dict(host_loop=True), dict(evaluate="async"), dict(evaluate="wave"), dict(tile=2),
             dict(evaluate="jump"), dict(evaluate="jump", host_loop=True), dict(tile=1),
             dict(evaluate="wave", host_loop=True), dict(group=16), dict(tile=3)]
    cuts = np.linspace(0, rm.m, len(forms) + 1).astype(int)
    with P.Graph(rm.n, rm.m, 0, dtype) as G:
        for i, kw in enumerate(forms):
            e0, e1 = cuts[i], cuts[i + 1]
            G.insert_batch(rm.n if i == 0 else 0, rm.u[e0:e1], rm.v[e0:e1], c[e0:e1])
            assert G.exploit(**kw)["converged"] == 1
            g, p = G.get_costs(), G.get_parents()
            d, _ = O.dijkstra(rm.n, rm.u[:e1], rm.v[:e1], c[:e1].astype(np.float64))
            np.testing.assert_array_equal(g, d)
            if i % 3 == 0:
                G.set_policy(p)
            elif i % 3 == 1:
                off, col, w = G.get_adjacency()
                assert off[-1] == 2 * e1 and sorted(w.tolist()) == sorted(np.repeat(c[:e1], 2).tolist())
            else:
                G.save(path)
                G.load(path)
            np.testing.assert_array_equal(G.get_costs(), g)
            np.testing.assert_array_equal(G.get_parents(), p)
