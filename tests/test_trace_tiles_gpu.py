"""The tile trace of the top-down Evaluate (pirrt_profile's share_* and local_*): both
ways of profiling keep all three of count, vertices and cycles, bucket by bucket."""
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


@pytest.mark.parametrize("mode", [True, 2])
def test_tiles_are_counted_and_timed(mode):
    rm = W.roadmap_c3(n=40_000, block=5_000)
    with P.Graph(rm.n, rm.m, 0, np.float32) as G:
        G.set_profiling(mode)
        for v0, v1, e0, e1 in rm.blocks():
            G.insert_batch(v1 - v0, rm.u[e0:e1], rm.v[e0:e1], rm.cost[e0:e1])
            G.exploit(evaluate="wave")
        prof = G.get_profile()
    for kind in ("share", "local"):
        tiles, vertices, cycles = (prof[f"{kind}_{x}"] for x in ("tiles", "vertices", "cycles"))
        assert sum(tiles) > 0
        for b, (n, items, cyc) in enumerate(zip(tiles, vertices, cycles)):
            assert (n > 0) == (items > 0) == (cyc > 0)
            if n and b < 23:
                assert n * (1 << (b - 1)) <= items <= n * ((1 << b) - 1)
                assert b <= 10  # a tile holds at most 512 vertices
    assert sum(prof["share_vertices"]) <= sum(prof["level_vertices"])
