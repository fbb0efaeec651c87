"""The searching autotuner's first trial is what an exploit does by default: the
options it starts from are the defaults of the form they select, written out."""
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


@pytest.mark.parametrize("dtype,start,want", [
    (np.float32, None, dict(group=4, wave_tail=-1, wave_local_max=32, wave_local_step=512)),
    (np.float64, None, dict(group=8, wave_tail=-1, wave_local_max=32, wave_local_step=512)),
    (np.float32, dict(tile=2), dict(group=4, wave_tail=64, wave_local_max=128,
                                    wave_local_step=4096)),
    (np.float64, dict(group=16), dict(group=16, wave_tail=64, wave_local_max=128,
                                      wave_local_step=4096)),
])
def test_the_search_starts_from_the_defaults(dtype, start, want):
    rm = W.random_graph(2, 500, 2500, connected=True)
    with P.Batch([rm.n], [rm.m], cost_dtype=dtype) as B:
        B.insert(0, rm.u, rm.v, rm.cost.astype(dtype))
        best, ms, trials = B.autotune_search(max_trials=1, start=start)
    assert trials == 1 and ms > 0
    assert {k: best[k] for k in want} == want
