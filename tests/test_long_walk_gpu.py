"""A thin subtree that one CTA walks alone, with no level limit, while the others wait
at the barrier: the wait is bounded, but the bound is far beyond two million tree
levels (some seconds)."""
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


def test_two_million_levels():
    n = 2_000_001
    u = np.arange(n - 1, dtype=np.int32)
    c = np.random.default_rng(0).integers(512, 1024, n - 1) / 1024.0  # sums are exact
    with P.Graph(n, n, 0, np.float32) as G:
        G.insert_batch(n, u, u + 1, c.astype(np.float32))
        G.set_policy(np.r_[np.int32(-1), u].astype(np.int32))
        assert G.exploit(evaluate="wave")["switches"] == 0
        c[0] = 0.25
        G.insert_batch(0, u[:1], u[:1] + 1, c[:1].astype(np.float32))
        st = G.exploit(evaluate="wave", wave_tail=64, dense_fraction=1.0)
        got = G.get_costs()
    print("ms_exploit", st["ms_exploit"])
    assert st["jump_evaluates"] == 0 and st["wave_levels"] < n
    np.testing.assert_array_equal(got, np.cumsum(np.r_[0.0, c]))
