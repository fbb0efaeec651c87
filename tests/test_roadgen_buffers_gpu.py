"""The edges of a roadmap come in buffers of their own size, through the two-step
calls; the one call with the caller's room still counts, refuses and writes as told."""
import ctypes

import numpy as np
import pytest

from paper_2003_04920_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _inputs(n, k, n_obs):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2003_04920_gb300.workloads import gpu as G
    rng = np.random.default_rng(n + k)
    radius = 2.0 if n_obs == 1 else 0.05  # one ball over the whole box: no edge left
    scene = W.Scene(2, 0.0, 1.0, rng.uniform(0, 1, (n_obs, 2)), np.full(n_obs, radius))
    pts = torch.from_numpy(rng.uniform(0, 1, (n, 2))).cuda()
    return torch, G, scene, pts, G.knn(pts, 0.0, 1.0, k)


@pytest.mark.parametrize("n,k,n_obs", [(200, 5, 8), (3000, 33, 60), (50, 4, 1)])
@pytest.mark.parametrize("f64", [False, True])
def test_buffers_hold_the_edges_and_nothing_else(n, k, n_obs, f64):
    torch, G, scene, pts, nbr = _inputs(n, k, n_obs)
    dt = np.float64 if f64 else np.float32
    u, v, c, start = G.edges(pts, nbr, scene, True, 16, dt)
    m = int(start[-1])
    assert (m == 0) == (n_obs == 1)
    for t, size in ((u, 4), (v, 4), (c, 8 if f64 else 4)):
        assert t.numel() == m and t.untyped_storage().nbytes() == size * m

    lib = G.load()
    cen, rad = G._scene_dev(scene)
    args = (2, n, pts.data_ptr(), k, nbr.data_ptr(), n_obs, cen.data_ptr(), rad.data_ptr(), 0, 16)
    off = torch.empty(n + 1, dtype=torch.int64, device="cuda")
    cnt = ctypes.c_int64(0)
    cu, cv = torch.full((2, m + 1), -7, dtype=torch.int32, device="cuda")
    cc = torch.full((m + 1,), -7, dtype=c.dtype, device="cuda")
    one = lambda cap, *out: lib.rgg_edges(*args, int(f64), *out, off.data_ptr(), cap,
                                          ctypes.byref(cnt), G._stream())
    if m:
        assert one(m - 1, cu.data_ptr(), cv.data_ptr(), cc.data_ptr()) == 3 and cnt.value == m
        assert one(0, None, None, None) == 3 and cnt.value == m
        assert one(m, None, None, None) == 1
    assert one(m + 1, cu.data_ptr(), cv.data_ptr(), cc.data_ptr()) == 0 and cnt.value == m
    for got, want in ((cu, u), (cv, v), (cc, c)):
        assert torch.equal(got[:m], want) and int(got[m]) == -7

    # the second step writes once
    h = ctypes.c_void_p()
    assert lib.rgg_links_mark(*args, off.data_ptr(), ctypes.byref(cnt), G._stream(),
                              ctypes.byref(h)) == 0
    fill = lambda: lib.rgg_links_fill(h, int(f64), cu.data_ptr(), cv.data_ptr(), cc.data_ptr(),
                                      G._stream())
    assert fill() == 0 and fill() == 1
    lib.rgg_links_destroy(h)
    assert lib.rgg_links_mark(*args[:3], 0, *args[4:], off.data_ptr(), ctypes.byref(cnt),
                              G._stream(), ctypes.byref(h)) == 1 and not h.value
