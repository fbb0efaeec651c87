"""The GPU roadmap generator's neighbour search and edges against the CPU
reference, bit for bit, in every dimension it serves and where its warps' chunks
end: k around 32 and at 128, barely more points than k, equal points and equal
distances, obstacles around 32, points on a coarse lattice (distances tie)."""
import math

import numpy as np
import pytest

from paper_2003_04920_gb300 import workloads as W
from tests import test_roadgen_gpu as R

pytestmark = pytest.mark.gpu


def _scene(rng, dim, n_obs):
    lo, hi = (0.0, 1.0) if dim == 2 else (-math.pi, math.pi)
    side = hi - lo
    return W.Scene(dim, lo, hi, rng.uniform(lo, hi, (n_obs, dim)),
                   rng.uniform(0.02, 0.12, n_obs) * side)


@pytest.mark.parametrize("dim,n,k,n_obs,lattice", [
    (1, 150, 5, 3, 0), (2, 300, 1, 0, 0), (2, 300, 31, 31, 0), (2, 300, 32, 32, 0),
    (2, 400, 33, 33, 16), (2, 140, 128, 70, 0), (3, 200, 20, 12, 6), (4, 129, 128, 5, 0),
    (5, 200, 30, 20, 0), (6, 260, 30, 64, 0), (7, 200, 37, 40, 3), (8, 150, 12, 9, 0)])
@pytest.mark.parametrize("f64", [False, True])
def test_neighbours_and_edges_equal_reference(dim, n, k, n_obs, lattice, f64):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2003_04920_gb300.workloads import gpu as G
    G.load()
    rng = np.random.default_rng(dim * 1000 + n + k)
    scene = _scene(rng, dim, n_obs)
    pts = rng.uniform(scene.lo, scene.hi, (n, dim))
    if lattice:
        pts = scene.lo + np.floor((pts - scene.lo) / (scene.hi - scene.lo) * lattice) * \
            ((scene.hi - scene.lo) / lattice)
    pts[n // 2] = pts[3]  # an equal pair: a link of length 0, no edge
    dev = torch.from_numpy(pts).cuda()
    nbr = G.knn(dev, scene.lo, scene.hi, k)
    want = R.knn_np(pts, k)
    np.testing.assert_array_equal(nbr.cpu().numpy(), want)
    dt = np.float64 if f64 else np.float32
    for exact in (True, False):
        u, v, c, start = G.edges(dev, nbr, scene, exact, 16, dt)
        ru, rv, rc, rs = R.edges_np(pts, want, scene, exact, 16, dt)
        np.testing.assert_array_equal(start, rs)
        np.testing.assert_array_equal(u.cpu().numpy(), ru)
        np.testing.assert_array_equal(v.cpu().numpy(), rv)
        np.testing.assert_array_equal(c.cpu().numpy(), rc)
