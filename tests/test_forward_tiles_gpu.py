"""The fused forward pass where its tiles end (128 rows, one to four tiles per CTA
of 152): against the oracle on dyadic inputs (whose layer sums are exact in FP32,
so that rounding cancellations cannot enter) with the bounds derived in
test_mlp_gpu, and the same rows in another order -- a row's arithmetic does not
depend on the tile, the lane or the neighbours it lands on, so its result is the
same bit for bit."""
import numpy as np
import pytest

import paper_2003_04920_gb300 as P
from oracle import mlp as M
from tests import test_mlp_gpu as T

pytestmark = pytest.mark.gpu
torch = T.torch


@pytest.mark.parametrize("rows", [31, 127, 129, 152 * 128 - 1, 152 * 128, 152 * 128 + 1,
                                  152 * 128 * 3 + 65])
def test_tile_edges(torch, rows):
    S = 6
    params, grids, scene, z, target = T._dyadic(seed=rows, S=S, R=rows)
    prop = P.Proposal(S, rows, seed=3)
    gd, sd, zd, _ = T._upload(torch, prop, params, grids, scene, z, target)
    y = prop.forward(gd, sd, zd).cpu().numpy().astype(np.float64)
    f = M.forward(params, grids, scene, z.astype(np.float64), rounded=True)
    atol = 0.25 * T.ACC * (f["h2"] @ np.abs(params["W3"]).T) + 2.0 ** -21
    assert not (np.abs(y - f["y"]) > 1e-5 * np.abs(f["y"]) + atol).any()
    prop.close()


@pytest.mark.parametrize("S,rows", [(1, 300), (40, 129), (40, 152 * 128 + 513)])
def test_rows_do_not_depend_on_their_place(torch, S, rows):
    rng = np.random.default_rng(S + rows)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    grids = dev((rng.random((S, M.GRID)) < 0.25).astype(np.float32))
    scene = rng.integers(0, S, rows).astype(np.int32)
    z = rng.normal(size=(rows, M.NOISE)).astype(np.float32)
    prop = P.Proposal(S, rows, seed=5)
    y = prop.forward(grids, dev(scene), dev(z)).cpu().numpy()
    order = rng.permutation(rows)
    got = prop.forward(grids, dev(scene[order]), dev(z[order])).cpu().numpy()
    np.testing.assert_array_equal(got, y[order])
    prop.close()
