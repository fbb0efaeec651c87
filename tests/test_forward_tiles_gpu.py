"""The fused forward pass where its tiles end (128 rows, one to four tiles per CTA
of 152), against the layered kernels with the bounds of test_mlp_gpu, and the
same rows in another order: a row's arithmetic does not depend on the tile, the
lane or the neighbours it lands on, so its result is the same bit for bit."""
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
    T.test_fused_forward_matches_layered(torch, rows)


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
