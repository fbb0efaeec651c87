"""The scene features and the backward pass at the sizes where their tiles end:
scenes around 16 and 32 (and a grid array off its 16-byte boundary), rows around
32 and beyond one tile per CTA, against the oracle with the bounds derived in
test_mlp_gpu."""
import numpy as np
import pytest

import paper_2003_04920_gb300 as P
from oracle import mlp as M
from tests import test_mlp_gpu as T

pytestmark = pytest.mark.gpu
torch = T.torch


@pytest.mark.parametrize("S", [1, 15, 16, 17, 32, 33, 70])
@pytest.mark.parametrize("shift", [0, 1])
def test_scene_features_at_tile_edges(torch, S, shift):
    R = 2 * S + 3
    params, grids, scene, z, target = T._dyadic(seed=S, S=S, R=R)
    scene[:S] = np.arange(S)  # every scene at least once
    prop = P.Proposal(S, R, seed=3)
    _, sd, zd, _ = T._upload(torch, prop, params, grids, scene, z, target)
    flat = torch.zeros(S * M.GRID + shift, device="cuda")
    flat[shift:] = torch.from_numpy(grids).cuda().reshape(-1)
    y = prop.forward(flat[shift:].view(S, M.GRID), sd, zd).cpu().numpy().astype(np.float64)
    f = M.forward(params, grids, scene, z.astype(np.float64), rounded=True)
    atol = 0.25 * T.ACC * (f["h2"] @ np.abs(params["W3"]).T) + 2.0 ** -21
    assert not (np.abs(y - f["y"]) > 1e-5 * np.abs(f["y"]) + atol).any()
    prop.close()


@pytest.mark.parametrize("S,R", [(1, 1), (8, 31), (8, 32), (3, 33), (2, 65), (8, 1000)])
def test_backward_at_tile_edges(torch, monkeypatch, S, R):
    whole = T._dyadic
    monkeypatch.setattr(T, "_dyadic", lambda seed: whole(seed, S=S, R=R))
    T.test_backward_matches_oracle_elementwise(torch)


def test_backward_with_several_tiles_per_cta_and_repeats(torch):
    """10,000 rows (three tiles per CTA on 152 SMs) in random scene order: the
    gradient is the same from run to run, and its per-scene part, db1 = the sum of
    the D's before rounding, agrees with the sum over shuffled rows."""
    rng = np.random.default_rng(4)
    S, R = 12, 10_000
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    grids = dev((rng.random((S, M.GRID)) < 0.25).astype(np.float32))
    scene = rng.integers(0, S, R).astype(np.int32)
    z = rng.normal(size=(R, M.NOISE)).astype(np.float32)
    t = rng.random((R, 2)).astype(np.float32)
    prop = P.Proposal(S, R, seed=9)
    got = []
    order = rng.permutation(R)
    for idx in (np.arange(R), np.arange(R), order):
        prop.zero_grads()
        loss = prop.backward(grids, dev(scene[idx]), dev(z[idx]), dev(t[idx]))
        got.append((loss, prop.get_grads().cpu().numpy().astype(np.float64)))
    assert got[0][0] == got[1][0]
    np.testing.assert_array_equal(got[0][1], got[1][1])
    # another order of the rows: FP32 sums of 10,000 terms regrouped, and a BF16
    # step of a per-scene sum here and there (2^-8 of one of 12 scenes)
    assert abs(got[0][0] - got[2][0]) <= 1e-5 * got[0][0]
    a, b = got[0][1], got[2][1]
    assert np.linalg.norm(a - b) <= 2.0 ** -8 * np.linalg.norm(a)
    prop.close()
