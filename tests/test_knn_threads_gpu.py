"""Neighbour search around the sizes from which a thread takes a query (by dimension and
number of neighbours), against brute force over every point for a sample of queries:
uniform points, a lattice (distances tie), and half of the points in a cluster so
tight that its queries go back to a warp."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _brute(torch, pts, k, rows):
    """k nearest by (FP32 squared distance, id), coordinates in order."""
    q, n = pts.float(), pts.shape[0]
    out = []
    for r in rows.split(200):
        d2 = torch.zeros((len(r), n), device="cuda")
        for d in range(pts.shape[1]):
            t = q[r, d, None] - q[None, :, d]
            d2 += t * t
        key = (d2.view(torch.int32).long() << 32) + torch.arange(n, device="cuda")
        key[torch.arange(len(r), device="cuda"), r] = 1 << 62
        out.append(torch.topk(key, k, dim=1, largest=False).values & 0xFFFFFFFF)
    return torch.cat(out).int()


@pytest.mark.parametrize("dim,n,k", [(1, 29_999, 1), (1, 30_000, 1), (2, 30_000, 6), (2, 49_999, 10),
                                     (2, 50_001, 10), (2, 120_000, 24), (2, 120_000, 25),
                                     (3, 80_000, 16), (4, 59_999, 6), (4, 60_000, 6),
                                     (4, 240_000, 24), (5, 60_000, 6)])
@pytest.mark.parametrize("spread", ["uniform", "lattice", "cluster"])
def test_neighbours(dim, n, k, spread):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2003_04920_gb300.workloads import gpu as G
    G.load()
    rng = np.random.default_rng(dim * n + k)
    pts = rng.uniform(0.0, 1.0, (n, dim))
    if spread == "lattice":
        side = max(2, int((n / 3) ** (1 / dim)))  # about three points a site
        pts = np.floor(pts * side) / side
    elif spread == "cluster":
        pts[rng.permutation(n)[:n // 2]] = 0.5 + 1e-4 * rng.normal(size=(n // 2, dim))
    dev = torch.from_numpy(pts).cuda()
    nbr = G.knn(dev, 0.0, 1.0, k)
    rows = torch.from_numpy(np.unique(np.r_[0, n - 1, rng.integers(0, n, 600)])).cuda()
    assert torch.equal(nbr[rows], _brute(torch, dev, k, rows))
    assert int(nbr.min()) >= 0 and int(nbr.max()) < n  # enough points: every row is full
