"""gp_nn where its cell list, its block planes and its shared lists have edges:
grids of one cell up to many blocks a side, cloud sizes around a chunk of four
points, batches around a warp and a block, points outside the grid's cube,
flat, clustered and repeated points, with and without normals and hints.  Every
index equals brute force (float64 distances, ties to the lowest index)."""
import numpy as np
import pytest

from oracle import gridpull as o
from paper_2308_13175_gb300 import synth

from gpu_common import build_lib, have_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not have_gpu():
        pytest.skip("no CUDA device")
    build_lib()
    from paper_2308_13175_gb300 import binding as gb
    return gb.gp_create(0)


def _cloud(kind):
    rng = np.random.default_rng(17)
    if kind == "one":
        p = np.array([[0.3, -0.7, 0.1]])
    elif kind == "five":
        p = rng.uniform(-1, 1, (5, 3))
    elif kind == "sphere":
        p = synth.sphere_cloud(3001, 0.7, seed=3)
    elif kind == "plane":   # a face of the cell grid, repeated points
        p = np.stack([rng.uniform(-1, 1, 2000), rng.uniform(-1, 1, 2000), np.full(2000, 0.25)], 1)
        p = np.concatenate([p, p[:500]])
    elif kind == "outside":  # kept in the boundary cells
        p = np.concatenate([rng.uniform(-3, 3, (900, 3)), rng.normal(scale=1e5, size=(50, 3)),
                            synth.sphere_cloud(500, 0.9, seed=4)])
    else:  # "clusters": hundreds of points to a cell, then empty space
        p = np.repeat(rng.uniform(-0.9, 0.9, (7, 3)), 300, axis=0) + rng.normal(scale=2e-3, size=(2100, 3))
    return p.astype(np.float32)


@pytest.mark.parametrize("nn_grid", [0, 1, 3, 4, 5, 17, 130])
@pytest.mark.parametrize("kind", ["one", "five", "sphere", "plane", "outside", "clusters"])
def test_nn_matches_brute_force(ctx, kind, nn_grid):
    import torch
    from paper_2308_13175_gb300 import binding as gb
    pts = _cloud(kind)
    J = len(pts)
    rng = np.random.default_rng(5)
    src = rng.integers(0, J, 700)
    near = pts[src] + rng.normal(scale=0.03, size=(700, 3))
    lattice = rng.integers(-8, 9, (100, 3)) / 8.0          # cell and block faces
    q = np.concatenate([near, lattice, rng.uniform(-6, 6, (80, 3)), pts[rng.integers(0, J, 60)],
                        [[2e9, -1e9, 3.0], [1e17, 0.0, 0.0]]]).astype(np.float32)
    hint = np.concatenate([src, rng.integers(-3, J + 3, len(q) - 700)]).astype(np.int32)
    want = o.nearest_point(q, pts)
    for knn_k in (0, 6) if J > 1 else (0,):
        band = gb.gp_build_band(ctx, torch.from_numpy(pts).cuda(), 32, 1, 1, knn_k, nn_grid=nn_grid)
        qd, hd = torch.from_numpy(q).cuda(), torch.from_numpy(hint).cuda()
        for n in (1, 31, 33, 129, len(q)):
            for h in (hd, None):
                nn = torch.full((n,), -7, dtype=torch.int32, device="cuda")
                rec = torch.empty((n, 6), dtype=torch.float32, device="cuda")
                gb.gp_nn(band, qd[len(q) - n:], nn, rec, hint=None if h is None else h[len(q) - n:])
                got = nn.cpu().numpy()
                assert np.array_equal(got, want[len(q) - n:]), (kind, nn_grid, knn_k, n)
                assert np.array_equal(rec.cpu().numpy(), np.concatenate([q[len(q) - n:], pts[got]], 1))
        work = gb.gp_nn_work(band, qd, nn, hint=hd)
        assert np.array_equal(nn.cpu().numpy(), want) and work >= len(q)
        band.close()
