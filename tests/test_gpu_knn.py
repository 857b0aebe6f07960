"""sigma_j where the gathering of neighbours has edges: as many neighbours as
points, clouds around a chunk of four, hundreds of equal distances,
isolated points, small and the largest k."""
import numpy as np
import pytest

from oracle import gridpull as o

from gpu_common import build_lib, have_gpu

pytestmark = pytest.mark.gpu


def _cloud(kind):
    rng = np.random.default_rng(3)
    if kind == "two":
        p = np.array([[0.1, 0.2, 0.3], [0.4, -0.2, 0.3]])
    elif kind == "five":
        p = rng.uniform(-1, 1, (5, 3))
    elif kind == "repeated":  # 900 points in one place, a few around it
        p = np.concatenate([np.tile([[0.25, 0.25, 0.25]], (900, 1)), rng.uniform(0.2, 0.3, (40, 3))])
    elif kind == "lattice":   # shells of equal distances
        g = np.linspace(-0.5, 0.5, 11)
        p = np.stack(np.meshgrid(g, g, g), -1).reshape(-1, 3)
    elif kind == "isolated":
        p = np.concatenate([rng.normal(scale=0.01, size=(600, 3)), [[0.9, 0.9, 0.9], [-0.95, 0.9, -0.9]]])
    else:                     # "dense": over 500 points to a cell
        p = rng.normal(scale=0.02, size=(4000, 3))
    return p.astype(np.float32)


@pytest.mark.parametrize("nn_grid", [0, 1, 4, 40])
@pytest.mark.parametrize("kind", ["two", "five", "repeated", "lattice", "isolated", "dense"])
def test_sigma_matches_brute_force(kind, nn_grid):
    if not have_gpu():
        pytest.skip("no CUDA device")
    import torch
    build_lib()
    from paper_2308_13175_gb300 import binding as gb
    ctx = gb.gp_create(0)
    pts = _cloud(kind)
    for k in (1, 4, 50, 64):
        band = gb.gp_build_band(ctx, torch.from_numpy(pts).cuda(), 32, 1, 1, k, nn_grid=nn_grid)
        got = gb.gp_band_sigma(band).cpu().numpy()
        # float32 distances: a few units in the last place
        assert np.allclose(got, o.knn_sigma(pts, min(k, len(pts) - 1)), rtol=1e-6, atol=0), (kind, nn_grid, k)
        band.close()
