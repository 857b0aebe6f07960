"""Clouds where nearly every query has several nearest points within the float32
margin: each is ranked by its float64 distance and index over all the cells its
ball meets, against brute force."""
import numpy as np
import pytest

from oracle import gridpull as o
from paper_2308_13175_gb300 import synth

from gpu_common import build_lib, have_gpu
from test_gpu_parity import _nn_gpu

pytestmark = pytest.mark.gpu


def _lattice(n, step):
    return (np.stack(np.meshgrid(*[np.arange(n) - n // 2] * 3, indexing="ij"), -1).reshape(-1, 3) * step).astype(np.float32)


def _case(name):
    rng = np.random.default_rng(11)
    if name == "lattice":           # exact 8-way ties, the points in any order
        pts = _lattice(12, 0.125)
        return pts[rng.permutation(len(pts))], pts + np.float32(0.0625)
    if name == "inexact lattice":   # the same within rounding
        pts = _lattice(13, 0.1)
        return pts, pts[rng.permutation(len(pts))] + np.float32(0.05)
    if name == "plane":             # 4-way ties, the lattice filling the domain and beyond
        pts = _lattice(33, 1.0 / 16) * np.float32([1, 1, 0]) * np.float32(1.2)
        pts = np.unique(pts, axis=0)
        return pts, pts + np.float32([0.0375, 0.0375, 0.02])
    if name == "repeated":          # every point 30 times
        pts = np.repeat(synth.sphere_cloud(200, 0.5, seed=4), 30, axis=0)
        return pts[rng.permutation(len(pts))], (pts[::7] + rng.normal(0, 0.02, pts[::7].shape)).astype(np.float32)
    if name == "one point":
        return np.tile(np.float32([[0.1, -0.2, 0.3]]), (700, 1)), rng.uniform(-2, 2, (300, 3)).astype(np.float32)
    pts = synth.sphere_cloud(3000, 0.5, seed=5)
    if name == "centre":            # all points nearly as far
        return pts, rng.normal(0, 1e-7, (200, 3)).astype(np.float32)
    far = rng.normal(0, 1, (200, 3))
    return pts, (far / np.linalg.norm(far, axis=1, keepdims=True) * rng.choice([50.0, 1e6], (200, 1))).astype(np.float32)


@pytest.mark.parametrize("name", ["lattice", "inexact lattice", "plane", "repeated", "one point", "centre", "far"])
@pytest.mark.parametrize("nn_grid", [0, 4, 67])
def test_ties_match_brute_force(name, nn_grid):
    if not have_gpu():
        pytest.skip("no CUDA device")
    build_lib()
    import torch
    from paper_2308_13175_gb300 import binding as gb
    pts, q = _case(name)
    band = gb.gp_build_band(gb.gp_create(0), torch.from_numpy(np.ascontiguousarray(pts)).cuda(), 32, 0, 0, 0, nn_grid)
    want = o.nearest_point(q, pts)
    for hint in (None, want, np.random.default_rng(0).integers(0, len(pts), len(q))):
        nn, rec = _nn_gpu(gb, band, q, hint)
        assert np.array_equal(nn, want)
        assert np.array_equal(rec[:, 3:], pts[want])
