"""Hints far from the nearest point: the same answers as without hints, and not
much more work (gp_nn_work's candidate distances), on a surface, in a volume
and on a grid of cells far finer than the points."""
import numpy as np
import pytest

from paper_2308_13175_gb300 import synth

from gpu_common import build_lib, have_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cloud", ["surface", "volume"])
@pytest.mark.parametrize("nn_grid", [0, 512])
@pytest.mark.parametrize("hints", ["random", "near", "one"])
def test_far_hints_cost_little(cloud, nn_grid, hints):
    if not have_gpu():
        pytest.skip("no CUDA device")
    build_lib()
    import torch
    from paper_2308_13175_gb300 import binding as gb
    rng = np.random.default_rng(3)
    pts = synth.object_cloud(30_000, seed=1) if cloud == "surface" else \
        rng.uniform(-0.9, 0.9, (30_000, 3)).astype(np.float32)
    band = gb.gp_build_band(gb.gp_create(0), torch.from_numpy(np.ascontiguousarray(pts)).cuda(), 128, 0, 0, 20, nn_grid)
    j = rng.integers(0, len(pts), 20_001)
    q = torch.from_numpy((pts[j] + rng.normal(0, 0.01, (len(j), 3))).astype(np.float32)).cuda()
    hint = {"random": rng.integers(0, len(pts), len(j)), "near": j, "one": np.full(len(j), 17)}[hints].astype(np.int32)
    plain = torch.empty(len(j), dtype=torch.int32, device="cuda")
    got = torch.empty_like(plain)
    work_plain = gb.gp_nn_work(band, q, plain)
    work = gb.gp_nn_work(band, q, got, hint=torch.from_numpy(hint).cuda())
    assert torch.equal(got, plain)
    # A wrong hint costs its own distance; a right one saves work.
    assert work <= 1.5 * work_plain + len(j), f"{work / len(j):.1f} against {work_plain / len(j):.1f} a query"
