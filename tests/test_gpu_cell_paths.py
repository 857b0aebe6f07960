"""The step's corner reads and corner sums where a cell's corners can lie: a
record's q and its s in every cell of a grid (each x mod 8, so every width of
the reads and sums, and each way of crossing brick faces), against the oracle."""
import numpy as np
import pytest

from oracle import gridpull as o

from gpu_common import build_lib, have_gpu
from test_gpu_parity import _band, _check_step, _set_field

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 4095, 4096 * 3])
@pytest.mark.parametrize("R,bands", [(16, (-1, -1)), (16, (2, 2)), (32, (-1, -1))])
@pytest.mark.parametrize("det", [False, True])
def test_step_in_every_cell(n, R, bands, det):
    if not have_gpu():
        pytest.skip("no CUDA device")
    build_lib()
    from paper_2308_13175_gb300 import binding as gb
    rng = np.random.default_rng(R + n)
    pts = rng.uniform(-0.99, 0.99, (60, 3)).astype(np.float32)
    band = _band(gb, gb.gp_create(0), pts, R, *bands, knn_k=0, deterministic=det)
    sets = o.band_sets(pts, R, *bands)
    cells = np.stack(np.meshgrid(*[np.arange(R)] * 3, indexing="ij"), -1).reshape(-1, 3)

    def somewhere():
        c = cells[rng.permutation(len(cells))]
        c = np.concatenate([c] * (n // len(c) + 1))[:n]
        return (-1 + 2 / R * (c + rng.uniform(0.05, 0.95, c.shape))).astype(np.float32)

    q, s = somewhere(), somewhere()
    D, _ = _set_field(gb, band, sets, R, 0.5, 0.05, seed=7)
    _check_step(gb, band, R, sets, q, s, (1.0, 1.0, 0.005), D, flags=gb.GP_STEP_DETERMINISTIC if det else 0)
    gb.gp_band_check(band)
