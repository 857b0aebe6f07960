"""Band sets where the bit rows of gp_build_band have edges: grids narrower than
a word of 32 cells, of exactly one word and of several, widths of 0, over 31 and
over the whole grid, and each pairing of a wide, a narrow and an all-cells band.
Sets, counts and stored bricks equal the oracle's."""
import numpy as np
import pytest

from oracle import gridpull as o

from gpu_common import build_lib, export_band, have_gpu, vertex_keys

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M1,M2", [(0, 0), (1, 4), (4, 1), (-1, 2), (2, -1), (-1, -1), (33, 40), (300, 1)])
@pytest.mark.parametrize("R", [8, 16, 32, 64, 128])
def test_band_sets_match_oracle(R, M1, M2):
    if not have_gpu():
        pytest.skip("no CUDA device")
    import torch
    build_lib()
    from paper_2308_13175_gb300 import binding as gb
    h = 2.0 / R
    pts = np.array([[-1, -1, -1], [1, 1, 1], [0, 0, 0], [1 - h, -1 + h, 0.25], [2.0, -3.0, 0.4],
                    [-0.5 + h / 2, 0.3, 0.9]], np.float32)
    if R == 128:
        pts = pts[2:4]                       # keeps the wide bands off parts of the grid
    ctx = gb.gp_create(0)
    band = gb.gp_build_band(ctx, torch.from_numpy(pts).cuda(), R, M1, M2, 0)
    ijk, _, fl, exists = export_band(band)
    keys = vertex_keys(ijk, R)
    sets = o.band_sets(pts, R, M1, M2)
    for bit, name in ((1, "tv"), (2, "trainable")):
        assert np.array_equal(np.sort(keys[exists & ((fl & bit) != 0)]), sets[name]), name
    pull = ijk[(fl & 8) != 0]
    assert np.array_equal(np.sort(pull[:, 0] + R * (pull[:, 1] + R * pull[:, 2])), sets["pull_cells"])
    need = o.key_to_vertex(sets["required"], R) // 8
    nb = R // 8 + 1
    want = np.unique(need[:, 0] + nb * (need[:, 1] + nb * need[:, 2]))
    have = ijk[::512] // 8
    assert np.array_equal(np.sort(have[:, 0] + nb * (have[:, 1] + nb * have[:, 2])), want)
    info = band.info
    assert info["V_tv"] == len(sets["tv"]) and info["V_trainable"] == len(sets["trainable"])
    assert info["n_pull_cells"] == len(sets["pull_cells"])
    assert info["n_occupied_cells"] == len(o.occupied_cells(pts, R))
    band.close()
