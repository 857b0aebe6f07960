"""L_TV and Adam in bricks at the grid's boundary and where the trainable set
is wider than T: the smallest grid (every brick both first and last), M1 > M2,
and dense grids.  The gradient against the oracle, the many-cloud sweep against
gp_step, and the fused update leaving every slot it does not train as it was,
padding slots (coordinates beyond R) among them."""
import numpy as np
import pytest

from oracle import gridpull as o

from gpu_common import build_lib, export_band, have_gpu
from test_gpu_parity import _band, _check_step, _set_field

pytestmark = pytest.mark.gpu

W = (1.0, 1.0, 0.005)
BANDS = [(8, -1, -1), (8, 2, 0), (16, 4, 1), (16, -1, -1), (32, 2, -1), (64, -1, 2)]


def _setup(R, M1, M2, det, knn_k=0):
    if not have_gpu():
        pytest.skip("no CUDA device")
    build_lib()
    from paper_2308_13175_gb300 import binding as gb
    rng = np.random.default_rng(R + 10 * M1 + 100 * M2 + 200)
    pts = rng.uniform(-0.99, 0.99, (60, 3)).astype(np.float32)
    j = rng.integers(0, len(pts), 4000)
    q = (pts[j] + rng.normal(0, 0.5 / R, (len(j), 3))).astype(np.float32)
    band = _band(gb, gb.gp_create(0), pts, R, M1, M2, knn_k=knn_k, deterministic=det)
    return gb, band, o.band_sets(pts, R, M1, M2), q, pts[j]


@pytest.mark.parametrize("R,M1,M2", BANDS)
@pytest.mark.parametrize("det", [False, True])
def test_step_matches_the_oracle(R, M1, M2, det):
    gb, band, sets, q, s = _setup(R, M1, M2, det)
    D, _ = _set_field(gb, band, sets, R, 0.5, 0.05, seed=7)
    _check_step(gb, band, R, sets, q, s, W, D, flags=gb.GP_STEP_DETERMINISTIC if det else 0)


@pytest.mark.parametrize("R,M1,M2", BANDS)
@pytest.mark.parametrize("flag", ["", "GP_STEP_DETERMINISTIC", "GP_STEP_NO_TV"])
def test_fused_update_leaves_the_rest_as_it_was(R, M1, M2, flag):
    import torch
    gb, band, sets, q, s = _setup(R, M1, M2, flag == "GP_STEP_DETERMINISTIC")
    _, vals = _set_field(gb, band, sets, R, 0.5, 0.05, seed=7)
    _, _, fl, exists = export_band(band)
    vals[~exists] = np.random.default_rng(1).normal(0, 1, int((~exists).sum()))  # the padding slots' own values
    gb.gp_band_set_values(band, torch.from_numpy(vals).cuda())
    rec = torch.from_numpy(np.concatenate([q, s], 1)).cuda()
    loss = torch.zeros(8, dtype=torch.float32, device="cuda")
    for t in range(3):  # both value buffers come into use
        gb.gp_step_update(band, rec, len(q), loss, 1e-3, t + 1, W, flags=getattr(gb, flag) if flag else 0)
        got, m, v = [x.cpu().numpy() for x in gb.gp_band_values(band)]
        kept = (fl & 2) == 0
        assert np.array_equal(got[kept].view(np.int32), vals[kept].view(np.int32)), f"step {t}"
        assert np.all(m[kept] == 0) and np.all(v[kept] == 0)
        assert np.count_nonzero(got != vals) > 0


@pytest.mark.parametrize("R,M1,M2", BANDS)
@pytest.mark.parametrize("det", [False, True])
def test_many_cloud_sweep_equals_gp_step(R, M1, M2, det):
    """One multi step's gradient against gp_step on the multi's own records:
    the same record and stencil code, float sums in another order."""
    import torch
    gb, band, sets, _, _ = _setup(R, M1, M2, False, knn_k=4)
    _, vals = _set_field(gb, band, sets, R, 0.5, 0.05, seed=7)
    m = gb.gp_multi_create(band.ctx, [band], [600], [600], seed=5, deterministic=det)
    loss = torch.zeros(8, dtype=torch.float32, device="cuda")
    gb.gp_multi_step(m, loss, W, lr=0.0)
    rec, _, grad = gb.gp_multi_buffers(m, 0)
    want = torch.empty(band.V_stored, dtype=torch.float32, device="cuda")
    loss1 = torch.zeros(8, dtype=torch.float32, device="cuda")
    gb.gp_step(band, rec, 600, want, loss1, W, d=torch.from_numpy(vals).cuda())
    g, w = grad.cpu().numpy(), want.cpu().numpy()
    assert float(loss1[gb.GP_LOSS_BV]) == float(loss[gb.GP_LOSS_BV])
    assert np.max(np.abs(g - w)) <= 1e-5 * np.max(np.abs(w))
    assert np.all(g[~export_band(band)[3]] == 0.0)
    m.close()
