"""Device memory of the library on a GPU, seen from the driver's own count of
free bytes; in a process of its own, where no other context keeps the pool."""
import os
import subprocess
import sys

import pytest

from gpu_common import build_lib, have_gpu

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
KEPT = 256 << 20   # what the pool may keep between calls
SLACK = 32 << 20   # the driver's own granularity

GIVEN_BACK = """
import torch
from paper_2308_13175_gb300 import binding as gb
free = lambda: torch.cuda.mem_get_info(0)[0]
pts = torch.rand(12_000_000, 3, device="cuda") * 1.8 - 0.9
first = gb.gp_build_band(gb.gp_create(0), pts[:1000], 64, 2, 2, 0)  # kernels and their module are loaded
first.close()
first.ctx.close()
torch.cuda.synchronize()
start = free()
ctx = gb.gp_create(0)
band = gb.gp_build_band(ctx, pts, 64, 2, 2, 0)
built = free()
band.close()
closed = free()
ctx.close()
print(start - built, start - closed, start - free())
"""


def test_memory_goes_back_with_the_band_and_the_context():
    if not have_gpu():
        pytest.skip("no CUDA device")
    build_lib()
    out = subprocess.run([sys.executable, "-c", GIVEN_BACK], cwd=ROOT, check=True, capture_output=True, text=True).stdout
    built, closed, gone = (int(x) for x in out.split())
    assert built > 2 * KEPT               # points, seeds and chunks: at least 12 + 16 + 16 bytes a point
    assert closed <= KEPT + SLACK, f"{closed >> 20} MiB still held after the band"
    assert gone <= SLACK, f"{gone >> 20} MiB still held after the last context"


def test_pointers_handed_out_have_an_ipc_handle():
    """The values, both value buffers in turn, the moments and a multi's buffers
    can be opened by another process (the driver's own word for the pointer)."""
    if not have_gpu():
        pytest.skip("no CUDA device")
    build_lib()
    import ctypes
    import torch
    from paper_2308_13175_gb300 import binding as gb
    cuda = ctypes.CDLL("libcuda.so.1")
    band = gb.gp_build_band(gb.gp_create(0), torch.rand(500, 3, device="cuda"), 16, 1, 1, 8)
    multi = gb.gp_multi_create(band.ctx, [band], [1000], [500])
    shown = list(gb.gp_multi_buffers(multi, 0)) + list(gb.gp_band_values(band))
    rec = torch.zeros(6, device="cuda")
    gb.gp_step_update(band, rec, 1, torch.zeros(8, device="cuda"), 0.0, 1)
    shown.append(gb.gp_band_values(band)[0])
    assert shown[-1].data_ptr() != shown[3].data_ptr()
    for t in shown:
        capable = ctypes.c_int(-1)
        attribute = 10  # CU_POINTER_ATTRIBUTE_IS_LEGACY_CUDA_IPC_CAPABLE
        assert cuda.cuPointerGetAttribute(ctypes.byref(capable), attribute, ctypes.c_uint64(t.data_ptr())) == 0
        assert capable.value == 1
    multi.close()
