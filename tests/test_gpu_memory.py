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
