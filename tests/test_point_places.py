"""Where the point list puts a point's parts (nn_place in gp_nn_device.cuh),
compiled for the host from the same source: chunk first + at // 4 is 16 floats,
its parts of four rotated by half the chunk's number, at any chunk a cloud of
fewer than 2^31 points can reach - from 2^29 chunks on a place counted from the
start of the cloud no longer fits 31 bits."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "tests", "native", "nn_place_host.cu")
# Chunks of J < 2^31 points in at most 1024^3 cells, each filled up to four.
MOST = (2 ** 31 - 1 + 3 * 2 ** 30) // 4


@pytest.fixture(scope="module")
def places(tmp_path_factory):
    nvcc = next((c for c in ("/usr/local/cuda/bin/nvcc", shutil.which("nvcc")) if c and os.path.exists(c)), None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    exe = str(tmp_path_factory.mktemp("place") / "nn_place_host")
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2308_13175_gb300", "csrc"), SRC, "-o", exe],
                   check=True, capture_output=True)

    def run(cases):
        text = "\n".join(" ".join(str(int(v)) for v in c) for c in cases) + "\n"
        return [int(x) for x in subprocess.run([exe], input=text, capture_output=True, text=True,
                                               check=True).stdout.split()]
    return run


@pytest.mark.parametrize("first", [0, 3, 2 ** 29 - 1, 2 ** 29, 2 ** 29 + 12345, 2 ** 30 + 7, MOST - 5])
def test_places(places, first):
    rng = np.random.default_rng(first % 1000)
    # A block's places: its first ones, and those of a block that holds all of J = 2^31 - 1 points.
    ats = list(range(20)) + [int(a) for a in rng.integers(0, 2 ** 31 + 4 * 64, 50)] if first < 2 ** 29 else list(range(20))
    cases = [(first, at, k) for at in ats for k in range(4)]
    want = [16 * (first + at // 4) + 4 * ((k + (first + at // 4) // 2) % 4) + at % 4 for _, at, k in cases]
    got = places(cases)
    assert got == want
    assert min(got) >= 0 and len(set(got)) == len(set(cases))
