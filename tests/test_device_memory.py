"""The library's host code around device memory and launches, run on a stand-in
for the CUDA runtime (tests/native/fake_cudart.cpp): two devices, kernels that do
nothing, and a record of which stream still had work in flight when memory was
freed and of what the memory pools hold.  No GPU is needed."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NATIVE = os.path.join(ROOT, "tests", "native")


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    nvcc = next((c for c in ("/usr/local/cuda/bin/nvcc", shutil.which("nvcc")) if c and os.path.exists(c)), None)
    if nvcc is None or shutil.which("g++") is None:
        pytest.skip("no CUDA toolkit")
    from paper_2308_13175_gb300 import build
    build.build()
    objs = [os.path.join(build.BUILD, s.replace(".cu", ".o")) for s in build.SOURCES]
    exe = str(tmp_path_factory.mktemp("memory") / "memory_host")
    include = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", include, "-I", os.path.join(ROOT, "include"), "-I", NATIVE,
                    os.path.join(NATIVE, "memory_host.cpp"), os.path.join(NATIVE, "fake_cudart.cpp"), *objs, "-o", exe],
                   check=True, capture_output=True)

    def call(what):
        out = subprocess.run([exe, what], check=True, capture_output=True, text=True).stdout
        assert "error" not in out, out
        return {k: int(v) for k, v in (line.split() for line in out.splitlines())}
    return call


def test_multi_destroyed_while_another_device_is_current(run):
    """Its device is waited for before its memory goes, and the caller's device
    is current again afterwards."""
    got = run("other_device")
    assert got == {"device": 0, "races": 0, "wrong_device": 0}


def test_tuning_on_another_stream_than_the_last_step(run):
    """The tile list that a step still reads is not given back under it."""
    assert run("tiles") == {"device": 0, "races": 0, "wrong_device": 0}


def test_pool_gives_memory_back(run):
    """What a destroyed band leaves beyond the bytes that the pool keeps goes
    back at once, and everything goes with the last context of the device."""
    assert run("given_back") == {"above_while_alive": 1, "above_after_the_band": 0, "after_the_last_context": 0}


def test_pool_without_its_threshold_is_not_kept(run):
    """A context whose pool cannot be set up fails; the next one gets a pool
    that is."""
    assert run("no_threshold") == {"first": 3, "second": 0, "keeps": 1}  # GP_ERR_CUDA, GP_OK


def test_pointers_handed_out_are_ordinary_allocations(run):
    """Callers may open them to other devices and processes, which a pool's
    memory is not.  A block given back serves the next band; none is left after
    the last context, nor after an object that outlived it."""
    assert run("shown") == {"values": 0, "moments": 0, "multi": 0, "kept": 1, "left": 0}


def test_search_runs_the_blocks_that_were_tuned(run):
    """The search's blocks per SM stay what gp_multi_info says and what the
    autotuner timed, whichever tile length the query stage then takes."""
    assert run("tuned") == {"default": 0, "records_per_tile": 512, "tuned": 0}


def test_kept_memory_is_given_up_for_an_allocation(run):
    """On a full device what is kept does not make an allocation fail."""
    assert run("full") == {"band": 1, "multi": 1}
