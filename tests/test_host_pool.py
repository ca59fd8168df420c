"""A context's memory pool on the CPU, against a fake of the CUDA calls: made once
for all threads, with its threshold; a failed creation is reported as it is and
tried again by the next allocation."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2605_19254_gb300", "csrc")


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if cxx is None or not os.path.exists(nvcc):
        pytest.skip("no C++ compiler or CUDA headers")
    exe = str(tmp_path_factory.mktemp("pool") / "pool_harness")
    subprocess.run([cxx, "-O1", "-std=c++17", "-pthread", "-I", CSRC, "-I",
                    os.path.join(os.path.dirname(nvcc), "..", "include"), os.path.join(HERE, "pool_harness.cpp"), "-o",
                    exe], check=True, capture_output=True, text=True)
    return lambda fails: [int(v) for v in subprocess.run([exe, str(fails)], capture_output=True, text=True,
                                                         check=True).stdout.split()]


@pytest.mark.parametrize("fails", [0, 1, 2])
def test_pool(harness, fails):
    oom = 2  # cudaErrorMemoryAllocation
    first, (bad, made, keep, live) = harness(fails)[:3], harness(fails)[3:]
    assert first == [oom] * fails + [0] * (3 - fails)
    assert (bad, made, keep, live) == (0, 2, 12345, 0)  # one pool for each of the two contexts
