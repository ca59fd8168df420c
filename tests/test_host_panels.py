"""The size rules of the eliminations by panels (csrc/panel.h), on the CPU: a panel
is as wide as its rows in shared memory allow, and no panel where one column does
not fit, so that the eliminations go by columns there instead of failing."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2605_19254_gb300", "csrc")
BLOCK = 227 * 1024  # shared memory of a block


@pytest.fixture(scope="module")
def widths(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if cxx is None or not os.path.exists(nvcc):
        pytest.skip("no C++ compiler or CUDA headers")
    exe = str(tmp_path_factory.mktemp("panels") / "panel_harness")
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, "-I", os.path.join(os.path.dirname(nvcc), "..", "include"),
                    os.path.join(HERE, "panel_harness.cpp"), "-o", exe], check=True, capture_output=True, text=True)

    def run(queries):
        r = subprocess.run([exe], input="".join("%d %d %d\n" % q for q in queries), capture_output=True, text=True,
                           check=True)
        return [tuple(int(v) for v in line.split()) for line in r.stdout.splitlines()]

    return run


def test_panels_fit(widths):
    sizes = sorted({n for k in range(4, 19) for n in (2 ** k - 1, 2 ** k, 2 ** k + 1, 3 << (k - 1))})
    queries = [(n, L, most) for n in sizes for L, most in ((1, 32), (2, 32), (4, 32), (1, 128))]
    for (n, L, most), (w, smem, wider, limit, stride) in zip(queries, widths(queries)):
        # the kernel's static arrays: rows of -B^-1, two batches of multipliers, lists
        static = 4 * (16 + 64) * L * 20 + 4 * (2 * L * 32 + 2 * L + 2 * 16 + 32 + 16 + 16 + 32 + 16 + 16 + 1 + 17 + 2)
        assert 0 <= w <= most and smem <= limit and limit + static + 64 <= BLOCK
        assert stride >= (w or 1) * L and stride % 8 == 4
        assert w == most or wider > limit  # as wide as fits; 0 only where one column does not
    # a matrix that 288 GB hold has a panel (a lane's words and A's, 12 bytes an entry)
    assert all(w > 0 for w, *_ in widths([(n, 1, 32) for n in (85_000, 86_000, 120_000, 140_000)]))
    assert widths([(300_000, 1, 32), (300_000, 4, 32)])[0][0] == 0


def test_widths_at_the_steps(widths):
    # four moduli: the sizes where the panel becomes narrower
    got = [w for w, *_ in widths([(n, 4, 32) for n in (5344, 5345, 10704, 10705, 20144, 20145)])]
    assert got == [32, 16, 16, 8, 8, 4]
