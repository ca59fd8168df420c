"""The memory that a Smith-form server's idle workers keep, on the CPU: with the
running jobs it stays within the budget, and pools are given back only for that."""
import os
import random
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2605_19254_gb300", "csrc")


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path_factory.mktemp("book") / "book_harness")
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, os.path.join(HERE, "pool_book_harness.cpp"), "-o", exe],
                   check=True, capture_output=True, text=True)

    def _run(workers, budget, ops):
        text = f"{workers} {budget}\n" + "".join(f"{o} {w} {v}\n" for o, w, v in ops)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.splitlines()
        return [([int(t) for t in line.split("|")[0].split()], int(line.split("|")[1])) for line in out]

    return _run


def test_a_job_of_the_whole_budget(run):
    # three workers have each run one job; the fourth takes the whole budget
    ops = [x for w in range(3) for x in (("s", w, 100), ("f", w, 64))] + [("s", 3, 100)]
    assert run(4, 100, ops) == [([], 0), ([0], 0), ([1], 0), ([2], 0)]
    assert run(4, 300, ops) == [([], 0), ([], 64), ([], 128), ([], 192)]
    assert run(4, 200, ops) == [([], 0), ([], 64), ([0], 64), ([1], 64)]  # (equal: the first)


def test_random_jobs(run):
    rng = random.Random(5)
    for _ in range(20):
        workers, budget = rng.randint(1, 8), rng.randint(100, 400)
        ops, jobs, running, starts = [], {}, 0, []
        for _ in range(60):
            w = rng.randrange(workers)
            if w in jobs:
                running -= jobs.pop(w)
                ops.append(("f", w, rng.randint(0, 64)))
            else:
                size = rng.randint(10, 100)
                if running + size <= budget:
                    running += size
                    jobs[w] = size
                    ops.append(("s", w, running))
                    starts.append(running)
        for used, (_, kept) in zip(starts, run(workers, budget, ops)):
            assert used + kept <= budget or kept == 0
