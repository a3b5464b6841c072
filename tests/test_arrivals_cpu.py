"""How many events are taken to run side by side (csrc/dgs_arrivals.h), for the patterns of arrivals that callers have."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "dgs_arrivals.h"
// argv: workers, then a worker's number for an arrival or -1 for a join; prints abreast() * 10 + lone() after each
int main(int argc, char** argv) {
  dgs::Arrivals a((uint32_t)std::atoi(argv[1]));
  for (int i = 2; i < argc; ++i) {
    const int w = std::atoi(argv[i]);
    if (w < 0) a.joined(); else a.arrived((uint32_t)w);
    std::printf("%u\n", a.abreast() * 10 + (a.lone() ? 1 : 0));
  }
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("arrivals")
    (d / "main.cpp").write_text(MAIN)
    subprocess.check_call([shutil.which("g++") or "c++", "-std=c++17", "-Wall", "-Werror", "-I",
                           os.path.join(ROOT, "paper_1910_10929_b200", "csrc"), "-o", str(d / "main"), str(d / "main.cpp")])

    def go(workers, calls):
        out = subprocess.check_output([str(d / "main"), str(workers)] + [str(int(c)) for c in calls], text=True)
        return [(int(x) // 10, int(x) % 10 == 1) for x in out.split()]
    return go


def rounds(workers, length, times):
    calls, w = [], 0
    for _ in range(times):
        for _ in range(length):
            calls.append(w % workers)
            w += 1
        calls.append(-1)
    return calls


@pytest.mark.parametrize("workers,length,abreast,lone", [
    (1, 1, 1, True),       # one arrival at a time
    (8, 1, 1, True),
    (1, 32, 1, False),     # a worker by itself: every event waits for the one before it
    (3, 32, 1, False),
    (4, 32, 4, False),
    (7, 32, 4, False),
    (8, 32, 8, False),
    (32, 32, 8, False),
    (4, 4, 1, False),      # short rounds: the last events have nothing beside them
    (8, 4, 1, False),
    (5, 5, 4, False),
    (8, 8, 8, False),
    (65535, 8, 8, False),
])
def test_workers_in_turn(run, workers, length, abreast, lone):
    calls = rounds(workers, length, 12)
    last = [r for r, c in zip(run(workers, calls), calls) if c >= 0][-length:]
    assert last == [(abreast, lone)] * length


@pytest.mark.parametrize("workers", [8, 32])
def test_workers_at_random(run, workers):
    calls = np.random.default_rng(workers).integers(0, workers, 400)
    got = [a for a, _ in run(workers, calls)][40:]
    assert got.count(8) < len(got) // 20 and got.count(1) > len(got) * 3 // 4


def test_a_change_of_pattern(run):
    chain, turns = [0] * 40, list(range(16)) * 6
    got = [a for a, _ in run(16, chain + turns)]
    assert got[39] == 1
    assert got[40 + 31] == 1 and set(got[40 + 32:]) == {8}     # two rounds of the workers later
    got = [a for a, _ in run(16, turns + chain)]
    assert got[len(turns) - 1] == 8 and set(got[len(turns) + 1:]) == {1}
    # joins with nothing between them say nothing, and one arrival does
    assert run(16, turns + [-1, -1, -1])[-1] == (8, False)
    assert run(16, turns + [-1, 3, -1])[-1] == (1, True)
