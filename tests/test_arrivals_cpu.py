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
// argv: workers, then a worker's number for an arrival or -1 for a join; prints abreast(), lone() and chained() after each
int main(int argc, char** argv) {
  dgs::Arrivals a((uint32_t)std::atoi(argv[1]));
  for (int i = 2; i < argc; ++i) {
    const int w = std::atoi(argv[i]);
    if (w < 0) a.joined(); else a.arrived((uint32_t)w);
    std::printf("%u %d %d\n", a.abreast(), a.lone(), a.chained());
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
        return [tuple(int(x) for x in line.split()) for line in out.splitlines()]
    return go


def rounds(workers, length, times):
    calls, w = [], 0
    for _ in range(times):
        for _ in range(length):
            calls.append(w % workers)
            w += 1
        calls.append(-1)
    return calls


@pytest.mark.parametrize("workers,length,abreast,lone,chained", [
    (1, 1, 1, 1, 0),       # one arrival at a time
    (8, 1, 1, 1, 0),
    (1, 32, 1, 0, 1),     # a worker by itself: every event waits for the one before it
    (3, 32, 1, 0, 1),
    (4, 32, 4, 0, 0),
    (7, 32, 4, 0, 0),
    (8, 32, 8, 0, 0),
    (32, 32, 8, 0, 0),
    (4, 4, 1, 0, 0),      # short rounds: the last events have nothing beside them
    (8, 4, 1, 0, 0),
    (5, 5, 4, 0, 0),
    (8, 8, 8, 0, 0),
    (65535, 8, 8, 0, 0),
])
def test_workers_in_turn(run, workers, length, abreast, lone, chained):
    calls = rounds(workers, length, 12)
    last = [r for r, c in zip(run(workers, calls), calls) if c >= 0][-length:]
    assert last == [(abreast, lone, chained)] * length


@pytest.mark.parametrize("workers", [8, 32])
def test_workers_at_random(run, workers):
    calls = np.random.default_rng(workers).integers(0, workers, 400)
    got = run(workers, calls)[40:]
    abreast = [a for a, _, _ in got]
    assert abreast.count(8) < len(got) // 20 and abreast.count(1) > len(got) * 3 // 4
    assert sum(c for _, _, c in got) > len(got) * 3 // 4


def test_a_change_of_pattern(run):
    chain, turns = [0] * 40, list(range(16)) * 6
    got = [a for a, _, _ in run(16, chain + turns)]
    assert got[39] == 1
    assert got[40 + 31] == 1 and set(got[40 + 32:]) == {8}     # two rounds of the workers later
    got = [a for a, _, _ in run(16, turns + chain)]
    assert got[len(turns) - 1] == 8 and set(got[len(turns) + 1:]) == {1}
    # joins with nothing between them say nothing, and one arrival does
    assert run(16, turns + [-1, -1, -1])[-1] == (8, 0, 0)
    assert run(16, turns + [-1, 3, -1])[-1] == (1, 1, 0)
