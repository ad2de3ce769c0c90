"""The ensemble's choice between one and two blocks of 256 per SM
(csrc/batch_plan.h), compiled for the host: the model's times on small plans
that can be followed by hand, and the rule on both sides of its lines."""
import os
import subprocess

import pytest

from paper_1505_02037_gb300 import autotune

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1505_02037_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "batch_plan.h"
int main(int argc, char** argv) {
  auto d = [&](int i) { return atof(argv[i]); };
  if (!strcmp(argv[1], "rule")) {
    puts(lbnr::two_per_sm((size_t)d(2), (int64_t)d(3), (int64_t)d(4), d(5), d(6), d(7)) ? "2" : "1");
  } else {  // workers, block, then cost, cells, team of each run
    std::vector<double> cost;
    std::vector<int64_t> cells;
    std::vector<int> team;
    for (int i = 4; i < argc; i += 3) {
      cost.push_back(d(i));
      cells.push_back((int64_t)d(i + 1));
      team.push_back((int)d(i + 2));
    }
    printf("%.17g\n", lbnr::imbalance(cost, cells, team, (int)d(2), (int)d(3)));
  }
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "p.cpp").write_text(PROGRAM)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-I" + CSRC, str(d / "p.cpp"), "-o",
                           str(d / "p")])
    return lambda *a: subprocess.check_output([str(d / "p"), *map(str, a)], text=True).strip()


@pytest.mark.parametrize("workers,block,runs,want", [
    (4, 100, [(400, 400, 2), (400, 400, 2)], 1.0),
    (4, 100, [(400, 400, 4)], 1.0),
    (4, 100, [(500, 500, 4)], 200 * 4 / 500),              # two rounds, the second a quarter full
    (4, 100, [(300, 100, 1)], 4.0),                        # three blocks idle
    (2, 100, [(300, 100, 1), (200, 100, 1), (100, 100, 1)], 1.0),   # longest first
    (3, 100, [(200, 200, 2), (100, 100, 1), (100, 100, 1)], 200 * 3 / 400),
    (4, 100, [(400, 400, 4), (999, 100, 0)], 1.0),         # a stopped run
    (4, 100, [(9, 1, 0)], 1.0),
])
def test_imbalance(run, workers, block, runs, want):
    got = float(run("model", workers, block, *[v for r in runs for v in r]))
    assert got == pytest.approx(want, rel=1e-12)


@pytest.mark.parametrize("nbytes,cells,cells_2d,single,one,two,want", [
    (2, 119999, 0, 0, 1, 1, 1), (4, 119999, 0, 0, 2, 1, 1), (8, 119999, 0, 0, 2, 1, 1),
    (2, 120000, 120000, 1, 1, 2, 2), (2, 50000000, 50000000, 0, 1, 2, 2),
    (8, 120000, 120000, 0.75, 1, 2, 2), (8, 5000000, 0, 0.76, 2, 1, 1),
    (4, 120000, 120000, 0, 1, 2, 2), (4, 5000000, 700000, 0, 1, 2, 2),
    (4, 800000, 700001, 0, 1.03, 1, 1), (4, 2000000, 2000000, 0, 1.04, 1, 2),
    (4, 2000001, 2000001, 0, 1.04, 1, 1), (4, 2000001, 2000001, 0, 1.1, 1, 2),
    (4, 18000000, 18000000, 0.27, 1.47, 1.77, 1),
])
def test_rule(run, nbytes, cells, cells_2d, single, one, two, want):
    assert int(run("rule", nbytes, cells, cells_2d, single, one, two)) == want


def test_the_tuner_times_every_shape_of_the_rule():
    assert {(256, 1), (256, 2)} <= set(autotune.batch_shapes())
