"""The work list of the one-launch step (csrc/schedule.h), compiled for the
host: every tile once per pass, no item waits for one behind it in the list,
and a collide tile's stencil neighbours are among the moment tiles it waits
for. Lattices of odd sizes, in units of one or several planes and in strips."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1505_02037_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "schedule.h"
using namespace lbnr;
int main(int argc, char** argv) {
  const uint32_t nx = atoi(argv[1]), ny = atoi(argv[2]), nz = atoi(argv[3]);
  const Schedule s = make_schedule(nx, ny, nz, atoi(argv[4]), atoi(argv[5]));
  const uint32_t cells = nx * ny * nz, T = (cells + 31) / 32;
  std::vector<int> pos(T, -1), need(T, -1), count(s.units, 0);
  uint32_t upto = 0;
  for (uint32_t i = 0; i < s.items; ++i) {
    const Item t = item_at(s, i);
    uint32_t tile, n;
    if (t.pos < s.units) {
      ++count[t.pos];
      if (moment_tile(s, t, tile)) {
        if (tile >= T || pos[tile] >= 0) return puts("moment tile twice or out of range"), 1;
        pos[tile] = t.pos;
      }
    }
    while (upto < s.units && count[upto] == (int)s.slots) ++upto;
    if (collide_tile(s, t, tile, n)) {
      if (tile >= T || need[tile] >= 0) return puts("collide tile twice or out of range"), 1;
      if (n >= s.units || upto <= n) return puts("waits for an item behind it"), 1;
      need[tile] = n;
    }
  }
  if (upto != s.units) return puts("a unit never completes"), 1;
  for (uint32_t t = 0; t < T; ++t)
    if (pos[t] < 0 || need[t] < 0) return puts("tile left out"), 1;
  for (uint32_t c = 0; c < cells; ++c) {
    const uint32_t x = c % nx, y = c / nx % ny, z = c / nx / ny;
    const uint32_t nb[7] = {c,
                            (x + 1) % nx + nx * (y + ny * z), (x + nx - 1) % nx + nx * (y + ny * z),
                            x + nx * ((y + 1) % ny + ny * z), x + nx * ((y + ny - 1) % ny + ny * z),
                            x + nx * (y + ny * ((z + 1) % nz)),
                            x + nx * (y + ny * ((z + nz - 1) % nz))};
    for (uint32_t m : nb)
      if (pos[m / 32] > need[c / 32]) return puts("neighbour not waited for"), 1;
  }
  for (uint32_t d : {s.slots, s.upu})
    for (uint32_t n : {0u, 1u, d - 1, d, d + 1, 7 * d - 1, 7 * d, s.items - 1})
      if (make_fastdiv(d).div(n) != n / d) return puts("division"), 1;
  return 0;
}
"""

SHAPES = [(3, 1, 1, 1), (3, 32, 1, 1), (3, 5, 1, 3), (3, 2, 5, 3), (3, 37, 9, 5), (3, 8, 6, 1),
          (3, 64, 64, 64), (3, 67, 131, 5), (3, 96, 60, 7), (3, 131, 37, 6), (3, 40, 8, 200),
          (3, 149, 101, 67), (3, 256, 256, 6), (3, 1, 300, 40), (3, 300, 2, 40), (2, 1000, 77, 1),
          (2, 7, 901, 1), (1, 4097, 1, 1), (1, 200, 1, 1)]


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("schedule")
    (d / "p.cpp").write_text(PROGRAM)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I" + CSRC, str(d / "p.cpp"),
                           "-o", str(d / "p")])
    return str(d / "p")


@pytest.mark.parametrize("vset,nx,ny,nz", SHAPES)
@pytest.mark.parametrize("unit", [32, 200, 1024, 4096])
def test_work_list(program, vset, nx, ny, nz, unit):
    r = subprocess.run([program, str(nx), str(ny), str(nz), str(vset), str(unit)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
