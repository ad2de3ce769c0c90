"""The short form of the Bona-Masso sources and fluxes (physics.cuh) against
the form that follows the printed sums, compiled for the host: every set's
axes, every slicing, FP64."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1505_02037_gb300", "csrc")

PROGRAM = r"""
#define __device__
#define __host__
#define __forceinline__ inline
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include "physics.cuh"
using namespace lbnr;
static double u() { return 2.0 * drand48() - 1.0; }
int main() {
  double worst = 0;
  for (int it = 0; it < 2000; ++it) {
    double al = 1 + 0.3 * u(), g[6] = {1, 0, 0, 1, 0, 1}, K[6], V[3], A[3], D[3][6];
    for (int q = 0; q < 6; ++q) { g[q] += 0.2 * u(); K[q] = u(); }
    for (int k = 0; k < 3; ++k) {
      V[k] = u();
      A[k] = k < DIM ? u() : 0;
      for (int q = 0; q < 6; ++q) D[k][q] = k < DIM ? u() : 0;
    }
    double S[16], P[16], F[6][3], G[6][3];
    bm_sources<double, DIM>(al, g, K, V, A, D, it % 3, S, 0.3);
    bm_sources_plain<double>(al, g, K, V, A, D, it % 3, P, 0.3);
    bm_flux<double, DIM>(al, g, V, A, D, F);
    bm_flux_plain<double, DIM>(al, g, V, A, D, G);
    for (int i = 0; i < 16; ++i) worst = fmax(worst, fabs(S[i] - P[i]));
    for (int q = 0; q < 6; ++q)
      for (int k = 0; k < 3; ++k) worst = fmax(worst, fabs(F[q][k] - G[q][k]));
  }
  printf("%.17g\n", worst);
}
"""


@pytest.mark.parametrize("dim", [1, 2, 3])
def test_short_sources_equal_the_printed_sums(tmp_path, dim):
    """A source is a sum of at most 400 products of at most four factors, each
    below 4 here (the metric is within 0.6 of the identity in norm, so its
    inverse is below 2.5): rounding moves it by at most (400 + 4) u 400 4^4,
    and twice that for the difference of the two."""
    src = tmp_path / "p.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "p"
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-Wno-unknown-pragmas", f"-DDIM={dim}",
                           "-I" + CSRC, str(src), "-o", str(exe)])
    worst = float(subprocess.check_output([str(exe)]))
    assert worst <= 2 * 404 * 400 * 4 ** 4 * 2.0 ** -53, worst
