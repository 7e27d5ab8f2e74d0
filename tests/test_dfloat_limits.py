"""The size by which a quadrupole's path length is judged fit for a float pair
(csrc/dfloat.h, quad_slip_size), on the host against long double: at states of
any size, with and without cancellation, it covers the pair's error."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2010_11540_gb300", "csrc")

HARNESS = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "dfloat.h"
using namespace sc;
typedef long double Q;
static Q val(F2 a) { return (Q)a.h + (Q)a.l; }
int main() {
  std::mt19937_64 g(11);
  std::uniform_real_distribution<double> U(-1, 1);
  long beyond = 0;
  for (int i = 0; i < 400000; ++i) {
    double d[12];
    const double amp = 20 * U(g);
    for (double& v : d) v = U(g) * ldexp(1.0, (int)(amp * 0.5 + 10 * U(g)));
    F2 f[12];
    for (int k = 0; k < 12; ++k) f[k] = f2_split(d[k]);
    const double kd = U(g);
    const F2 K = f2_split(kd);
    Q q[12];
    for (int k = 0; k < 12; ++k) q[k] = d[k];
    const Q t = q[4] * q[5] + q[6] * q[7] + q[0] * (kd * q[0] - q[1]) - q[2] * (kd * q[2] + q[3]);
    const Q ref = q[8] * q[11] - q[10] * (q[1] * q[1] + q[3] * q[3]) - q[9] * t;
    const F2 L4{fabsf(f[10].h), f[10].h < 0 ? -f[10].l : f[10].l};
    const Q ref4 = q[10] < 0 ? ref + 2 * q[10] * (q[1] * q[1] + q[3] * q[3]) : ref;
    const Q got = val(quad_slip(f[0], f[1], f[2], f[3], f[4], f[5], f[6], f[7], f[8], f[9], L4, f[11], K));
    const float size = quad_slip_size(f[0], f[1], f[2], f[3], f[4], f[5], f[6], f[7], f[8], f[9], L4, f[11], K);
    // the sums' 14 2^-46, and 2^-46 of each of at most four factors split from float64
    if (!(fabsl(got - ref4) <= 18 * ldexpl(1, -46) * size)) ++beyond;
  }
  printf("%ld\n", beyond);
  return 0;
}
"""


def test_sizes_cover_the_errors(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    (tmp_path / "h.cpp").write_text(HARNESS)
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-I", CSRC, str(tmp_path / "h.cpp"), "-o",
                    str(tmp_path / "h")], check=True)
    out = subprocess.run([str(tmp_path / "h")], check=True, capture_output=True, text=True).stdout
    assert int(out) == 0, out
