"""Float pairs (csrc/dfloat.h) against long double on the host: the split of a
double, the way back, the two power series over their whole ranges, and the
quadrupole's path-length sum.  Bounds are the ones the header derives."""
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
static double worst = 0;
static void see(Q err, Q bound) { const double r = (double)(fabsl(err) / bound); if (!(r <= worst)) worst = r; }
static Q val(F2 a) { return (Q)a.h + (Q)a.l; }
int main() {
  std::mt19937_64 g(7);
  std::uniform_real_distribution<double> U(-1, 1);
  const Q p46 = ldexpl(1, -46), p52 = ldexpl(1, -52), p53 = ldexpl(1, -53);
  // split and back: any size from 2^-95 to 2^127
  for (int i = 0; i < 400000; ++i) {
    const double v = U(g) * ldexp(1.0, (int)(U(g) * 60));
    if (fabs(v) < ldexp(1.0, -70)) continue;
    const F2 a = f2_split(v);
    see(val(a) - v, p46 * fabsl((Q)v));
    const F2 b{a.h, (float)(a.h * 5e-8 * U(g))};
    see(f2_to_double(b) - val(b), p52 * fabsl(val(b)));
    const F2 c = f2_unpack(f2_pack(b));
    if (c.h != b.h || c.l != b.l) see(2, 1);
  }
  printf("split %.3f\n", worst); worst = 0;
  for (double v : {1.0, -1.0, 2.0, 1.5, 0x1.fffffffffffffp0, -0x1.0000000000001p5, 0x1p-60, 0x1p126}) {
    see(val(f2_split(v)) - v, p46 * fabsl((Q)v));
    see(f2_to_double(f2_split(v)) - val(f2_split(v)), p52 * fabsl((Q)v));
  }
  for (double v : {0.0, -0.0, 5e-324, 1e-300}) see(fabsl(val(f2_split(v))), ldexpl(1, -94));
  if (f2_to_double(F2{0.f, 0.f}) != 0.0) see(2, 1);
  printf("edges %.3f\n", worst); worst = 0;
  for (int e = -60; e <= -10; ++e)
    for (int i = 0; i < 4000; ++i) {
      const F2 u = f2_split(ldexp(1.0 - 0.5 * fabs(U(g)) - 1e-9, e));
      const Q x = val(u);
      Q s = 0;  // the binomial series, summed until it no longer matters
      Q c = 1;
      for (int k = 1; k < 40; ++k) { c *= x * (2 * k - 1) / (2 * k); s += c; }
      see(val(rsqrt1m_series(u)) - s, ldexpl(1, -54));
    }
  printf("rsqrt %.3f\n", worst); worst = 0;
  for (int e = -60; e <= -9; ++e)
    for (int i = 0; i < 4000; ++i) {
      const double sgn = U(g) < 0 ? -1 : 1;
      const F2 v = f2_split(sgn * ldexp(1.0 - 0.5 * fabs(U(g)) - 1e-9, e));
      const Q x = val(v);
      see(val(one_minus_sqrt1m(v)) - x / (1 + sqrtl(1 - x)), p53);
    }
  printf("sqrt %.3f\n", worst); worst = 0;
  for (int e = -60; e <= -7; ++e)
    for (int i = 0; i < 4000; ++i) {
      const double sgn = U(g) < 0 ? -1 : 1;
      const F2 u = f2_split(sgn * ldexp(1.0 - 0.5 * fabs(U(g)) - 1e-9, e));
      const Q x = val(u);
      see(val(rsqrt1m_wide(u)) - x / (sqrtl(1 - x) * (1 + sqrtl(1 - x))), ldexpl(1, -53));
    }
  printf("wide %.3f\n", worst); worst = 0;
  for (int i = 0; i < 200000; ++i) {
    double d[12];
    for (double& v : d) v = U(g) * ldexp(1.0, (int)(U(g) * 12));
    F2 f[12];
    for (int k = 0; k < 12; ++k) f[k] = f2_split(d[k]);
    const F2 K = f2_split(U(g));
    Q q[12];
    for (int k = 0; k < 12; ++k) q[k] = val(f[k]);
    const Q k = val(K);
    const Q t = q[4] * q[5] + q[6] * q[7] + q[0] * (k * q[0] - q[1]) - q[2] * (k * q[2] + q[3]);
    const Q ref = q[8] * q[11] - q[10] * (q[1] * q[1] + q[3] * q[3]) - q[9] * t;
    const Q size = fabsl(q[8] * q[11]) + fabsl(q[10]) * (q[1] * q[1] + q[3] * q[3]) +
                   fabsl(q[9]) * (fabsl(q[4] * q[5]) + fabsl(q[6] * q[7]) + fabsl(k) * (q[0] * q[0] + q[2] * q[2]) +
                                  fabsl(q[0] * q[1]) + fabsl(q[2] * q[3]));
    const F2 got = quad_slip(f[0], f[1], f[2], f[3], f[4], f[5], f[6], f[7], f[8], f[9], f[10], f[11], K);
    see(val(got) - ref, 14 * p46 * size);  // three products (3 each) and five sums in a row
  }
  printf("slip %.3f\n", worst);
  return 0;
}
"""


@pytest.fixture(scope="module")
def results(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("dfloat")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-I", CSRC, str(d / "h.cpp"), "-o", str(d / "h")],
                   check=True)
    out = subprocess.run([str(d / "h")], check=True, capture_output=True, text=True).stdout
    return {k: float(v) for k, v in (line.split() for line in out.splitlines())}


@pytest.mark.parametrize("what", ["split", "edges", "rsqrt", "sqrt", "wide", "slip"])
def test_within_the_stated_bound(results, what):
    assert results[what] <= 1.0, results
