"""Cell fractions from 64-bit integers (csrc/fixpt.h, fix_fraction) are taken
where fix_fraction_serves says so: there they are within the two-rounding
fraction's own error, cells 2^-53, of the exact one; grids far off centre, whose
integers are short of that, are refused.  Host compile, no GPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2010_11540_gb300", "csrc")

HARNESS = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include "fixpt.h"
using namespace sc;
int main(int argc, char** argv) {
  const double xmin = atof(argv[1]), xmax = atof(argv[2]);
  const int cells = atoi(argv[3]) - 1;
  const double inv = 1.0 / ((xmax - xmin) / cells);
  const FixAxis ax = make_fix_axis(xmin, inv, cells);
  std::mt19937_64 g(cells);
  std::uniform_real_distribution<double> U(0, 1);
  long double worst = 0;
  for (int k = 0; ax.top && k < 400000; ++k) {
    const double x = xmin + (xmax - xmin) * U(g);
    int i, w;
    uint64_t z;
    if (fix_split(ax, x, i, w, z) != 1) continue;
    const long double e = fabsl(((long double)x - xmin) * inv - i - fix_fraction(ax, z));
    if (!(e <= worst)) worst = e;
  }
  printf("%d %.6Lg\n", (int)fix_fraction_serves(ax), worst / (cells * ldexpl(1, -53)));
  return 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("fix_fraction")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run([cxx, "-std=gnu++17", "-O2", "-ffp-contract=off", "-I", CSRC, str(d / "h.cpp"), "-o", str(d / "h")],
                   check=True)
    return d / "h"


@pytest.mark.parametrize("xmin,xmax,n,serves", [
    (-0.02, 0.02, 128, True), (-0.015, 0.015, 256, True), (0.0, 1.0, 16, True), (0.01, 0.02, 512, True),
    (-4.0, 4.0, 4097, True), (-0.02, 0.02, 2, True), (0.5, 0.54, 64, True), (1000.0, 1000.3, 64, False),
    (-300.3, -300.0, 33, False), (1e9, 1000000000.5, 64, False)])
def test_served_fractions_are_as_exact(harness, xmin, xmax, n, serves):
    out = subprocess.run([str(harness), repr(xmin), repr(xmax), str(n)], check=True, capture_output=True, text=True).stdout
    got, worst = out.split()
    assert int(got) == serves, out
    if serves:
        assert float(worst) <= 1.0, out
    elif xmin < 1e6:
        assert float(worst) > 1.0, out  # what the rule keeps out
