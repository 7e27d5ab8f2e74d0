"""The integer form of the deposit's cell decision (csrc/fixpt.h, fix_split)
against cic_split of the two-rounding coordinate: wherever it decides, cell,
weight and inside / outside are the same bits; it leaves few coordinates
undecided; the fraction agrees to the coordinate's own rounding.  Random
coordinates over and around the grid, node lines and weight ties with their
neighbours, the ends of the grid, tiny, huge and non-finite values, grids of
several sizes, off-centre and one-sided.  Host compile, no GPU."""
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
#include <limits>
#include <random>
#include "fixpt.h"
using namespace sc;
static long bad = 0, unsure = 0, seen = 0;
static bool sum;
static SumAxis sx;
static void one(const FixAxis& ax, double x, double xmin, double inv, int cells) {
  const volatile double d = x - xmin;
  const volatile double xi = d * inv;
  int i = 0, a = 0;
  double f = 0;
  const bool in = cic_split(xi, cells, i, a, &f);
  int gi, gw;
  uint64_t z = 0;
  const int r = sum ? sum_split(sx, x, gi, gw) : fix_split(ax, x, gi, gw, z);
  ++seen;
  if (r < 0) { ++unsure; return; }
  bool ok = (r == 1) == in;
  if (ok && in) ok = gi == i && gw == a && (sum || fabs(fix_fraction(ax, z) - f) <= (cells + 1) * 0x1p-52 + 0x1p-52);
  if (!ok && ++bad < 6) printf("bad x %.17g xi %.17g in %d/%d i %d/%d w %d/%d\n", x, xi, r, in, gi, i, gw, a);
}
int main(int argc, char** argv) {
  const double xmin = atof(argv[1]), xmax = atof(argv[2]);
  const int n = atoi(argv[3]), cells = n - 1;
  const double h = (xmax - xmin) / cells, inv = 1.0 / h;
  const FixAxis ax = make_fix_axis(xmin, inv, cells);
  sum = argc > 4 && argv[4][0] == 's';
  sx = make_sum_axis(xmin, inv, cells);
  if (sum ? !sx.f : !ax.top) { printf("off\n"); return 0; }
  std::mt19937_64 g(n);
  std::uniform_real_distribution<double> U(0, 1);
  for (long k = 0; k < 2000000; ++k) one(ax, xmin + (xmax - xmin) * (1.2 * U(g) - 0.1), xmin, inv, cells);
  const long random_unsure = unsure, random_seen = seen;
  for (int k = 0; k <= 200000; ++k) {  // places where the decision changes, and their neighbours
    const double units = k < 4 * n ? k * 0.25 : floor(U(g) * cells * 2097152.0) / 2097152.0;
    double x = xmin + units * h;
    for (int s = 0; s < 3; ++s) x = nextafter(x, -INFINITY);
    for (int s = 0; s < 7; ++s, x = nextafter(x, INFINITY)) one(ax, x, xmin, inv, cells);
  }
  const double inf = std::numeric_limits<double>::infinity(), nan = std::nan("");
  for (double x : {0.0, -0.0, 5e-324, -5e-324, 1e-300, xmin, xmax, -xmin, -xmax, 2 * xmax, 2 * xmin, 1e6, -1e6, 1e300, -1e300,
                   inf, -inf, nan})
    one(ax, x, xmin, inv, cells);
  for (int k = 0; k < 200000; ++k) {  // bit patterns
    uint64_t b = g();
    one(ax, bits_f64(b), xmin, inv, cells);
  }
  printf("%ld %ld %ld\n", bad, random_unsure, random_seen);
  return 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("fix_axis")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run([cxx, "-std=gnu++17", "-O2", "-ffp-contract=off", "-I", CSRC, str(d / "h.cpp"), "-o", str(d / "h")],
                   check=True)
    return d / "h"


@pytest.mark.parametrize("kind", ["bits", "sum"])
@pytest.mark.parametrize("xmin,xmax,n", [
    (-0.02, 0.02, 128), (-0.015, 0.015, 256), (-0.01, 0.01, 64), (-0.02, 0.02, 129), (0.0, 1.0, 16), (-0.012, 0.009, 33),
    (0.01, 0.02, 512), (-0.03, -0.01, 65), (-60.0, 60.0, 33), (-1e-9, 1e-9, 128), (-4.0, 4.0, 4097), (-1e6, 1e6, 9),
    (-0.02, 1e-7, 100), (1000.0, 1000.5, 64), (-0.02, 0.02, 2)])
def test_decides_as_the_two_roundings(harness, xmin, xmax, n, kind):
    out = subprocess.run([str(harness), repr(xmin), repr(xmax), str(n), kind], check=True, capture_output=True,
                         text=True).stdout
    if kind == "sum" and out.strip() == "off":  # too few bits for this axis: the caller keeps cic_split
        assert xmin >= 1000.0
        return
    bad, unsure, seen = map(int, out.split()[-3:])
    assert bad == 0, out
    if kind == "bits":
        share = 2.0 ** -7 * (1 if xmin >= 100 else 2.0 ** -8)
    else:  # 2 T of each 2^(F - 21) units, T <= 10, F >= 50 - log2(cells) (less what an off-centre grid loses)
        share = 20 * (n - 1) * 2.0 ** -29 * max(1.0, 2 * max(abs(xmin), abs(xmax)) / (xmax - xmin))
    assert unsure <= 20 + seen * share, out


def test_unusable_axes_are_refused(harness):
    """Axes whose integers would leave too much undecided: the caller keeps cic_split."""
    for args in (("1e9", "1000000000.5", "64"), ("-0.02", "0.02", "5000"), ("-1e300", "1e300", "8")):
        assert subprocess.run([str(harness), *args], check=True, capture_output=True, text=True).stdout.strip() == "off"
