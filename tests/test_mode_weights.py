"""Integer mode weights of the uniform term and the 2PCF (csrc/mass.cuh) on the CPU: each within 2^-57 of the
exact product, the fixed-point units rounded to nearest, and the tables that they read even in the frequency."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2507_15209_gb300 import zeta as Z

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_15209_gb300", "csrc")

SOURCE = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "mass.cuh"
using namespace zk;
typedef __int128 i128;
// |value| of a float as mant 2^exp
static i128 mant(float x, int& e) {
  int q;
  const double m = frexp(fabs((double)x), &q);
  e = q - 24;
  return (i128)ldexp(m, 24);
}
// w / exact - 1 with the exact product in three words: the error of w.m 2^w.e, relative, in long double steps that
// are exact up to the last division
static double rel_err(float x, float y, float a, float b, float c, int twice, WideFactor w) {
  int ex, ey, ea, eb, ec;
  i128 mx = mant(x, ex), my = mant(y, ey), ma = mant(a, ea), mb = mant(b, eb), mc = mant(c, ec);
  if (mx == 0) ex = ey;
  if (my == 0) ey = ex;
  if (ex < ey) { std::swap(ex, ey); std::swap(mx, my); }
  const int d = 2 * (ex - ey);
  // s 2^(2 ex - 60): the smaller square shifted in when it reaches that far (else it is below 2^-60 of s)
  i128 s = ((mx * mx) << 60) + (d <= 60 ? (my * my) << (60 - d) : d < 170 ? (my * my) >> (d - 60) : 0);
  // s has at most 109 bits, t = ma mb mc at most 72: the product in 64-bit limbs
  const i128 t = ma * mb * mc;
  const unsigned long long s0 = (unsigned long long)s, s1 = (unsigned long long)(s >> 64);
  const unsigned long long t0 = (unsigned long long)t, t1 = (unsigned long long)(t >> 64);
  unsigned __int128 p00 = (unsigned __int128)s0 * t0, p01 = (unsigned __int128)s0 * t1, p10 = (unsigned __int128)s1 * t0,
                    p11 = (unsigned __int128)s1 * t1;
  unsigned __int128 mid = (p00 >> 64) + (unsigned long long)p01 + (unsigned long long)p10;
  unsigned __int128 hi = p11 + (p01 >> 64) + (p10 >> 64) + (mid >> 64);
  // exact = hi 2^128 + mid 2^64 + ..., times 2^(2 ex - 60 + ea + eb + ec + twice)
  const int e0 = 2 * ex - 60 + ea + eb + ec + twice;
  // compare w.m 2^w.e with it: bring both to 2^(e0 + 64)
  unsigned __int128 lo64 = (hi << 64) | (unsigned long long)mid;  // hi stays below 2^54
  const int sh = w.e - (e0 + 64);
  if (sh < 0 || sh > 60) return 1.0;
  const i128 diff = (i128)((unsigned __int128)w.m << sh) - (i128)lo64;
  return (double)diff / (double)lo64;
}
int main() {
  std::mt19937_64 g(3);
  auto rnd = [&](int lo, int hi) { return (float)ldexp(1 + (g() >> 41) * 0x1p-23, lo + (int)(g() % (unsigned)(hi - lo))); };
  double worst = 0;
  long long bad = 0;
  for (int k = 0; k < 1000000; ++k) {
    const int base = (int)(g() % 240) - 120;
    float x = rnd(base, base + 1), y = rnd(base - (int)(g() % 40), base + 1);
    if (y < 1e-37f || k % 50 == 0) y = 0.f;
    if (g() & 1) x = -x;
    if (g() & 1) y = -y;
    if (g() & 1) std::swap(x, y);
    const float a = rnd(-15, 0), b = rnd(-15, 0), c = k % 9 ? rnd(-15, 0) : 1.f;
    const int twice = g() & 1;
    const WideFactor w = mode_weight(x, y, wide_product(a, b, c), twice);
    if (w.m < (1ULL << 60)) ++bad;
    const double r = rel_err(x, y, a, b, c, twice, w);
    if (fabs(r) > worst) worst = fabs(r);
    // the bound and the units: w.m 2^w.e in [2^(k-1), 2^k); rounding to nearest
    const int top = wide_ceil(w);
    const long double v = ldexpl((long double)w.m, w.e - top);
    if (!(v >= 0.5L && v < 1.0L)) ++bad;
    const int unit = top - 52 + (int)(g() % 3) * 20;
    const long double q = ldexpl((long double)w.m, w.e - unit);
    const unsigned long long u = wide_units(w, unit);
    if (fabsl((long double)u - q) > 0.5L || u > (1ULL << 52)) ++bad;
  }
  const WideFactor one = wide_product(1.f, 1.f, 1.f);
  if (mode_weight(0.f, 0.f, one, 1).m || mode_weight(1.f, 0.f, wide_product(1.f, 0.f, 1.f), 0).m) ++bad;
  if (wide_units(mode_weight(3.f, 4.f, one, 1), -1) != 100) ++bad;            // 25 * 2 in halves
  if (wide_units(mode_weight(1e-45f, 0.f, one, 0), -298) != 1) ++bad;         // the smallest denormal, squared
  printf("%lld %g\n", bad, worst);
}
"""


def test_mode_weights(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src = tmp_path / "mass.cpp"
    src.write_text(SOURCE)
    exe = tmp_path / "mass"
    subprocess.run([cxx, "-std=c++17", "-O2", "-x", "c++", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    bad, worst = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert int(bad) == 0
    assert float(worst) < 2.0 ** -57  # a float64 evaluation: five roundings of 2^-53


@pytest.mark.parametrize("n", [16, 32, 64, 128, 256, 512])
@pytest.mark.parametrize("dsup", [2, 3, 4])
def test_tables_are_even(n, dsup):
    """The kernels take the table value of |n_d| for both signs."""
    m = Z.host_mass_hat(n, dsup)
    ph = np.empty(n)
    assert Z.lib().zeta_host_phi_hat(n, dsup, ph.ctypes.data) == 0
    for t in (m, ph, m * ph * ph):
        f = t.astype(np.float32)
        np.testing.assert_array_equal(f[1:], f[:0:-1])
        assert 0 < f.min() and f.max() <= 1
