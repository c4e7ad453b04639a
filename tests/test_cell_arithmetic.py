"""Integer cell arithmetic (csrc/cell.cuh) against the float64 formula it stands for: the cell, the
in-cell offset and the fixed-point contributions, bit for bit, on the CPU."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_15209_gb300", "csrc")

SOURCE = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "cell.cuh"
using namespace zk;
static int f64(float x, double ih, int n, float& t) {
  double u = (double)x * ih;
  u -= floor(u / n) * n;
  int i = (int)floor(u);
  double fr = u - i;
  if (i >= n) i -= n;
  if (i < 0) i += n;
  t = (float)fr;
  if (t >= 1.0f) t = 0.99999994f;
  return i;
}
int main() {
  std::mt19937_64 g(1);
  std::uniform_real_distribution<double> U(0, 1);
  long long bad = 0, fast = 0, inside = 0;
  const double boxes[] = {500.0, 1000.0, 2000.0, 333.3, 0.1, 7.7e5};
  for (int n = 16; n <= 512; n *= 2)
    for (double box : boxes) {
      const CellScale c = make_cell_scale(n, box);
      for (int k = 0; k < 60000; ++k) {
        float x;
        if (k % 4 < 2) x = (float)(U(g) * box);                             // anywhere
        else if (k % 4 == 2) {                                              // at and beside a face
          x = (float)((int)(U(g) * n + 0.5) * (box / n));
          for (int q = (int)(U(g) * 3); q > 0; --q) x = nextafterf(x, g() & 1 ? 1e30f : -1e30f);
        } else x = (float)(U(g) * box * pow(2.0, -60 * U(g)) * (g() & 1 ? 1 : -1));  // tiny, negative
        float t0, t1 = -1.f;
        int i1 = -1;
        const int i0 = f64(x, c.inv_h, n, t0);
        if (k % 4 < 2) ++inside;
        if (cell_int(x, c, n, i1, t1)) {
          if (k % 4 < 2) ++fast;
          if (i0 != i1 || zk_float_bits(t0) != zk_float_bits(t1)) ++bad;
        }
      }
    }
  for (int k = 0; k < 3000000; ++k) {
    const float w = (float)ldexp((double)((g() >> 40) | 1), (int)(g() % 40) - 40) * (g() & 1 ? 1 : -1);
    float b = (float)(g() >> 40) / (1 << 24);
    if (k % 4 == 0) b = ldexpf(b, -(int)(g() % 60));
    int e;
    frexp((double)fabsf(w) * (1 + (double)(g() % 1000000)), &e);
    if (llrint((double)w * ldexp(1.0, 61 - e) * (double)b) != fix64_prod(w, b, 61 - e)) ++bad;
  }
  printf("%lld %lld %lld\n", bad, fast, inside);
}
"""


def test_integer_forms_equal_the_float64_formula(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src = tmp_path / "cell.cpp"
    src.write_text(SOURCE)
    exe = tmp_path / "cell"
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-x", "c++", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    bad, fast, inside = map(int, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert bad == 0
    assert fast > 0.99 * inside  # particles inside the box take the integer form
