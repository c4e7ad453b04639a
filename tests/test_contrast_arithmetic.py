"""The contrast of a node in float32 pairs (csrc/cell.cuh) against its float64 formula, bit for bit, and the
fixed-point products with factors of either sign, on the CPU."""
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
int main() {
  std::mt19937_64 g(2);
  long long bad = 0;
  for (int k = 0; k < 2000000; ++k) {
    const double inv = ldexp(1 + (g() >> 12) * 0x1p-52, -20 - (int)(g() % 60)) * (g() % 16 ? 1 : -1);
    const float ih = (float)inv, il = (float)(inv - (double)ih);
    // v inv - 1: ordinary contrasts, large ones, nearly empty nodes, and values next to the mean
    double c = ldexp(1 + (g() >> 12) * 0x1p-52, (int)(g() % 40) - 20);
    if (k % 4 == 0) c = 1 + ldexp((double)(g() >> 11) * 0x1p-53 - 0.5, -(int)(g() % 40));
    if (k % 5 == 0) c = -c;
    const double t = c / inv;
    if (!(fabs(t) < 9e18)) continue;
    long long v = (long long)t + (long long)(g() % 3) - 1;
    if (k % 7 == 0) v = (long long)(g() % 100) - 50;
    if (zk_float_bits(contrast_of(v, ih, il, inv)) != zk_float_bits((float)std::fma((double)v, inv, -1.0))) ++bad;
  }
  long long prod = 0;
  for (int k = 0; k < 1000000; ++k) {
    const float w = (float)ldexp((double)((g() >> 40) | 1), (int)(g() % 40) - 40) * (g() & 1 ? 1 : -1);
    float b = (float)((long long)(g() >> 39) - (1 << 24)) / (1 << 24);
    if (k % 4 == 0) b = ldexpf(b, -(int)(g() % 60));
    int e;
    frexp((double)fabsf(w) * (1 + (double)(g() % 1000000)), &e);
    if (llrint((double)w * ldexp(1.0, 61 - e) * (double)b) != fix64_prod(w, b, 61 - e)) ++prod;
  }
  printf("%lld %lld\n", bad, prod);
}
"""


# contracted products would break the pairs: the arithmetic may not depend on that choice of the compiler
@pytest.mark.parametrize("contract", ["off", "fast"])
def test_contrast_and_signed_products(tmp_path, contract):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src = tmp_path / "contrast.cpp"
    src.write_text(SOURCE)
    exe = tmp_path / "contrast"
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=" + contract, "-x", "c++", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True)
    bad, prod = map(int, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert bad == 0
    assert prod == 0
