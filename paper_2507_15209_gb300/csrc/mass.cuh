// Weight of a Fourier mode in the uniform term and the 2PCF, (1 or 2) |delta_hat|^2 M(n_x) M(n_y) M(n_z) with
// float32 delta_hat and tables, in integer arithmetic (the float64 pipe of this part retires about two
// operations per SM and clock).  A squared float32 and a product of two are 48-bit integers; they are
// carried on in 64 bits with their binary exponent, and what is cut off on the way is below 2^-58 of the
// weight: less than the float64 expression rounds (five roundings of 2^-53).
#pragma once
#include "cell.cuh"

namespace zk {

// m 2^e, m == 0 or m >= 2^61
struct WideFactor {
  unsigned long long m;
  int e;
};

// |f| as mant 2^(exp - 150)
ZK_HD unsigned long long float_mant(uint32_t bits, int& exp) {
  exp = static_cast<int>((bits >> 23) & 0xffu);
  if (exp == 0) {
    exp = 1;
    return bits & 0x7fffffu;
  }
  return (bits & 0x7fffffu) | 0x800000u;
}

// a b c of non-negative table entries (a denormal one counts as zero)
ZK_HD WideFactor wide_product(float a, float b, float c) {
  int ea, eb, ec;
  const unsigned long long ma = float_mant(zk_float_bits(a), ea), mb = float_mant(zk_float_bits(b), eb),
                           mc = float_mant(zk_float_bits(c), ec);
  if (((ma & mb & mc) >> 23) == 0) return {0, 0};
  return {zk_mulhi((ma * mb) << 16, mc << 40), ea + eb + ec - 450 - 56 + 64};
}

// (x^2 + y^2) f 2^twice for finite x and y
ZK_HD WideFactor mode_weight(float x, float y, WideFactor f, int twice) {
  int ex, ey;
  const unsigned long long mx = float_mant(zk_float_bits(x), ex), my = float_mant(zk_float_bits(y), ey);
  const unsigned long long sx = (mx * mx) << 15, sy = (my * my) << 15;  // below 2^63
  const int d = ex - ey, e = d >= 0 ? ex : ey;
  const int cut = 2 * (d >= 0 ? d : -d);
  const unsigned long long s = (d >= 0 ? sx : sy) + (cut < 64 ? (d >= 0 ? sy : sx) >> cut : 0ULL);
  if (s == 0 || f.m == 0) return {0, 0};
  const int l = zk_clz(s);
  return {zk_mulhi(s << l, f.m), 2 * (e - 150) - 15 - l + f.e + 64 + twice};
}

// the least k with w < 2^k (w.m != 0)
ZK_HD int wide_ceil(WideFactor w) { return w.e + 64 - zk_clz(w.m); }

// w in units of 2^unit, rounded, for w < 2^(unit + 52)
ZK_HD unsigned long long wide_units(WideFactor w, int unit) {
  const int sh = unit - w.e;  // at least 8: w.m is 0 or at least 2^60
  if (w.m == 0 || sh > 64) return 0;
  return (sh == 64 ? 0ULL : w.m >> sh) + ((w.m >> (sh - 1)) & 1ULL);
}

}  // namespace zk
