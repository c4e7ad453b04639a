// Cell and in-cell offset of a coordinate and the fixed-point contributions of the assignment in integer
// arithmetic, and the contrast of a node in float32 pairs, for sm_103a.
//
// The float64 pipe of this part retires about two operations per SM and clock, so the float64
// formula (multiply, two floors, a division, three conversions per axis) costs more than the
// memory traffic of the kernels that need it.  The integer form below reproduces that formula bit
// for bit: a float32 coordinate is a 24-bit integer and 1/H a 53-bit one, so their product is a
// 77-bit integer whose rounding to 53 bits is the float64 product, whose upper bits are the cell
// and whose lower bits are the offset.  Measured on GB300, 16M particles: preparation of a sorted
// catalogue 1417 -> 209 us.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>
#ifdef __CUDACC__
#define ZK_HD __host__ __device__ __forceinline__
#else
#define ZK_HD inline
#endif

namespace zk {

// 1/H = n / box as the float64 value itself and as mant 2^exp with mant in [2^52, 2^53).
struct CellScale {
  double inv_h;
  unsigned long long mant;
  int exp;
};

inline CellScale make_cell_scale(int n, double box) {
  CellScale c;
  c.inv_h = n / box;
  unsigned long long b;
  std::memcpy(&b, &c.inv_h, sizeof b);
  const int e = static_cast<int>(b >> 52) & 0x7ff;
  c.mant = (b & 0xfffffffffffffULL) | 0x10000000000000ULL;
  c.exp = e - 1075;
  if (e == 0 || e == 0x7ff) c.mant = 0;  // denormal or infinite 1/H: the float64 formula alone
  return c;
}

ZK_HD uint32_t zk_float_bits(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  uint32_t b;
  std::memcpy(&b, &x, sizeof b);
  return b;
#endif
}
ZK_HD float zk_bits_float(uint32_t b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float x;
  std::memcpy(&x, &b, sizeof x);
  return x;
#endif
}
ZK_HD unsigned long long zk_mulhi(unsigned long long a, unsigned long long b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return static_cast<unsigned long long>((static_cast<unsigned __int128>(a) * b) >> 64);
#endif
}
ZK_HD int zk_clz(unsigned long long v) {
#ifdef __CUDA_ARCH__
  return __clzll(static_cast<long long>(v));
#else
  return v ? __builtin_clzll(v) : 64;
#endif
}

// floor(u) and float32(u - floor(u)) (at most the float below 1) for u = float64(x) * inv_h, when
// x is zero or a normal positive number with 2^-9 <= u < n; false (nothing written) otherwise.
ZK_HD bool cell_int(float x, const CellScale& c, int n, int& cell, float& t) {
  const uint32_t b = zk_float_bits(x);
  if (b == 0) {
    cell = 0;
    t = 0.f;
    return true;
  }
  const int ex = static_cast<int>(b >> 23);  // the sign is its bit 8
  if (ex == 0 || ex >= 255 || c.mant == 0) return false;
  const unsigned long long mx = (b & 0x7fffffu) | 0x800000u;
  const unsigned long long lo = mx * c.mant, hi = zk_mulhi(mx, c.mant);  // 76 or 77 bits
  const int s = 23 + static_cast<int>(hi >> 12);                          // bits below the 53
  unsigned long long q = (hi << (64 - s)) | (lo >> s);
  const unsigned long long rem = lo & ((1ULL << s) - 1), half = 1ULL << (s - 1);
  q += (rem > half || (rem == half && (q & 1))) ? 1 : 0;  // u = q 2^-f, round to nearest even
  const int f = -(ex - 150 + c.exp + s);
  if (f < 1 || f > 61) return false;
  const unsigned long long i = q >> f;
  if (i >= static_cast<unsigned long long>(n)) return false;
  cell = static_cast<int>(i);
  const unsigned long long fr = q & ((1ULL << f) - 1);
  if (fr == 0) {
    t = 0.f;
    return true;
  }
  const int top = 63 - zk_clz(fr);
  unsigned long long m;  // fr with its leading bit at bit 23, rounded to nearest even
  if (top <= 23) {
    m = fr << (23 - top);
  } else {
    const int d = top - 23;
    m = (fr + ((1ULL << (d - 1)) - 1) + ((fr >> d) & 1)) >> d;
  }
  // a carry to 2^24 moves into the exponent field
  const uint32_t tb = (static_cast<uint32_t>(127 + top - f) << 23) + (static_cast<uint32_t>(m) - 0x800000u);
  t = tb >= 0x3f800000u ? 0.99999994f : zk_bits_float(tb);
  return true;
}

// round(w b 2^k) as a 64-bit integer, ties to even, for finite w (not denormal) and b >= 0 or b < 0
// with |w b| 2^k < 2^62: the 48-bit product of the mantissas is exact, so this is the float64
// formula llrint((w 2^k) * b) bit for bit.
ZK_HD long long fix64_prod(float w, float b, int k) {
  const uint32_t wb = zk_float_bits(w), bb = zk_float_bits(b);
  const int ew = static_cast<int>((wb >> 23) & 0xffu), eb = static_cast<int>((bb >> 23) & 0xffu);
  if (ew == 0 || eb == 0) return 0;  // zero (or a denormal weight factor, far below half a unit)
  const unsigned long long p =
      static_cast<unsigned long long>((wb & 0x7fffffu) | 0x800000u) * ((bb & 0x7fffffu) | 0x800000u);
  const int sh = ew + eb - 300 + k;
  unsigned long long r;
  if (sh >= 0) {
    r = p << sh;
  } else if (sh <= -49) {
    r = 0;  // below half a unit
  } else {
    const int d = -sh;
    r = (p + ((1ULL << (d - 1)) - 1) + ((p >> d) & 1)) >> d;
  }
  const long long v = static_cast<long long>(r);
  return ((wb ^ bb) >> 31) ? -v : v;
}

// Float32 products and sums that are rounded where they stand: error-free transformations fail when the
// compiler fuses a product into the addition that uses it (its default), so every step of one goes
// through these.
ZK_HD float rn_mul(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  volatile float r = a * b;
  return r;
#endif
}
ZK_HD float rn_add(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fadd_rn(a, b);
#else
  volatile float r = a + b;
  return r;
#endif
}
ZK_HD float rn_fma(float a, float b, float c) {
#ifdef __CUDA_ARCH__
  return __fmaf_rn(a, b, c);
#else
  return std::fma(a, b, c);
#endif
}

// The contrast of a node in float64, one fused multiply-add rounded to float32.
ZK_HD float contrast_f64(long long v, double inv) {
#ifdef __CUDA_ARCH__
  return static_cast<float>(__fma_rn(static_cast<double>(v), inv, -1.0));
#else
  return static_cast<float>(std::fma(static_cast<double>(v), inv, -1.0));
#endif
}

// contrast_f64 off the float64 pipe, the same value: with inv = ih + il and v as the float32 values of its
// leading and following 24 bits, the product and the difference are float32 pairs within
// 2^-45 (|v inv| + 1); a result that close to a rounding boundary (one in 10^5, or any much smaller
// than 1) takes the float64 formula.  That formula for every node (three conversions, two operations) took
// 118 us for 256^3 nodes, bound by the float64 pipe; this 41 us.
ZK_HD float contrast_of(long long v, float ih, float il, double inv) {
  const bool neg = v < 0;
  const unsigned long long a = neg ? 0ULL - static_cast<unsigned long long>(v) : static_cast<unsigned long long>(v);
  if (a == 0) return -1.f;
  const int lz = zk_clz(a);
  const unsigned long long m = a << lz;
  const float sc = zk_bits_float(static_cast<uint32_t>(127 + 40 - lz) << 23);  // 2^(40 - lz)
  float hi = rn_mul(static_cast<float>(static_cast<uint32_t>(m >> 40)), sc);
  float lo = rn_mul(static_cast<float>(static_cast<uint32_t>(m >> 16) & 0xffffffu), rn_mul(sc, 5.9604644775390625e-8f));
  if (neg) {
    hi = -hi;
    lo = -lo;
  }
  const float p = rn_mul(hi, ih);
  const float e = rn_add(rn_fma(hi, ih, -p), rn_fma(hi, il, rn_mul(lo, ih)));
  const float s = rn_add(p, -1.f), bb = rn_add(s, -p);
  const float rest = rn_add(rn_add(rn_add(p, -rn_add(s, -bb)), rn_add(-1.f, -bb)), e);
  const float r = rn_add(s, rest);
  const float miss = fabsf(rn_add(rn_add(s, -r), rest));  // r is off by this much
  const float size = fabsf(p) + 1.f, tol = size * 5.684341886080802e-14f;  // 2^-44 (|p| + 1)
  const uint32_t rb = zk_float_bits(r);
  const float h = zk_bits_float((rb & 0x7f800000u) - (24u << 23));  // half a unit in the last place
  const bool near = fabsf(miss - h) < tol || ((rb & 0x7fffffu) == 0 && fabsf(miss - 0.5f * h) < tol);
  if (near || fabsf(r) < size * 2.44140625e-4f) return contrast_f64(v, inv);
  return r;
}

}  // namespace zk
