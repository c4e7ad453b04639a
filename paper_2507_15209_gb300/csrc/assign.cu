// MRA assignment of the catalogue and particle tiling, sm_103a.
//
// Assignment (Sec. 2.1 expansion n = sum eps phi; Fig. 1 step (2); contrast of Sec. 3):
//   eps_l = sum_p w_p phi(u_p - l), u = x / H, periodic in l, phi the centred B-spline of
//   order D or the genus-4 Daubechies function (tabulated); delta_l = eps_l / eps_bar - 1 with
//   eps_bar = W / N_g.
// Contributions are scattered as 64-bit fixed point (scale 2^k with k chosen from sum |w|
// so no cell can overflow), so the result does not depend on the order of the atomics.
// The cell and in-cell offset of each particle are those of the float64 formula, bit for bit (formed with
// integers, cell.cuh), so that a float32 position of a 512^3 grid keeps its full in-cell resolution.
//
// Tiling: particles are counted into 8x8x8-cell tiles, prefix-summed, scattered, and each
// tile's list is put back into original order, so particle-form sums are reproducible.
#include <mutex>

#include "cell.cuh"
#include "zeta_internal.h"

namespace zk {
namespace {

constexpr int kRedCtas = 1024;
// launch_assign groups the records by tile when the fixed-point grid is larger than L2 (8 n^3 bytes at
// n >= 256) and there are at least 2^24 contributions.  Measured, us per call, grouped / direct:
// 256^3 D = 4 with 0.01 and 0.12 particles a cell 171 / 156 and 456 / 697, D = 2 with 0.12 277 / 249;
// 512^3 D = 4 1069 / 1424 and 3525 / 11762, D = 2 799 / 702 and 2085 / 3182; 128^3 D = 4 with 0.12
// 116 / 83.
constexpr int kGroupMinN = 256;
constexpr int64_t kGroupMinContributions = 1LL << 24;

__device__ __forceinline__ bool finite4(float4 p) {
  return isfinite(p.x) && isfinite(p.y) && isfinite(p.z) && isfinite(p.w);
}

// The float64 formula: cell and in-cell offset of the coordinate x wrapped into the box.
__device__ __noinline__ int cell_f64(float x, double inv_h, int n, float& t) {
  double u = static_cast<double>(x) * inv_h;
  u -= floor(u / n) * n;
  int i = static_cast<int>(floor(u));
  double fr = u - i;
  if (i >= n) {
    i -= n;
  }
  if (i < 0) i += n;
  t = static_cast<float>(fr);
  if (t >= 1.0f) t = 0.99999994f;
  return i;
}

// grid coordinate wrapped into [0, n): returns cell (less shift, periodic) and in-cell offset t in
// [0, 1).  Coordinates inside the box take the integer form of the float64 formula (cell.cuh), the
// rest (negative, past the box, closer to 0 than 2^-9 cells) the formula itself.
__device__ __forceinline__ int cell_of(float x, const CellScale& cs, int n, int shift, float& t) {
  int i;
  if (!cell_int(x, cs, n, i, t)) i = cell_f64(x, cs.inv_h, n, t);
  i -= shift;
  if (i < 0) i += n;
  return i;
}

template <int D>
__device__ __forceinline__ void bspline_weights(float t, float* w) {
  if (D == 2) {
    w[0] = 1.f - t;
    w[1] = t;
  } else {
    const float t2 = t * t, t3 = t2 * t, s = 1.f - t;
    w[0] = s * s * s * (1.f / 6.f);
    w[1] = (3.f * t3 - 6.f * t2 + 4.f) * (1.f / 6.f);
    w[2] = (-3.f * t3 + 3.f * t2 + 3.f * t + 1.f) * (1.f / 6.f);
    w[3] = t3 * (1.f / 6.f);
  }
}

// Stencil weights of the basis: the B-spline of order D, or with a table (D = 4) the Daubechies
// function's.
template <int D>
__device__ __forceinline__ void stencil_weights(float t, const float* __restrict__ dtab, float* w) {
  if (D == 4 && dtab != nullptr)
    daub4_weights(t, dtab, w);
  else
    bspline_weights<D>(t, w);
}

// Sum of two float64 values over the 256 threads of a CTA (fixed butterfly, then the warps in order);
// the totals are valid in thread 0.
__device__ __forceinline__ void cta_sum2(double& a, double& b) {
  __shared__ double w1[8], w2[8];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, off);
    b += __shfl_xor_sync(0xffffffffu, b, off);
  }
  if ((threadIdx.x & 31) == 0) {
    w1[threadIdx.x >> 5] = a;
    w2[threadIdx.x >> 5] = b;
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int i = 1; i < 8; ++i) {
      a += w1[i];
      b += w2[i];
    }
}

// Per-CTA sums of w and |w| (the latter as sum w + 2 sum |negative w|: catalogues seldom have any, and
// the float64 pipe is what bounds this kernel).
__global__ void __launch_bounds__(256) k_weight_partials(const float4* __restrict__ p, long long np,
                                                         double* __restrict__ part, int* __restrict__ status) {
  double a = 0.0, b = 0.0;
  bool bad = false;
  constexpr int U = 4;  // loads in flight per thread
  const long long step = 256LL * gridDim.x;
  for (long long i = blockIdx.x * 256LL + threadIdx.x; i < np; i += U * step) {
    float4 q[U];
#pragma unroll
    for (int u = 0; u < U; ++u) q[u] = i + u * step < np ? p[i + u * step] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (!finite4(q[u])) {
        bad = true;
        continue;
      }
      a += q[u].w;
      if (q[u].w < 0.f) b -= 2.0 * q[u].w;
    }
  }
  if (bad) atomicOr(status, 1);
  b += a;
  cta_sum2(a, b);
  if (threadIdx.x == 0) {
    part[2 * blockIdx.x] = a;
    part[2 * blockIdx.x + 1] = b;
  }
}

// out[0] = W, out[1] = sum |w|, out[2] = fixed-point scale 2^k (sum |w| * 2^k < 2^62), out[4] = the factor
// N_g / (W 2^k) of the contrast and out[3] the same as a pair of float32 (NaN when the pair cannot hold it).
// One CTA: thread t adds the partials t, t + 256, ..., then the CTA adds its threads in a fixed order (one
// thread adding the 1024 partials in turn took 107 us, this 5 us).
__global__ void __launch_bounds__(256) k_weight_final(const double* __restrict__ part, int nparts, double ng,
                                                      double* __restrict__ out, double* __restrict__ wsum) {
  double a = 0.0, b = 0.0;
  for (int i = threadIdx.x; i < nparts; i += 256) {
    a += part[2 * i];
    b += part[2 * i + 1];
  }
  cta_sum2(a, b);
  if (threadIdx.x != 0) return;
  out[0] = a;
  out[1] = b;
  double scale = 1.0;
  if (b > 0.0) {
    int e;
    frexp(b, &e);  // b < 2^e
    scale = ldexp(1.0, 61 - e);
  }
  out[2] = scale;
  // the pair and its products stay normal numbers in this range (any catalogue but one of weights that
  // are denormal or cancel to W = 0 almost exactly)
  const double inv = (a != 0.0) ? ng / (a * scale) : 0.0;
  const double ai = fabs(inv);
  const float ih = static_cast<float>(inv);
  float2 f = make_float2(ih, static_cast<float>(inv - static_cast<double>(ih)));
  if (ai != 0.0 && !(ai > 1e-26 && ai < 1e18)) f.x = __int_as_float(0x7fc00000);
  *reinterpret_cast<float2*>(out + 3) = f;
  out[4] = inv;
  if (wsum) *wsum = a;
}

// The cell arithmetic of a particle (cell_of), done once per catalogue: cell (linear index
// z n^2 + y n + x), in-cell offsets t in [0, 1) and the weight (0 for a non-finite particle,
// which sits in cell 0 with t = 0 and so contributes nothing anywhere).
__device__ __forceinline__ void prep_one(float4 q, const CellScale& cs, int n, int shift, int& cell, float4& tq,
                                         int& tile) {
  const int nt = n / kTile;
  if (!finite4(q)) {
    cell = 0;
    tile = 0;
    tq = make_float4(0.f, 0.f, 0.f, 0.f);
    return;
  }
  float tx, ty, tz;
  const int cx = cell_of(q.x, cs, n, shift, tx), cy = cell_of(q.y, cs, n, shift, ty),
            cz = cell_of(q.z, cs, n, shift, tz);
  cell = (cz * n + cy) * n + cx;
  tile = ((cz / kTile) * nt + cy / kTile) * nt + cx / kTile;
  tq = make_float4(tx, ty, tz, q.w);
}

// The D^3 contributions of one prepared particle per group of D lanes, added to the fixed-point grid:
// lane ox of the group holds the nodes x = cx - OFF + ox of every row of the stencil.  w == 0: nothing.
template <int D>
__device__ __forceinline__ void scatter_rows(int cell, float4 q, int ox, int n, int lg, int k2, double scale,
                                             const float* __restrict__ dtab, unsigned long long* __restrict__ acc) {
  if (q.w == 0.f) return;
  constexpr int OFF = D / 2 - 1;
  const int mask = n - 1;
  const bool tiny = fabsf(q.w) < 1.17549435e-38f;  // a denormal weight takes the float64 formula
  float wx[D], wy[D], wz[D];
  stencil_weights<D>(q.x, dtab, wx);
  stencil_weights<D>(q.y, dtab, wy);
  stencil_weights<D>(q.z, dtab, wz);
  float wxo = wx[0];
#pragma unroll
  for (int o = 1; o < D; ++o) wxo = ox == o ? wx[o] : wxo;
  const int cx = cell & mask, cy = (cell >> lg) & mask, cz = cell >> (2 * lg);
  const int lx = (cx - OFF + ox) & mask;
#pragma unroll
  for (int oz = 0; oz < D; ++oz) {
    const int lz = (cz - OFF + oz) & mask;
#pragma unroll
    for (int oy = 0; oy < D; ++oy) {
      const int ly = (cy - OFF + oy) & mask;
      const float b = wz[oz] * wy[oy] * wxo;
      const long long v = tiny ? __double2ll_rn(static_cast<double>(q.w) * scale * static_cast<double>(b))
                               : fix64_prod(q.w, b, k2);
      atomicAdd(acc + ((((lz << lg) + ly) << lg) + lx), static_cast<unsigned long long>(v));
    }
  }
}

// Scatter of the catalogue into the 64-bit fixed-point grid (order-free integer sums).  D neighbouring
// lanes hold the D nodes of one particle's stencil row, so that one atomic instruction covers 32 / D
// rows of D x 8 contiguous bytes and the L2 sees a few whole sectors instead of 32 scattered words, and
// the contribution round(w beta 2^k) is formed with integers (fix64_prod), not on the float64 pipe.
//
// k_assign_records: the particles come grouped by tile as prepared (cell, t) records, so the rows in
// flight share cache lines.  Bound: L1 (81 % busy with the atomics), then issue (73 %) and L2 (66 %).  256^3, 2M
// particles, D = 4: 255 us (one CTA per tile walking the 27 neighbour tiles' particles into shared memory:
// 1825 us).
template <int D>
__global__ void __launch_bounds__(256) k_assign_records(const float4* __restrict__ s_tq,
                                                        const int* __restrict__ s_cell, long long np, int n,
                                                        const float* __restrict__ dtab,
                                                        const double* __restrict__ wstat,
                                                        unsigned long long* __restrict__ acc) {
  const double scale = wstat[2];
  const int k2 = ilogb(scale);
  const int lg = __ffs(n) - 1;
  const int ox = threadIdx.x % D;
  for (long long i = (blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x) / D; i < np;
       i += static_cast<long long>(blockDim.x) * gridDim.x / D)
    scatter_rows<D>(s_cell[i], s_tq[i], ox, n, lg, k2, scale, dtab, acc);
}

// k_assign_scatter: particles in any order; a warp prepares 32 of them (one per lane), then takes 32 / D
// at a time.  Same case: 596 us (one thread per particle with float64 rounding: 938 us).
template <int D>
__global__ void __launch_bounds__(256) k_assign_scatter(const float4* __restrict__ p, long long np, int n,
                                                        CellScale cs, int shift, const float* __restrict__ dtab,
                                                        const double* __restrict__ wstat,
                                                        unsigned long long* __restrict__ acc) {
  const double scale = wstat[2];
  const int k2 = ilogb(scale);
  const int lg = __ffs(n) - 1;
  const int lane = threadIdx.x & 31;
  const long long nwarp = (static_cast<long long>(blockDim.x) * gridDim.x) >> 5;
  for (long long base = ((blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x) >> 5) * 32; base < np;
       base += nwarp * 32) {
    int mycell = 0, tile;
    float4 my = make_float4(0.f, 0.f, 0.f, 0.f);
    if (base + lane < np) prep_one(p[base + lane], cs, n, shift, mycell, my, tile);
#pragma unroll 1
    for (int r = 0; r < D; ++r) {
      const int src = r * (32 / D) + lane / D;
      const int cell = __shfl_sync(0xffffffffu, mycell, src);
      const float4 q = make_float4(__shfl_sync(0xffffffffu, my.x, src), __shfl_sync(0xffffffffu, my.y, src),
                                   __shfl_sync(0xffffffffu, my.z, src), __shfl_sync(0xffffffffu, my.w, src));
      scatter_rows<D>(cell, q, lane % D, n, lg, k2, scale, dtab, acc);
    }
  }
}

__global__ void k_assign_finalize(const unsigned long long* __restrict__ acc, long long ng,
                                  const double* __restrict__ wstat, float* __restrict__ delta) {
  const float2 f = *reinterpret_cast<const float2*>(wstat + 3);
  const bool pair = !isnan(f.x);
  const double inv = wstat[4];
  for (long long i = (blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x) * 2; i < ng;
       i += static_cast<long long>(blockDim.x) * gridDim.x * 2) {  // ng is even, acc 16-byte aligned
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(acc + i);
    const long long v0 = static_cast<long long>(v.x), v1 = static_cast<long long>(v.y);
    float d0, d1;
    if (pair) {
      d0 = contrast_of(v0, f.x, f.y, inv);
      d1 = contrast_of(v1, f.x, f.y, inv);
    } else {
      d0 = contrast_f64(v0, inv);
      d1 = contrast_f64(v1, inv);
    }
    delta[i] = d0;
    delta[i + 1] = d1;
  }
}

__device__ __forceinline__ long long tile_of(float4 q, const CellScale& cs, int n, int shift) {
  float t;
  const int nt = n / kTile;
  if (!finite4(q)) return 0;
  const int cx = cell_of(q.x, cs, n, shift, t) / kTile;
  const int cy = cell_of(q.y, cs, n, shift, t) / kTile;
  const int cz = cell_of(q.z, cs, n, shift, t) / kTile;
  return (static_cast<long long>(cz) * nt + cy) * nt + cx;
}

__global__ void k_tile_count(const float4* __restrict__ p, long long np, int n, CellScale cs, int shift,
                             int* __restrict__ cnt) {
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < np;
       i += static_cast<long long>(blockDim.x) * gridDim.x)
    atomicAdd(cnt + tile_of(p[i], cs, n, shift), 1);
}

// Exclusive prefix sum of cnt[0..m) into start[0..m] (start[m] = total, at most 2^31 - 1) with one CTA of
// 1024 threads, eight counts per thread and step (warp shuffles, then the 32 warp totals), the next
// step's counts loaded ahead; cnt is reset to zero so it can serve as the scatter cursor.  m is a
// power of eight, so a thread's eight counts are all in range when its first is.
__global__ void __launch_bounds__(1024) k_tile_scan(int* __restrict__ cnt, long long m, long long* __restrict__ start) {
  __shared__ int wtot[2][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int carry = 0, par = 0;
  int4 a = make_int4(0, 0, 0, 0), b = a;
  auto fetch = [&](long long i) {
    a = make_int4(0, 0, 0, 0);
    b = a;
    if (i < m) {
      int4* c4 = reinterpret_cast<int4*>(cnt + i);
      a = c4[0];
      b = c4[1];
      c4[0] = make_int4(0, 0, 0, 0);
      c4[1] = make_int4(0, 0, 0, 0);
    }
  };
  fetch(8 * threadIdx.x);
  for (long long base = 0; base < m; base += 8192, par ^= 1) {
    const long long i = base + 8 * threadIdx.x;
    const int v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    fetch(i + 8192);
    int mine = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) mine += v[j];
    int inc = mine;  // inclusive over the warp
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, inc, off);
      if (lane >= off) inc += o;
    }
    if (lane == 31) wtot[par][warp] = inc;
    __syncthreads();  // the other buffer's readers are past it one step later
    const int t = wtot[par][lane];
    int pre = t;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, pre, off);
      if (lane >= off) pre += o;
    }
    const int before = __shfl_sync(0xffffffffu, pre - t, warp);
    const int total = __shfl_sync(0xffffffffu, pre, 31);
    if (i < m) {
      int run = carry + before + inc - mine;
      longlong2* o = reinterpret_cast<longlong2*>(start + i);  // a caller's array may be 8-byte aligned only
      const bool al = (reinterpret_cast<uintptr_t>(start) & 15) == 0;
#pragma unroll
      for (int j = 0; j < 8; j += 2) {
        if (al) {
          o[j / 2] = make_longlong2(run, run + v[j]);
        } else {
          start[i + j] = run;
          start[i + j + 1] = run + v[j];
        }
        run += v[j] + v[j + 1];
      }
    }
    carry += total;
  }
  if (threadIdx.x == 0) start[m] = carry;
}

__global__ void k_tile_scatter(const float4* __restrict__ p, long long np, int n, CellScale cs, int shift,
                               const long long* __restrict__ start, int* __restrict__ cursor,
                               int* __restrict__ orig) {
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < np;
       i += static_cast<long long>(blockDim.x) * gridDim.x) {
    const long long t = tile_of(p[i], cs, n, shift);
    const int slot = atomicAdd(cursor + t, 1);
    orig[start[t] + slot] = static_cast<int>(i);
  }
}

// Prepared records grouped by tile, in any order within a tile (for the order-free assignment).
__global__ void k_tile_records(const float4* __restrict__ p, long long np, int n, CellScale cs, int shift,
                               const long long* __restrict__ start, int* __restrict__ cursor,
                               int* __restrict__ r_cell, float4* __restrict__ r_tq) {
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < np;
       i += static_cast<long long>(blockDim.x) * gridDim.x) {
    int cell, tile;
    float4 tq;
    prep_one(p[i], cs, n, shift, cell, tq, tile);
    const long long at = start[tile] + atomicAdd(cursor + tile, 1);
    r_cell[at] = cell;
    r_tq[at] = tq;
  }
}

// One warp per tile: rank every entry by its original index and gather the particles (and,
// when given, their prepared cell and offsets).
__global__ void k_tile_order(const float4* __restrict__ p, const long long* __restrict__ start, long long ntiles,
                             const int* __restrict__ orig, float4* __restrict__ sorted, int* __restrict__ sorted_idx,
                             const int* __restrict__ o_cell, const float4* __restrict__ o_tq, int* __restrict__ s_cell,
                             float4* __restrict__ s_tq) {
  const long long warp = (blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (warp >= ntiles) return;
  const long long s = start[warp], e = start[warp + 1];
  const int c = static_cast<int>(e - s);
  for (int i = lane; i < c; i += 32) {
    const int v = orig[s + i];
    int rank = 0;
    for (int j = 0; j < c; ++j) rank += (orig[s + j] < v);
    sorted[s + rank] = p[v];
    if (sorted_idx) sorted_idx[s + rank] = v;
    if (s_cell) {
      s_cell[s + rank] = o_cell[v];
      s_tq[s + rank] = o_tq[v];
    }
  }
}

// Prepared data in the original order and the particle count of every tile.
__global__ void k_particle_prep(const float4* __restrict__ p, long long np, int n, CellScale cs, int shift,
                                int* __restrict__ o_tile, int* __restrict__ o_cell, float4* __restrict__ o_tq,
                                int* __restrict__ cnt) {
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < np;
       i += static_cast<long long>(blockDim.x) * gridDim.x) {
    int cell, tile;
    float4 tq;
    prep_one(p[i], cs, n, shift, cell, tq, tile);
    o_tile[i] = tile;
    o_cell[i] = cell;
    o_tq[i] = tq;
    atomicAdd(cnt + tile, 1);
  }
}

__global__ void k_tile_scatter_pre(const int* __restrict__ o_tile, long long np, const long long* __restrict__ start,
                                   int* __restrict__ cursor, int* __restrict__ orig) {
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < np;
       i += static_cast<long long>(blockDim.x) * gridDim.x) {
    const int t = o_tile[i];
    const int slot = atomicAdd(cursor + t, 1);
    orig[start[t] + slot] = static_cast<int>(i);
  }
}

// Prepared data of particles that are already sorted (a caller's sorted array).
__global__ void k_prep_sorted(const float4* __restrict__ sorted, long long np, int n, CellScale cs, int shift,
                              int* __restrict__ s_cell, float4* __restrict__ s_tq) {
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < np;
       i += static_cast<long long>(blockDim.x) * gridDim.x) {
    int cell, tile;
    float4 tq;
    prep_one(sorted[i], cs, n, shift, cell, tq, tile);
    s_cell[i] = cell;
    s_tq[i] = tq;
  }
}

inline int grid_for(long long work, int threads, int sms) {
  long long g = (work + threads - 1) / threads;
  const long long cap = static_cast<long long>(sms) * 32;
  if (g > cap) g = cap;
  if (g < 1) g = 1;
  return static_cast<int>(g);
}

}  // namespace

namespace {

// acc and the contrast from prepared records
int assign_records(const zeta_ctx* c, const float4* tq, const int* cell, int64_t np, unsigned long long* acc,
                   const double* wstat, float* delta, cudaStream_t s) {
  const int g = grid_for(np * (c->p.dsup == 2 ? 2 : 4), 256, c->num_sms);
  if (c->p.dsup == 2)
    k_assign_records<2><<<g, 256, 0, s>>>(tq, cell, np, c->n, nullptr, wstat, acc);
  else
    k_assign_records<4><<<g, 256, 0, s>>>(tq, cell, np, c->n, c->d_daub, wstat, acc);
  k_assign_finalize<<<grid_for(c->ng / 2, 256, c->num_sms), 256, 0, s>>>(acc, c->ng, wstat, delta);
  return cudaGetLastError() == cudaSuccess ? ZETA_OK : ZETA_ECUDA;
}

}  // namespace

int launch_assign(const zeta_ctx* c, const float4* parts, int64_t np, float* delta, double* wsum,
                  const AssignScratch& a, cudaStream_t s) {
  // a.small: 2*kRedCtas partials then 5 values (k_weight_final)
  double* wstat = a.small + 2 * kRedCtas;
  const CellScale cs = make_cell_scale(c->n, c->p.box);
  const int g = grid_for(np, 256, c->num_sms);
  const int64_t contributions = np * (c->p.dsup == 2 ? 8 : 64);
  const bool group = c->n >= kGroupMinN && contributions >= kGroupMinContributions &&
                     a.tq_bytes >= sizeof(float4) * static_cast<size_t>(np) &&
                     a.cell_bytes >= sizeof(int) * static_cast<size_t>(np);
  StageScope prof(c, ST_ASSIGN, group ? 7 : 4, s);
  k_weight_partials<<<kRedCtas, 256, 0, s>>>(parts, np, a.small, c->d_status);
  k_weight_final<<<1, 256, 0, s>>>(a.small, kRedCtas, static_cast<double>(c->ng), wstat, wsum);
  if (cudaMemsetAsync(a.acc, 0, sizeof(unsigned long long) * c->ng, s) != cudaSuccess) return ZETA_ECUDA;
  if (group) {
    long long* st = reinterpret_cast<long long*>(a.tile_start);
    if (cudaMemsetAsync(a.counts, 0, sizeof(int) * c->ntiles, s) != cudaSuccess) return ZETA_ECUDA;
    k_tile_count<<<g, 256, 0, s>>>(parts, np, c->n, cs, cell_shift(c), a.counts);
    k_tile_scan<<<1, 1024, 0, s>>>(a.counts, c->ntiles, st);
    k_tile_records<<<g, 256, 0, s>>>(parts, np, c->n, cs, cell_shift(c), st, a.counts, a.cell, a.tq);
    return assign_records(c, a.tq, a.cell, np, a.acc, wstat, delta, s);
  }
  if (c->p.dsup == 2)
    k_assign_scatter<2><<<g, 256, 0, s>>>(parts, np, c->n, cs, 0, nullptr, wstat, a.acc);
  else
    k_assign_scatter<4><<<g, 256, 0, s>>>(parts, np, c->n, cs, cell_shift(c), c->d_daub, wstat, a.acc);
  k_assign_finalize<<<grid_for(c->ng / 2, 256, c->num_sms), 256, 0, s>>>(a.acc, c->ng, wstat, delta);
  return cudaGetLastError() == cudaSuccess ? ZETA_OK : ZETA_ECUDA;
}

int launch_wsum(const zeta_ctx* c, const float4* parts, int64_t np, double* wsum, double* scratch, cudaStream_t s) {
  StageScope prof(c, ST_ASSIGN, 2, s);
  double* wstat = scratch + 2 * kRedCtas;
  k_weight_partials<<<kRedCtas, 256, 0, s>>>(parts, np, scratch, c->d_status);
  k_weight_final<<<1, 256, 0, s>>>(scratch, kRedCtas, static_cast<double>(c->ng), wstat, wsum);
  return cudaGetLastError() == cudaSuccess ? ZETA_OK : ZETA_ECUDA;
}

int launch_sort(const zeta_ctx* c, const float4* parts, int64_t np, float4* sorted, int64_t* tile_start,
                int* counts, int* orig, cudaStream_t s, int* sorted_idx, const PartPrep* prep) {
  StageScope prof(c, ST_SORT, 4, s);
  const CellScale cs = make_cell_scale(c->n, c->p.box);
  if (cudaMemsetAsync(counts, 0, sizeof(int) * c->ntiles, s) != cudaSuccess) return ZETA_ECUDA;
  const int g = grid_for(np, 256, c->num_sms);
  long long* st = reinterpret_cast<long long*>(tile_start);
  if (prep) {
    k_particle_prep<<<g, 256, 0, s>>>(parts, np, c->n, cs, cell_shift(c), prep->o_tile, prep->o_cell, prep->o_tq,
                                      counts);
    k_tile_scan<<<1, 1024, 0, s>>>(counts, c->ntiles, st);
    k_tile_scatter_pre<<<g, 256, 0, s>>>(prep->o_tile, np, st, counts, orig);
  } else {
    k_tile_count<<<g, 256, 0, s>>>(parts, np, c->n, cs, cell_shift(c), counts);
    k_tile_scan<<<1, 1024, 0, s>>>(counts, c->ntiles, st);
    k_tile_scatter<<<g, 256, 0, s>>>(parts, np, c->n, cs, cell_shift(c), st, counts, orig);
  }
  const long long warps = c->ntiles;
  k_tile_order<<<static_cast<unsigned>((warps * 32 + 255) / 256), 256, 0, s>>>(
      parts, st, c->ntiles, orig, sorted, sorted_idx, prep ? prep->o_cell : nullptr, prep ? prep->o_tq : nullptr,
      prep ? prep->s_cell : nullptr, prep ? prep->s_tq : nullptr);
  return cudaGetLastError() == cudaSuccess ? ZETA_OK : ZETA_ECUDA;
}

// Szapudi-Szalay fields from the two contrasts: a = delta_D - delta_R (in place of delta_D) and
// r = 1 + delta_R (in place of delta_R).
__global__ void k_ss_fields(float* __restrict__ a, float* __restrict__ r, long long ng) {
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < ng;
       i += static_cast<long long>(blockDim.x) * gridDim.x) {
    const float dr = r[i];
    a[i] = a[i] - dr;
    r[i] = 1.0f + dr;
  }
}

int launch_ss_fields(const zeta_ctx* c, float* data_delta, float* rand_delta, cudaStream_t s) {
  StageScope prof(c, ST_ASSIGN, 1, s);
  k_ss_fields<<<grid_for(c->ng, 256, c->num_sms), 256, 0, s>>>(data_delta, rand_delta, c->ng);
  return cudaGetLastError() == cudaSuccess ? ZETA_OK : ZETA_ECUDA;
}

int launch_prep_sorted(const zeta_ctx* c, const float4* sorted, int64_t np, int* s_cell, float4* s_tq, cudaStream_t s) {
  StageScope prof(c, ST_SORT, 1, s);
  k_prep_sorted<<<grid_for(np, 256, c->num_sms), 256, 0, s>>>(sorted, np, c->n, make_cell_scale(c->n, c->p.box), cell_shift(c),
                                                              s_cell, s_tq);
  return cudaGetLastError() == cudaSuccess ? ZETA_OK : ZETA_ECUDA;
}

int launch_assign_sorted(const zeta_ctx* c, const float4* parts, int64_t np, const int* s_cell, const float4* s_tq,
                         float* delta, double* wsum, unsigned long long* acc, double* small, cudaStream_t s) {
  StageScope prof(c, ST_ASSIGN, 4, s);
  double* wstat = small + 2 * kRedCtas;
  k_weight_partials<<<kRedCtas, 256, 0, s>>>(parts, np, small, c->d_status);
  k_weight_final<<<1, 256, 0, s>>>(small, kRedCtas, static_cast<double>(c->ng), wstat, wsum);
  if (cudaMemsetAsync(acc, 0, sizeof(unsigned long long) * c->ng, s) != cudaSuccess) return ZETA_ECUDA;
  return assign_records(c, s_tq, s_cell, np, acc, wstat, delta, s);
}

}  // namespace zk

// ---------------------------------------------------------------------------------------
// Assignment without any allocation, for callers that cannot allocate device memory when
// they call: code inside a host framework whose memory pool already owns the device (a raw
// allocation would fail or fragment that pool), latency-critical loops that cannot afford
// the implicit synchronisation of an allocation, and services that must not hit an
// out-of-memory error once they are up.  Its scratch lives in a fixed array that every GPU
// which loads this library holds until the process exits.
namespace zk {
namespace {

constexpr int kStaticMaxN = 128;  // largest grid side the fixed scratch can hold
constexpr long long kStaticAcc = static_cast<long long>(kStaticMaxN) * kStaticMaxN * kStaticMaxN;
// layout (64-bit words): [fixed-point grid kStaticAcc][reduction partials 2*kRedCtas]
//                        [the 5 values of k_weight_final, spare][status word]
constexpr long long kStaticWords = kStaticAcc + 2 * kRedCtas + 6 + 1;

static __device__ __align__(256) unsigned long long g_assign_scratch[kStaticWords];

// A non-finite particle latched the status word: make the whole result NaN, so that the
// caller sees the bad input in the output itself (this entry point has no context to report
// through and does not synchronise).
__global__ void k_poison_if_bad(const int* __restrict__ status, float* __restrict__ delta, long long ng,
                                double* __restrict__ wsum) {
  if (*status == 0) return;
  const float qnan = __int_as_float(0x7fc00000);
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < ng;
       i += static_cast<long long>(blockDim.x) * gridDim.x)
    delta[i] = qnan;
  if (wsum && blockIdx.x == 0 && threadIdx.x == 0) *wsum = __longlong_as_double(0x7ff8000000000000LL);
}

constexpr int kMaxDevices = 64;
std::mutex g_static_mu;
unsigned long long* g_static_ptr[kMaxDevices] = {};

// Device address of the fixed scratch on the current device, looked up once per device.
int static_scratch(unsigned long long** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return ZETA_ECUDA;
  std::lock_guard<std::mutex> lock(g_static_mu);
  if (!g_static_ptr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_assign_scratch) != cudaSuccess || !p) return ZETA_ECUDA;
    g_static_ptr[dev] = static_cast<unsigned long long*>(p);
  }
  *out = g_static_ptr[dev];
  return ZETA_OK;
}

}  // namespace
}  // namespace zk

extern "C" int zeta_assign_noalloc(int n, double box, int dsup, const float* particles, int64_t np, float* delta,
                                   double* wsum, zeta_stream stream) {
  using namespace zk;
  if (n < 16 || n > kStaticMaxN || (n & (n - 1)) || !(box > 0) || (dsup != 2 && dsup != 4)) return ZETA_EINVAL;
  if (!particles || np < 1 || np > 0x7fffffffLL || !delta) return ZETA_EINVAL;
  unsigned long long* base = nullptr;
  if (static_scratch(&base) != ZETA_OK) return ZETA_ECUDA;
  const long long ng = static_cast<long long>(n) * n * n;
  unsigned long long* acc = base;
  double* part = reinterpret_cast<double*>(base + kStaticAcc);
  double* wstat = part + 2 * kRedCtas;
  int* status = reinterpret_cast<int*>(base + kStaticAcc + 2 * kRedCtas + 6);
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return ZETA_ECUDA;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 1;
  cudaStream_t s = stream;
  const float4* p = reinterpret_cast<const float4*>(particles);
  if (cudaMemsetAsync(status, 0, sizeof(int), s) != cudaSuccess) return ZETA_ECUDA;
  k_weight_partials<<<kRedCtas, 256, 0, s>>>(p, np, part, status);
  k_weight_final<<<1, 256, 0, s>>>(part, kRedCtas, static_cast<double>(ng), wstat, wsum);
  if (cudaMemsetAsync(acc, 0, sizeof(unsigned long long) * ng, s) != cudaSuccess) return ZETA_ECUDA;
  const CellScale cs = make_cell_scale(n, box);
  const int g = grid_for(np, 256, sms);
  if (dsup == 2)
    k_assign_scatter<2><<<g, 256, 0, s>>>(p, np, n, cs, 0, nullptr, wstat, acc);
  else
    k_assign_scatter<4><<<g, 256, 0, s>>>(p, np, n, cs, 0, nullptr, wstat, acc);
  k_assign_finalize<<<grid_for(ng / 2, 256, sms), 256, 0, s>>>(acc, ng, wstat, delta);
  k_poison_if_bad<<<grid_for(ng, 256, sms), 256, 0, s>>>(status, delta, ng, wsum);
  return cudaGetLastError() == cudaSuccess ? ZETA_OK : ZETA_ECUDA;
}

