// Adjoint (reverse-mode) kernels for gradients of a scalar loss L = sum_l sum_ij W_l[i,j]
// zeta_l[i,j] (field-level inference).  With S_l = (W_l + W_l^T)/2 and the reconstruction
// a_b = A_b delta, A_b = IDFT diag(K_b) DFT, the transpose is A_b^T = (-1)^l IDFT diag(K_b) DFT,
// so every (l, m) adds (-1)^l sum_b K_b DFT(h_b) to one k-space accumulator that is transformed
// back once at the end (fft.cu: launch_adj_spectral, launch_c2r_inplace).
//   node form:      q += sum S a a,  h_b = 2 delta (S a)_b          dL/d delta = (q + IDFT)/N_g
//   particle form:  per particle c_b = (2 w_p / W)(S f)_b; the direct term sum_b c_b grad f_b;
//                   h_b = assignment of c_b;  the mass term's share -2 Mhat delta_hat c_l(k) in
//                   k-space; dL/dx_p = direct + (N_g w_p / W) grad(interpolated dL/d delta).
// The particle scatter uses float atomics, so those gradients are reproducible only to float32
// rounding; everything else is order-fixed.
#include "cell.cuh"
#include "zeta_internal.h"

namespace zk {
namespace {

constexpr int kAT = 256;

template <int D>
__device__ __forceinline__ void bs_w(float t, float* w, float* dw) {
  if (D == 2) {
    w[0] = 1.f - t;
    w[1] = t;
    dw[0] = -1.f;
    dw[1] = 1.f;
  } else {
    const float t2 = t * t, t3 = t2 * t, s = 1.f - t;
    w[0] = s * s * s * (1.f / 6.f);
    w[1] = (3.f * t3 - 6.f * t2 + 4.f) * (1.f / 6.f);
    w[2] = (-3.f * t3 + 3.f * t2 + 3.f * t + 1.f) * (1.f / 6.f);
    w[3] = t3 * (1.f / 6.f);
    dw[0] = -0.5f * s * s;
    dw[1] = 1.5f * t2 - 2.f * t;
    dw[2] = -1.5f * t2 + t + 0.5f;
    dw[3] = 0.5f * t2;
  }
}

// The float64 formula of a coordinate's cell and offset, for what the integer form does not take (cell.cuh).
__device__ __noinline__ int cell_f64(float x, double inv_h, int n, float& t) {
  const double u = static_cast<double>(x) * inv_h;
  const double v = u - floor(u / n) * n;
  int c = static_cast<int>(floor(v));
  const double fr = v - c;
  if (c >= n) c -= n;
  t = static_cast<float>(fr);
  if (t >= 1.f) t = 0.99999994f;
  return c;
}
__device__ __forceinline__ int cell_t(float x, const CellScale& cs, int n, float& t) {
  int c;
  return cell_int(x, cs, n, c, t) ? c : cell_f64(x, cs.inv_h, n, t);
}

// q += sum S a a and the fields replaced by h = 2 delta S a, two points per thread so that each float4 of S
// read from shared memory serves eight multiply-adds.  The loop over the groups of h is rolled (unrolled, S
// fills the registers and spills).  Bound: HBM, the fields read once and written once.  256^3, us, with 8, 10,
// 16, 20, 28 and 32 bins: 203, 278, 418, 470, 772, 914 (one point per thread, both loops unrolled: 330, 703,
// 745, 934, 1348, 1374; each group's values read a second time, which missed L1: 306, 546, 745, 978, 1408, 902).
template <int NBP>
__global__ void __launch_bounds__(kAT) k_adj_node(const float* __restrict__ delta, float4* __restrict__ f4, long long ng,
                                                  int nb, const float* __restrict__ S, float* __restrict__ q) {
  constexpr int G = NBP / 4, P = 2;
  __shared__ __align__(16) float s_s[NBP * NBP];
  for (int i = threadIdx.x; i < NBP * NBP; i += blockDim.x) {
    const int r = i / NBP, c = i % NBP;
    s_s[i] = (r < nb && c < nb) ? S[r * nb + c] : 0.f;
  }
  __syncthreads();
  // ng is a multiple of P kAT (n >= 16)
  for (long long i0 = blockIdx.x * static_cast<long long>(P * kAT) + threadIdx.x; i0 < ng;
       i0 += static_cast<long long>(P * kAT) * gridDim.x) {
    float a[P][NBP], d[P], qs[P];
#pragma unroll
    for (int u = 0; u < P; ++u) {
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const float4 v = f4[g * ng + i0 + u * kAT];
        a[u][4 * g] = v.x;
        a[u][4 * g + 1] = v.y;
        a[u][4 * g + 2] = v.z;
        a[u][4 * g + 3] = v.w;
      }
      d[u] = 2.f * delta[i0 + u * kAT];
      qs[u] = 0.f;
    }
#pragma unroll 1
    for (int g = 0; g < G; ++g) {
      float h[P][4];
      float4 own[P];  // this group's values, by selects (a is indexed by constants only)
#pragma unroll
      for (int u = 0; u < P; ++u) {
        own[u] = make_float4(a[u][0], a[u][1], a[u][2], a[u][3]);
#pragma unroll
        for (int g2 = 1; g2 < G; ++g2)
          if (g == g2) own[u] = make_float4(a[u][4 * g2], a[u][4 * g2 + 1], a[u][4 * g2 + 2], a[u][4 * g2 + 3]);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int b = 4 * g + j;
        float t[P];
#pragma unroll
        for (int u = 0; u < P; ++u) t[u] = 0.f;
#pragma unroll
        for (int g2 = 0; g2 < G; ++g2) {
          const float4 sv = *reinterpret_cast<const float4*>(s_s + b * NBP + 4 * g2);
#pragma unroll
          for (int u = 0; u < P; ++u) {
            t[u] = fmaf(sv.x, a[u][4 * g2], t[u]);
            t[u] = fmaf(sv.y, a[u][4 * g2 + 1], t[u]);
            t[u] = fmaf(sv.z, a[u][4 * g2 + 2], t[u]);
            t[u] = fmaf(sv.w, a[u][4 * g2 + 3], t[u]);
          }
        }
#pragma unroll
        for (int u = 0; u < P; ++u) {
          qs[u] = fmaf(j == 0 ? own[u].x : j == 1 ? own[u].y : j == 2 ? own[u].z : own[u].w, t[u], qs[u]);
          h[u][j] = d[u] * t[u];
        }
      }
#pragma unroll
      for (int u = 0; u < P; ++u) f4[g * ng + i0 + u * kAT] = make_float4(h[u][0], h[u][1], h[u][2], h[u][3]);
    }
#pragma unroll
    for (int u = 0; u < P; ++u) q[i0 + u * kAT] += qs[u];
  }
}

// The uniform term's share of gk: gk(n) -= 2 Mhat(n) delta_hat(n) sum_l (2l+1)/(4 pi) sum_bb' S_l[b,b'] T_lb(n)
// T_lb'(n) over the non-Nyquist modes.  The sum over l and bins depends on the mode only through |n|^2, so it
// is formed once per value of |n|^2 and the modes are visited once (256^3, 7 multipoles, 10 bins:
// 7 x 2179 us with the sums per mode and multipole, 56 us in all now).
__global__ void __launch_bounds__(kAT) k_adj_mass_table(const float* __restrict__ jt, long long nn2, int nbp, int nb,
                                                        int lmax, const float* __restrict__ S, float* __restrict__ tab) {
  extern __shared__ float s_s[];  // [lmax + 1][nb][nb]
  for (int i = threadIdx.x; i < (lmax + 1) * nb * nb; i += blockDim.x) s_s[i] = S[i];
  __syncthreads();
  const long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if (i >= nn2) return;
  float sum = 0.f;
  for (int l = 0; l <= lmax; ++l) {
    const float* t = jt + (l * nn2 + i) * nbp;
    const float* sl = s_s + l * nb * nb;
    float c = 0.f;
    for (int b = 0; b < nb; ++b) {
      float r = 0.f;
      for (int b2 = 0; b2 < nb; ++b2) r = fmaf(sl[b * nb + b2], __ldg(t + b2), r);
      c = fmaf(__ldg(t + b), r, c);
    }
    sum = fmaf(2.f * (2.f * l + 1.f) / 12.566370614359172f, c, sum);
  }
  tab[i] = sum;
}

__global__ void __launch_bounds__(kAT) k_adj_mass(const float2* __restrict__ dhat, const float* __restrict__ tab,
                                                  const float* __restrict__ mhat, int n, float2* __restrict__ gk) {
  const int nc = n / 2;
  const long long total = static_cast<long long>(n) * n * nc;
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < total;
       i += static_cast<long long>(blockDim.x) * gridDim.x) {
    const int ix = static_cast<int>(i % nc), iy = static_cast<int>((i / nc) % n),
              iz = static_cast<int>(i / (static_cast<long long>(nc) * n));
    if (iy == n / 2 || iz == n / 2) continue;
    const int fy = iy < n / 2 ? iy : iy - n, fz = iz < n / 2 ? iz : iz - n;
    const float f = __ldg(tab + (ix * ix + fy * fy + fz * fz)) * (mhat[ix] * mhat[iy] * mhat[iz]);
    const float2 d = dhat[i], g = gk[i];
    gk[i] = make_float2(g.x - f * d.x, g.y - f * d.y);
  }
}

// Particle adjoint.  A warp takes eight particles of the tile-sorted catalogue, four lanes each, and keeps
// everything in registers, without a barrier: the lanes of a particle hold the four nodes along x of every
// stencil row (D = 4; for D = 2 the four nodes of a z-layer), so a gather and an atomic of a row each cover
// 64 contiguous bytes.  Per bin group the lanes sum w v and the parts of its gradient over their nodes, then
// reduce-scatter: lane i holds f and grad f of bin 4 g + i.  c = (2 w_p / W) S f takes f from the other
// lanes by shuffles; the direct term sum_b c_b grad f_b is added to the particle's slot; and c is
// scattered with the assignment stencil by float4 atomics.  Bound: the latency of the gathers and atomics at 24
// warps per SM (10 bins: long scoreboard 13.9 cycles an instruction, L1 74 % and L2 59 % busy).  256^3, 1M
// particles, D = 4, us, with 10, 16, 20
// and 32 bins: 852, 1198, 1525, 2785 (one thread per particle and bin group, values and gradients through
// shared memory: 2179, 2846, 3403, 5638).  Three CTAs per SM cost spills of 44 to 124 bytes a thread from 13 bins
// on and are still faster than two, but for 32 bins: 930, 1243, 1560, 2714 with two.  With the sixteen rows
// unrolled, two CTAs and 10 bins: 974.
template <int NBP, int D>
__global__ void __launch_bounds__(kAT, 3)
    k_adj_points(const int* __restrict__ s_cell, const float4* __restrict__ s_tq, const int* __restrict__ sidx,
                 long long np, const float4* __restrict__ f4, long long ng, int n, int nb, float hinv,
                 const float* __restrict__ S, const double* __restrict__ wsum, float4* __restrict__ h4,
                 float* __restrict__ direct) {
  constexpr int OFF = D / 2 - 1, G = NBP / 4;
  __shared__ __align__(16) float s_s[NBP * NBP];
  for (int i = threadIdx.x; i < NBP * NBP; i += blockDim.x) {
    const int r = i / NBP, c = i % NBP;
    s_s[i] = (r < nb && c < nb) ? S[r * nb + c] : 0.f;
  }
  __syncthreads();
  const float wscale = static_cast<float>(2.0 / wsum[0]);
  const int mask = n - 1, lg = __ffs(n) - 1;
  const int lane = threadIdx.x & 31, li = lane & 3, l0 = lane & ~3;
  const long long nwarp = (static_cast<long long>(gridDim.x) * kAT) >> 5;
  for (long long base = ((blockIdx.x * static_cast<long long>(kAT) + threadIdx.x) >> 5) * 8; base < np;
       base += nwarp * 8) {
    const long long p = base + (lane >> 2);
    const bool act = p < np;
    const int cell = act ? s_cell[p] : 0;
    const float4 t = act ? s_tq[p] : make_float4(0.f, 0.f, 0.f, 0.f);
    float wx[D], wy[D], wz[D], dx[D], dy[D], dz[D];
    bs_w<D>(t.x, wx, dx);
    bs_w<D>(t.y, wy, dy);
    bs_w<D>(t.z, wz, dz);
    const int cx = (cell & mask) - OFF, cy = ((cell >> lg) & mask) - OFF, cz = (cell >> (2 * lg)) - OFF;
    constexpr int NY = D == 4 ? 4 : 1;  // stencil rows of a z-layer that a lane takes
    const int ox = D == 4 ? li : (li & 1);
    float lx = wx[0], ldx = dx[0];  // this lane's x factor (for D = 2 times the y factor)
#pragma unroll
    for (int o = 1; o < D; ++o) {
      lx = ox == o ? wx[o] : lx;
      ldx = ox == o ? dx[o] : ldx;
    }
    const int xo = (cx + ox) & mask;
    const bool y1 = li >> 1;
    const float ly = y1 ? wy[1] : wy[0], ldy = y1 ? dy[1] : dy[0];  // D = 2 only
    int yo[NY];
#pragma unroll
    for (int o = 0; o < NY; ++o) yo[o] = (((cy + (D == 4 ? o : static_cast<int>(y1))) & mask) << lg) + xo;
    // the layers are a rolled loop: unrolled, the row addresses and weight products of all sixteen rows
    // stay in registers over the bin groups and spill
    auto layer = [&](int oz, float& w, float& d) {
      w = wz[0];
      d = dz[0];
#pragma unroll
      for (int o = 1; o < D; ++o) {
        w = oz == o ? wz[o] : w;
        d = oz == o ? dz[o] : d;
      }
      return ((cz + oz) & mask) << (2 * lg);
    };
    float f[G], gx[G], gy[G], gz[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const float4* src = f4 + g * ng;
      float vp[4] = {0.f, 0.f, 0.f, 0.f}, vy[4] = {0.f, 0.f, 0.f, 0.f}, vz[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
      for (int oz = 0; oz < D; ++oz) {
        float wo, zo;
        const int at = layer(oz, wo, zo);
        float4 vr[NY];
#pragma unroll
        for (int oy = 0; oy < NY; ++oy) vr[oy] = __ldg(src + (at + yo[oy]));
#pragma unroll
        for (int oy = 0; oy < NY; ++oy) {
          const float vv[4] = {vr[oy].x, vr[oy].y, vr[oy].z, vr[oy].w};
          const float a = D == 4 ? wo * wy[oy] : wo, az = D == 4 ? zo * wy[oy] : zo, ay = D == 4 ? wo * dy[oy] : 0.f;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            vp[j] = fmaf(a, vv[j], vp[j]);
            vz[j] = fmaf(az, vv[j], vz[j]);
            if (D == 4) vy[j] = fmaf(ay, vv[j], vy[j]);
          }
        }
      }
      float k4[4][4];  // [kind][bin]: f, df/dx, df/dy, df/dz of this lane's nodes
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (D == 4) {
          k4[0][j] = lx * vp[j];
          k4[1][j] = ldx * vp[j];
          k4[2][j] = lx * vy[j];
          k4[3][j] = lx * vz[j];
        } else {
          k4[0][j] = lx * ly * vp[j];
          k4[1][j] = ldx * ly * vp[j];
          k4[2][j] = lx * ldy * vp[j];
          k4[3][j] = lx * ly * vz[j];
        }
      }
      float res[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {  // reduce-scatter over the four lanes: lane i keeps bin i
        const bool hi = li & 2;
        float a0 = hi ? k4[c][2] : k4[c][0], a1 = hi ? k4[c][3] : k4[c][1];
        a0 += __shfl_xor_sync(0xffffffffu, hi ? k4[c][0] : k4[c][2], 2);
        a1 += __shfl_xor_sync(0xffffffffu, hi ? k4[c][1] : k4[c][3], 2);
        const bool odd = li & 1;
        const float keep = odd ? a1 : a0;
        res[c] = keep + __shfl_xor_sync(0xffffffffu, odd ? a0 : a1, 1);
      }
      f[g] = res[0];
      gx[g] = res[1];
      gy[g] = res[2];
      gz[g] = res[3];
    }
    float c[G];
#pragma unroll
    for (int g = 0; g < G; ++g) c[g] = 0.f;
#pragma unroll
    for (int g2 = 0; g2 < G; ++g2) {
      float fb[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) fb[j] = __shfl_sync(0xffffffffu, f[g2], l0 + j);
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const float4 sv = *reinterpret_cast<const float4*>(s_s + (4 * g + li) * NBP + 4 * g2);
        c[g] = fmaf(sv.x, fb[0], c[g]);
        c[g] = fmaf(sv.y, fb[1], c[g]);
        c[g] = fmaf(sv.z, fb[2], c[g]);
        c[g] = fmaf(sv.w, fb[3], c[g]);
      }
    }
    float ex = 0.f, ey = 0.f, ez = 0.f;
#pragma unroll
    for (int g = 0; g < G; ++g) {
      c[g] *= wscale * t.w;
      ex = fmaf(c[g], gx[g], ex);
      ey = fmaf(c[g], gy[g], ey);
      ez = fmaf(c[g], gz[g], ez);
    }
#pragma unroll
    for (int off = 1; off < 4; off <<= 1) {
      ex += __shfl_xor_sync(0xffffffffu, ex, off);
      ey += __shfl_xor_sync(0xffffffffu, ey, off);
      ez += __shfl_xor_sync(0xffffffffu, ez, off);
    }
    if (act && li < 3) {
      float* o = direct + 3 * static_cast<long long>(sidx[p]) + li;
      *o += hinv * (li == 0 ? ex : li == 1 ? ey : ez);
    }
#pragma unroll
    for (int g = 0; g < G; ++g) {
      float cb[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) cb[j] = __shfl_sync(0xffffffffu, c[g], l0 + j);
      if (act && t.w != 0.f) {
        float4* dst = h4 + g * ng;
#pragma unroll 1
        for (int oz = 0; oz < D; ++oz) {
          float wo, zo;
          const int at = layer(oz, wo, zo);
#pragma unroll
          for (int oy = 0; oy < NY; ++oy) {
            const float a = (D == 4 ? wo * wy[oy] : wo * ly) * lx;
            atomicAdd(dst + (at + yo[oy]), make_float4(a * cb[0], a * cb[1], a * cb[2], a * cb[3]));
          }
        }
      }
    }
  }
}

__global__ void k_adj_finish_node(const float* __restrict__ q, const float* __restrict__ g, long long ng, float inv_ng,
                                  float* __restrict__ grad) {
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < ng;
       i += static_cast<long long>(blockDim.x) * gridDim.x)
    grad[i] = (q[i] + g[i]) * inv_ng;
}

template <int D>
__global__ void k_adj_finish_particles(const float4* __restrict__ parts, long long np, const float* __restrict__ gd, int n,
                                       CellScale cs, const double* __restrict__ wsum, const float* __restrict__ direct,
                                       float* __restrict__ grad) {
  constexpr int OFF = D / 2 - 1;
  const int mask = n - 1;
  const float scale = static_cast<float>(static_cast<double>(n) * n * n / wsum[0]);
  const float hinv = static_cast<float>(cs.inv_h);
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < np;
       i += static_cast<long long>(blockDim.x) * gridDim.x) {
    const float4 pp = parts[i];
    float tx, ty, tz;
    const int cx = cell_t(pp.x, cs, n, tx), cy = cell_t(pp.y, cs, n, ty), cz = cell_t(pp.z, cs, n, tz);
    float wx[D], wy[D], wz[D], dx[D], dy[D], dz[D];
    bs_w<D>(tx, wx, dx);
    bs_w<D>(ty, wy, dy);
    bs_w<D>(tz, wz, dz);
    float g0 = 0.f, g1 = 0.f, g2 = 0.f;
    for (int oz = 0; oz < D; ++oz)
      for (int oy = 0; oy < D; ++oy) {
        const long long row = (static_cast<long long>((cz - OFF + oz) & mask) * n + ((cy - OFF + oy) & mask)) * n;
        for (int ox = 0; ox < D; ++ox) {
          const float v = __ldg(gd + row + ((cx - OFF + ox) & mask));
          g0 = fmaf(dx[ox] * wy[oy] * wz[oz], v, g0);
          g1 = fmaf(wx[ox] * dy[oy] * wz[oz], v, g1);
          g2 = fmaf(wx[ox] * wy[oy] * dz[oz], v, g2);
        }
      }
    const float f = (isfinite(pp.w) ? pp.w : 0.f) * scale * hinv;
    grad[3 * i] = direct[3 * i] + f * g0;
    grad[3 * i + 1] = direct[3 * i + 1] + f * g1;
    grad[3 * i + 2] = direct[3 * i + 2] + f * g2;
  }
}

inline int grid1(long long work, int sms) {
  long long g = (work + kAT - 1) / kAT;
  const long long cap = static_cast<long long>(sms) * 16;
  return static_cast<int>(g < 1 ? 1 : (g > cap ? cap : g));
}
#define ZK_ADJ_SWITCH(nb, CALL) \
  switch ((nb + 3) / 4) {       \
    case 1: CALL(4); break;     \
    case 2: CALL(8); break;     \
    case 3: CALL(12); break;    \
    case 4: CALL(16); break;    \
    case 5: CALL(20); break;    \
    case 6: CALL(24); break;    \
    case 7: CALL(28); break;    \
    default: CALL(32); break;   \
  }

}  // namespace

int launch_adj_node_point(const zeta_ctx* c, const float* delta, float* fields, const float* S, float* q,
                          cudaStream_t s) {
  StageScope prof(c, ST_ADJ_POINT, 1, s);
  float4* f4 = reinterpret_cast<float4*>(fields);
  const int g = grid1(c->ng / 2, c->num_sms);
#define ZK_CALL(P) k_adj_node<P><<<g, kAT, 0, s>>>(delta, f4, c->ng, c->p.nbins, S, q)
  ZK_ADJ_SWITCH(c->p.nbins, ZK_CALL)
#undef ZK_CALL
  return cudaGetLastError() == cudaSuccess ? ZETA_OK : ZETA_ECUDA;
}

int launch_adj_mass(const zeta_ctx* c, const float2* dhat, const float* S, float* tab, float2* gk, cudaStream_t s) {
  StageScope prof(c, ST_ADJ_OTHER, 2, s);
  const int nb = c->p.nbins, nbp = 4 * ((nb + 3) / 4);
  const size_t sm = sizeof(float) * (c->p.lmax + 1) * nb * nb;
  if (ensure_smem(reinterpret_cast<const void*>(k_adj_mass_table), sm)) return ZETA_ECUDA;
  k_adj_mass_table<<<static_cast<unsigned>((c->nn2 + kAT - 1) / kAT), kAT, sm, s>>>(c->d_jtab, c->nn2, nbp, nb, c->p.lmax,
                                                                                 S, tab);
  k_adj_mass<<<grid1(c->ng / 2, c->num_sms), kAT, 0, s>>>(dhat, tab, c->d_mhat, c->n, gk);
  return cudaGetLastError() == cudaSuccess ? ZETA_OK : ZETA_ECUDA;
}

int launch_adj_points(const zeta_ctx* c, const int* s_cell, const float4* s_tq, const int* sorted_idx, int64_t np,
                      const float* fields, const float* S, const double* wsum, float* hfield, float* direct,
                      cudaStream_t s) {
  StageScope prof(c, ST_ADJ_POINT, 1, s);
  const auto* f4 = reinterpret_cast<const float4*>(fields);
  auto* h4 = reinterpret_cast<float4*>(hfield);
  const float hinv = static_cast<float>(c->n / c->p.box);
  const int g = grid1(np * 4, c->num_sms);
#define ZK_CALL2(P) \
  k_adj_points<P, 2><<<g, kAT, 0, s>>>(s_cell, s_tq, sorted_idx, np, f4, c->ng, c->n, c->p.nbins, hinv, S, wsum, h4, direct)
#define ZK_CALL4(P) \
  k_adj_points<P, 4><<<g, kAT, 0, s>>>(s_cell, s_tq, sorted_idx, np, f4, c->ng, c->n, c->p.nbins, hinv, S, wsum, h4, direct)
  if (c->p.dsup == 2) {
    ZK_ADJ_SWITCH(c->p.nbins, ZK_CALL2)
  } else {
    ZK_ADJ_SWITCH(c->p.nbins, ZK_CALL4)
  }
#undef ZK_CALL2
#undef ZK_CALL4
  return cudaGetLastError() == cudaSuccess ? ZETA_OK : ZETA_ECUDA;
}

int launch_adj_finish_node(const zeta_ctx* c, const float* q, const float* g, float* grad, cudaStream_t s) {
  StageScope prof(c, ST_ADJ_OTHER, 1, s);
  k_adj_finish_node<<<grid1(c->ng, c->num_sms), kAT, 0, s>>>(q, g, c->ng, static_cast<float>(1.0 / c->ng), grad);
  return cudaGetLastError() == cudaSuccess ? ZETA_OK : ZETA_ECUDA;
}

int launch_adj_finish_particles(const zeta_ctx* c, const float4* parts, int64_t np, const float* gdelta,
                                const double* wsum, const float* direct, float* grad, cudaStream_t s) {
  StageScope prof(c, ST_ADJ_OTHER, 1, s);
  const CellScale cs = make_cell_scale(c->n, c->p.box);
  if (c->p.dsup == 2)
    k_adj_finish_particles<2><<<grid1(np, c->num_sms), kAT, 0, s>>>(parts, np, gdelta, c->n, cs, wsum, direct, grad);
  else
    k_adj_finish_particles<4><<<grid1(np, c->num_sms), kAT, 0, s>>>(parts, np, gdelta, c->n, cs, wsum, direct, grad);
  return cudaGetLastError() == cudaSuccess ? ZETA_OK : ZETA_ECUDA;
}

}  // namespace zk
