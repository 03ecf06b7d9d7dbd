// kernels_small.cu -- small bodies in the FP64 / FP32 modes: all of a call's
// iterations in one launch (Sections 4.3-4.5, no equalities).
//
// Walkers are independent chains (Section 4.1), so nothing but the kernel
// boundary of a draw, a chord and an update kernel ties the walkers of a small
// body together, and there each launch is a few microseconds of latency: the
// 10-dimensional cube with 100 walkers took 12 us an iteration in two launches.
// Here a CTA of 128 threads keeps G walkers (points and directions in shared
// memory, beside the rows of A) and loops over the iterations.
//   Draw: a thread per Box-Muller pair of the G walkers, for as many iterations
//     ahead (R) as one pass of the 128 threads covers: a draw depends on no
//     point, and its FP64 functions are a serial chain as long as the rest of an
//     iteration.
//   Chord, direct (FP32; FP64 with few entries): 128 / G threads per walker, a
//     thread per row, the sums in index order -- the arithmetic and the bits of
//     chord_warp_kernel.
//   Chord, screened (FP64): a lower bound of every row's ratio from FP32 dot
//     products and the standard bound gamma_{n+8} ||a_i|| ||x|| on their errors
//     (kernels_screen.cu does the same on the tensor cores), then FP64 in index
//     order for the least one and for every row whose bound does not exceed the
//     ratio found: FP64 runs at 1/64 of the FP32 rate, and the 300 rows of a
//     37-dimensional body need two.  Walkers whose coordinates leave the range
//     the bound covers evaluate every row in FP64.
// Measured per iteration, launches of 1024 iterations (before: a draw and
// chord_warp_kernel each, in a graph): FP64 10 x 20, 100 walkers 2.6 us (16.5);
// 8000 walkers 22 (209, chord_simt_kernel); 37 x 300, 301 walkers 7.3 (62);
// 64 x 500, 100 walkers 9.8 (137); 100 x 390, 20 walkers 13.3 (164); FP32 2.3,
// 9.1, 4.1, 4.5 and 5.9 us.  What is left is latency: the serial FP64 sums and
// division, and four barriers of the block (six screened).
#include <cmath>
#include <cuda_fp16.h>
#include <type_traits>

#include "mhar_device.cuh"
#include "mhar_internal.h"
#include "normals_f64.cuh"

namespace mhar {
namespace {

constexpr int kThreadsSmall = 128;
constexpr int kMaxGroup = 16;
constexpr int kMaxAhead = 16;

__device__ __forceinline__ float rcp_approx(float v) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}

template <typename T>
struct SmallParams {
  const T* A;               // m x n_ld (FP64 / FP32)
  const float* At;          // n x m_ld: FP32 columns (screened); T columns otherwise
  const T* b;
  const float* an;          // screened: gamma ||a_i||_2, rounded up
  const T* kr;              // FP32: margins, 3 per row
  const float* sigma;
  const T* delta;           // preconditioner (pc_rank >= 0)
  const T* U;
  uint64_t seed, step0;
  uint32_t walker0;
  double* out;              // samples of walkers 0 .. emit - 1, or null
  int emit, thin, phase;    // after iterations it with (phase + it + 1) % thin == 0
  int iters, m, m_ld, n, n_ld, z, pc_rank;
  double* lmin;
  double* lmax;
  double* theta;
  int* status;
  unsigned long long* counters;
  double* X64;
  float* Xhi;
  float* Xlo;
};

// Not inlined: its constants would take registers of the whole loop over the iterations.
__device__ __noinline__ double2 normals_f64(uint32_t a, uint32_t b) {
  double2 z;
  box_muller_f64(a, b, z.x, z.y);
  return z;
}
__device__ __forceinline__ void box_muller(uint32_t a, uint32_t b, double& z0, double& z1) {
  const double2 z = normals_f64(a, b);
  z0 = z.x;
  z1 = z.y;
}
__device__ __forceinline__ void box_muller(uint32_t a, uint32_t b, float& z0, float& z1) {
  box_muller_f32(a, b, z0, z1);
}

// Shared memory: the columns of A, then the per-walker arrays.  Sizes by the
// same function on the host and the device.
struct SmallLayout {
  size_t at, x, xlo, d, xd, lbs, rows, gs, nrm, u, lam, key, total;
};
template <typename T, bool SCREEN>
__host__ __device__ inline SmallLayout small_layout(int m, int m_ld, int n, int G, int R) {
  SmallLayout l;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o += (bytes + 15) / 16 * 16;
    return at;
  };
  l.at = take((SCREEN ? sizeof(float) : sizeof(T)) * static_cast<size_t>(m_ld) * n);
  l.x = take(sizeof(T) * n * G);
  l.xlo = take(sizeof(T) == 4 ? sizeof(float) * n * G : 0);
  l.d = take(sizeof(T) * n * G * R);
  l.xd = take(SCREEN ? sizeof(float2) * n * G : 0);
  l.lbs = take(SCREEN ? 2 * sizeof(float) * static_cast<size_t>(m) * G : 0);
  l.rows = take(SCREEN ? 2 * sizeof(double) * n * G : 0);
  l.gs = take(sizeof(T) * (kMaxPcRank + 1) * G * R);
  l.nrm = take(4 * sizeof(float) * G);
  l.u = take(sizeof(double) * G * R);
  l.lam = take(2 * sizeof(unsigned long long) * G);
  l.key = take(2 * sizeof(unsigned long long) * G);
  l.total = o;
  return l;
}

// The chord's ratios as bits: non-negative floats order as unsigned integers, and
// comparisons of doubles would go to the FP64 pipe.
template <typename T>
struct Bits;
template <>
struct Bits<double> {
  using U = unsigned long long;
  static constexpr U inf = 0x7ff0000000000000ull;
  static __device__ __forceinline__ U of(double v) { return static_cast<U>(__double_as_longlong(v)); }
  static __device__ __forceinline__ double value(U u) { return __longlong_as_double(static_cast<long long>(u)); }
};
template <>
struct Bits<float> {
  using U = unsigned int;
  static constexpr U inf = 0x7f800000u;
  static __device__ __forceinline__ U of(float v) { return __float_as_uint(v); }
  static __device__ __forceinline__ float value(U u) { return __uint_as_float(u); }
};

// Ratio of one row from its slack and a_i . d (clamped at 0, skipped at 0),
// folded into |lambda_max| / |lambda_min|.
template <typename T>
__device__ __forceinline__ void fold_row(T s, T g, typename Bits<T>::U& hi, typename Bits<T>::U& lo,
                                         bool& bad) {
  using B = Bits<T>;
  using U = typename B::U;
  constexpr U sign = ~(~U(0) >> 1);
  const U us = B::of(s), ug = B::of(g), ag = ug & ~sign;
  if ((us & ~sign) >= B::inf || ag >= B::inf) {
    bad = true;
    return;
  }
  if (ag == 0) return;
  const U r = B::of((us & sign ? T(0) : s) / B::value(ag));   // |s / g|
  if (ug & sign) lo = r < lo ? r : lo;
  else hi = r < hi ? r : hi;
}

template <typename T, bool SCREEN>
__global__ void __launch_bounds__(kThreadsSmall)
small_kernel(const SmallParams<T> p, int G, int R) {
  extern __shared__ __align__(16) uint8_t smem_small[];
  __shared__ double adx[SCREEN ? 1 : kThreadsSmall / 2];     // a . d of few rows
  using AT = std::conditional_t<SCREEN, float, T>;
  const SmallLayout l = small_layout<T, SCREEN>(p.m, p.m_ld, p.n, G, R);
  AT* at = reinterpret_cast<AT*>(smem_small + l.at);
  T* xs = reinterpret_cast<T*>(smem_small + l.x);
  float* xlo = reinterpret_cast<float*>(smem_small + l.xlo);
  T* ds_all = reinterpret_cast<T*>(smem_small + l.d);   // [R][G][n]
  float2* xd = reinterpret_cast<float2*>(smem_small + l.xd);
  float* lbs = reinterpret_cast<float*>(smem_small + l.lbs);
  double* rows = reinterpret_cast<double*>(smem_small + l.rows);
  T* gs = reinterpret_cast<T*>(smem_small + l.gs);
  float* nrm = reinterpret_cast<float*>(smem_small + l.nrm);
  double* us_all = reinterpret_cast<double*>(smem_small + l.u);
  unsigned long long* lam = reinterpret_cast<unsigned long long*>(smem_small + l.lam);
  unsigned long long* key = reinterpret_cast<unsigned long long*>(smem_small + l.key);

  const int tid = threadIdx.x;
  const int tpw = kThreadsSmall / G;        // threads of a walker's rows
  const int g = tid / tpw, t = tid - g * tpw;
  const int k0 = blockIdx.x * G;
  const int k = k0 + g;
  const int live = min(G, p.z - k0);        // walkers of this CTA
  const int n = p.n, m = p.m;
  const uint64_t step0 = p.step0;
  constexpr unsigned long long kInf = 0x7ff0000000000000ull;
  const float kNoBound = __int_as_float(0x7fffffff);

  if constexpr (sizeof(T) == 8) prefetch_normals_f64(tid);
  {
    const float4* src = reinterpret_cast<const float4*>(p.At);
    float4* dst = reinterpret_cast<float4*>(at);
    const int words = static_cast<int>(sizeof(AT) * p.m_ld * n / 16);
    for (int i = tid; i < words; i += kThreadsSmall) dst[i] = __ldg(src + i);
  }
  for (int i = tid; i < live * n; i += kThreadsSmall) {
    const int w = i / n, c = i - w * n;
    const size_t o = static_cast<size_t>(k0 + w) * p.n_ld + c;
    if constexpr (sizeof(T) == 8) {
      xs[i] = p.X64[o];
    } else {
      xs[i] = p.Xhi[o];
      xlo[i] = p.Xlo[o];
    }
  }
  const bool pre = p.pc_rank >= 0;
  const int pairs = (n + 1) >> 1, gpairs = pre ? (p.pc_rank + 1) >> 1 : 0;
  const int draws = pairs + gpairs + 1;
  if (pre)
    for (int i = tid; i < R * G * (kMaxPcRank + 1); i += kThreadsSmall) gs[i] = T(0);
  bool bad = false;
  __syncthreads();

  for (int it = 0; it < p.iters; ++it) {
    // Section 4.3, R iterations at a time: the directions' pairs, the low-rank
    // normals, the chords' uniforms.
    const int ahead = it % R;
    if (ahead == 0) {
      const int steps = min(R, p.iters - it);
      for (int i = tid; i < steps * live * draws; i += kThreadsSmall) {
        const int sw = i / draws, e = i - sw * draws;
        const int s = sw / live, w = sw - s * live;
        const uint64_t step = step0 + static_cast<uint64_t>(it + s);
        const uint32_t walker = p.walker0 + static_cast<uint32_t>(k0 + w);
        if (e == draws - 1) {
          us_all[s * G + w] = open_unit_f64(philox_block(p.seed, step, walker, 0u, kStreamChord).x);
          continue;
        }
        const bool low = e >= pairs;
        const int pi = low ? e - pairs : e;
        const U4 r = philox_block(p.seed, step, walker, static_cast<uint32_t>(pi >> 1),
                                  low ? kStreamLowRank : kStreamDirection);
        T v0, v1;
        box_muller((pi & 1) ? r.z : r.x, (pi & 1) ? r.w : r.y, v0, v1);
        const int c = 2 * pi;
        T* dst = low ? gs + (s * G + w) * (kMaxPcRank + 1) : ds_all + (s * G + w) * n;
        dst[c] = v0;
        if (c + 1 < (low ? p.pc_rank : n)) dst[c + 1] = v1;
      }
      __syncthreads();
      if (pre) {
        // d = delta .* h + U g, the terms in column order.
        for (int i = tid; i < steps * live * n; i += kThreadsSmall) {
          const int sw = i / n, c = i - sw * n;
          const int s = sw / live, w = sw - s * live;
          T* d = ds_all + (s * G + w) * n + c;
          T acc = p.delta[c] * *d;
          const T* u = p.U + static_cast<size_t>(c) * kMaxPcRank;
          const T* gw = gs + (s * G + w) * (kMaxPcRank + 1);
#pragma unroll 8
          for (int q = 0; q < kMaxPcRank; ++q) acc = fma(u[q], gw[q], acc);
          *d = acc;
        }
        if (!SCREEN) __syncthreads();
      }
    }
    const T* ds = ds_all + ahead * G * n;
    const double* us = us_all + ahead * G;
    for (int i = tid; i < 2 * G; i += kThreadsSmall) {
      lam[i] = kInf;
      key[i] = ~0ull;
    }
    if constexpr (SCREEN) {
      if (ahead == 0 && pre) __syncthreads();
      for (int i = tid; i < live * n; i += kThreadsSmall)
        xd[i] = make_float2(static_cast<float>(xs[i]), static_cast<float>(ds[i]));
    }
    __syncthreads();

    // Section 4.4.
    using B = Bits<T>;
    typename B::U hi = B::inf, lo = B::inf;
    if constexpr (!SCREEN) {
      if constexpr (sizeof(T) == 4) {
        // The FP32 margins' norms, added as chord_warp_kernel adds them.
        if (g < live && t < 32) {
          T nx = T(0), nd = T(0), ix = T(0), id = T(0);
          for (int c = t; c < n; c += 32) {
            const T is = T(1) / static_cast<T>(p.sigma[c]);
            const T xv = xs[g * n + c] * is, dv = ds[g * n + c] * is;
            nx += xv * xv;
            nd += dv * dv;
            ix = fmax(ix, fabs(xv));
            id = fmax(id, fabs(dv));
          }
#pragma unroll
          for (int off = 16; off > 0; off >>= 1) {
            nx += __shfl_xor_sync(0xffffffffu, nx, off);
            nd += __shfl_xor_sync(0xffffffffu, nd, off);
            ix = fmax(ix, __shfl_xor_sync(0xffffffffu, ix, off));
            id = fmax(id, __shfl_xor_sync(0xffffffffu, id, off));
          }
          if (t == 0) {
            nrm[4 * g] = sqrt(nx) * 1.0009765625f;
            nrm[4 * g + 1] = sqrt(nd) * 1.0009765625f;
            nrm[4 * g + 2] = ix;
            nrm[4 * g + 3] = id;
          }
        }
        __syncthreads();
      }
      const int half = tpw >> 1;
      if (sizeof(T) == 8 && m <= half) {
        // Few rows: one thread forms a row's a . x, another, half the walker's
        // threads on, its a . d.  (FP64 takes a warp 64 clocks an operation
        // whatever its lanes do; two rows a thread as below took four for each
        // column.)
        const int which = t >= half, r = which ? t - half : t;
        T acc = T(0);
        if (g < live && r < m) {
          const T* v = (which ? ds : xs) + g * n;
          for (int c = 0; c < n; ++c) acc += at[static_cast<size_t>(c) * p.m_ld + r] * v[c];
          if (which) adx[g * half + r] = static_cast<double>(acc);
        }
        __syncthreads();
        if (g < live && r < m && !which)
          fold_row<T>(p.b[r] - acc, static_cast<T>(adx[g * half + r]), hi, lo, bad);
      } else if (g < live) {
        for (int r0 = t; r0 < m; r0 += 2 * tpw) {
          // Two rows at a time: their serial sums overlap.
          const int r1 = r0 + tpw < m ? r0 + tpw : r0;
          T ax[2] = {T(0), T(0)}, ad[2] = {T(0), T(0)};
          for (int c = 0; c < n; ++c) {
            const T xv = xs[g * n + c], dv = ds[g * n + c];
            const T a0 = at[static_cast<size_t>(c) * p.m_ld + r0], a1 = at[static_cast<size_t>(c) * p.m_ld + r1];
            ax[0] += a0 * xv;
            ad[0] += a0 * dv;
            ax[1] += a1 * xv;
            ad[1] += a1 * dv;
          }
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const int r = q ? r1 : r0;
            if (q && r1 == r0) break;
            T s = p.b[r] - ax[q];
            T gg = ad[q];
            if constexpr (sizeof(T) == 4) {
              const T k2 = p.kr[3 * r], k1 = p.kr[3 * r + 1];
              s -= fmin(k2 * nrm[4 * g], k1 * nrm[4 * g + 2]);
              const T eg = fmin(k2 * nrm[4 * g + 1], k1 * nrm[4 * g + 3]);
              gg = gg > T(0) ? gg + eg : (gg < T(0) ? gg - eg : gg);
            }
            fold_row(s, gg, hi, lo, bad);
          }
        }
      }
    } else {
      // Bounds from FP32, ||x||_2 and ||d||_2 summed on the way (every thread
      // the same).
      bool force = false;
      unsigned long long kh = ~0ull, kl = ~0ull;
      if (g < live) {
        const float2* v = xd + g * n;
        for (int r0 = t; r0 < m; r0 += 4 * tpw) {
          float ax[4], ad[4], nx2 = 0.0f, nd2 = 0.0f;
          int rq[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            ax[q] = ad[q] = 0.0f;
            rq[q] = min(r0 + q * tpw, m - 1);
          }
#pragma unroll 4
          for (int c = 0; c < n; ++c) {
            const float2 e = v[c];
            const AT* col = at + static_cast<size_t>(c) * p.m_ld;
            nx2 = fmaf(e.x, e.x, nx2);
            nd2 = fmaf(e.y, e.y, nd2);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const float a = static_cast<float>(col[rq[q]]);
              ax[q] = fmaf(a, e.x, ax[q]);
              ad[q] = fmaf(a, e.y, ad[q]);
            }
          }
          force = !(nx2 >= 0x1p-90f && nx2 <= 0x1p90f && nd2 >= 0x1p-90f && nd2 <= 0x1p90f);
          if (force) break;
          const float nx = sqrtf(nx2) * 1.0009765625f, nd = sqrtf(nd2) * 1.0009765625f;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int r = r0 + q * tpw;
            if (r >= m) break;
            // Lowered slack over a_i . d moved towards each side by its bound;
            // (1 - 2^-20) covers the roundings of both and of the quotient.
            const float ga = __ldg(p.an + r), bf = static_cast<float>(p.b[r]);
            const float s = fmaxf(bf - ax[q] - fmaf(ga, nx, 0x1p-22f * fabsf(bf)), 0.0f) *
                            (1.0f - 0x1p-20f);
            const float dh = fmaf(ga, nd, ad[q]), dl = fmaf(ga, nd, -ad[q]);
            // NaN: not on that side.  (+Inf is a quotient past FP32's range, from short
            // directions, and a row's like any other.)
            const float bh = dh > 0.0f ? s * rcp_approx(dh) : kNoBound;
            const float bl = dl > 0.0f ? s * rcp_approx(dl) : kNoBound;
            lbs[(2 * g) * m + r] = bh;
            lbs[(2 * g + 1) * m + r] = bl;
            if (dh > 0.0f)
              kh = min(kh, (static_cast<unsigned long long>(__float_as_uint(bh)) << 32) | r);
            if (dl > 0.0f)
              kl = min(kl, (static_cast<unsigned long long>(__float_as_uint(bl)) << 32) | r);
          }
        }
      }
      const int width = min(tpw, 32);
      for (int off = width / 2; off > 0; off >>= 1) {
        kh = min(kh, __shfl_xor_sync(0xffffffffu, kh, off));
        kl = min(kl, __shfl_xor_sync(0xffffffffu, kl, off));
      }
      if ((t & (width - 1)) == 0) {
        atomicMin(&key[2 * g], kh);
        atomicMin(&key[2 * g + 1], kl);
      }
      __syncthreads();
      // The two rows into shared memory, then their four serial sums.
      const unsigned long long bh = key[2 * g], bl = key[2 * g + 1];
      const int rh = static_cast<int>(bh & 0xffffffffu), rl = static_cast<int>(bl & 0xffffffffu);
      const bool on = g < live;
      if (on)
        for (int i = t; i < 2 * n; i += tpw) {
          const int side = i >= n, c = side ? i - n : i;
          if ((side ? bl : bh) != ~0ull)
            rows[(2 * g + side) * n + c] = p.A[static_cast<size_t>(side ? rl : rh) * p.n_ld + c];
        }
      __syncthreads();
      {
        const int side = (t >> 1) & 1, which = t & 1;
        const bool has = on && t < 4 && (side ? bl : bh) != ~0ull;
        double acc = 0.0;
        if (has) {
          const double* a = rows + (2 * g + side) * n;
          const T* v = (which ? ds : xs) + g * n;
#pragma unroll 8
          for (int c = 0; c < n; ++c) acc += a[c] * v[c];
        }
        const double oth = __shfl_xor_sync(0xffffffffu, acc, 1);
        if (has && which == 0) {
          unsigned long long h2 = kInf, l2 = kInf;
          fold_row<double>(p.b[side ? rl : rh] - acc, oth, h2, l2, bad);
          lam[2 * g + side] = side ? l2 : h2;
        }
      }
      __syncthreads();
      // Every other row that may lower a ratio found.
      if (g < live) {
        const unsigned long long lh = lam[2 * g], ll = lam[2 * g + 1];
        const float fh = lh ? static_cast<float>(B::value(lh)) * (1.0f + 0x1p-20f) : -1.0f;
        const float fl = ll ? static_cast<float>(B::value(ll)) * (1.0f + 0x1p-20f) : -1.0f;
        for (int r = t; r < m; r += tpw) {
          bool take = force;
          if (!force) {
            const float qh = lbs[(2 * g) * m + r], ql = lbs[(2 * g + 1) * m + r];
            take = (qh <= fh && r != rh) || (ql <= fl && r != rl);
          }
          if (take) {
            const T* a = p.A + static_cast<size_t>(r) * p.n_ld;
            T ax = T(0), ad = T(0);
            for (int c = 0; c < n; ++c) {
              ax += a[c] * xs[g * n + c];
              ad += a[c] * ds[g * n + c];
            }
            fold_row<T>(p.b[r] - ax, ad, hi, lo, bad);
          }
        }
      }
    }
    {
      // Fold the threads' ratios.
      const int width = min(tpw, 32);
      if constexpr (!SCREEN) {
        for (int off = width / 2; off > 0; off >>= 1) {
          const auto oh = __shfl_xor_sync(0xffffffffu, hi, off);
          const auto ol = __shfl_xor_sync(0xffffffffu, lo, off);
          hi = oh < hi ? oh : hi;
          lo = ol < lo ? ol : lo;
        }
        if (t & (width - 1)) hi = lo = B::inf;
      }
      if (hi < B::inf) atomicMin(&lam[2 * g], Bits<double>::of(static_cast<double>(B::value(hi))));
      if (lo < B::inf) atomicMin(&lam[2 * g + 1], Bits<double>::of(static_cast<double>(B::value(lo))));
    }
    __syncthreads();

    // Section 4.5; every thread draws theta for its own coordinates.
    auto theta_of = [&](int w, double& L, double& H) {
      H = __longlong_as_double(static_cast<long long>(lam[2 * w]));
      L = -__longlong_as_double(static_cast<long long>(lam[2 * w + 1]));
      if (lam[2 * w] == kInf || lam[2 * w + 1] == kInf || L > H) return 0.0;
      const double tt = L + us[w] * (H - L);
      return sizeof(T) != 8 ? static_cast<double>(static_cast<float>(tt)) : tt;
    };
    if (g < live && t == 0) {
      double L, H;
      const double tt = theta_of(g, L, H);
      if (isinf(L) || isinf(H)) {
        atomicOr(p.status, MHAR_ST_UNBOUNDED);
        atomicAdd(&p.counters[1], 1ull);
      } else if (L > H) {
        atomicOr(p.status, MHAR_ST_STALL);
        atomicAdd(&p.counters[0], 1ull);
      }
      if (it == p.iters - 1) {
        p.lmin[k] = L;
        p.lmax[k] = H;
        p.theta[k] = tt;
      }
    }
    for (int i = tid; i < live * n; i += kThreadsSmall) {
      double L, H;
      const double tt = theta_of(i / n, L, H);
      if constexpr (sizeof(T) == 8) {
        xs[i] += tt * ds[i];
      } else {
        df_axpy(xs[i], xlo[i], static_cast<float>(tt), ds[i]);
      }
    }
    __syncthreads();
    if (p.out != nullptr && (p.phase + it + 1) % p.thin == 0) {
      double* dst = p.out + static_cast<size_t>((p.phase + it + 1) / p.thin - 1) * p.emit * n +
                    static_cast<size_t>(k0) * n;
      for (int i = tid; i < min(live, p.emit - k0) * n; i += kThreadsSmall) {
        if constexpr (sizeof(T) == 8) dst[i] = xs[i];
        else dst[i] = static_cast<double>(xs[i]) + static_cast<double>(xlo[i]);
      }
    }
  }
  if (bad) atomicOr(p.status, MHAR_ST_NONFINITE);
  for (int i = tid; i < live * n; i += kThreadsSmall) {
    const int w = i / n, c = i - w * n;
    const size_t o = static_cast<size_t>(k0 + w) * p.n_ld + c;
    if constexpr (sizeof(T) == 8) {
      p.X64[o] = xs[i];
    } else {
      p.Xhi[o] = xs[i];
      p.Xlo[o] = xlo[i];
    }
  }
}

// A in the layout the kernel copies (columns of m_ld entries), and, screened,
// gamma_{n+8} ||a_i||_2 and a flag when a row or its b lies outside 2^-50 .. 2^50.
// A warp per row.
template <typename T, bool SCREEN>
__global__ void small_prepare_kernel(int m, int m_ld, int n, int n_ld, const T* A, const double* b,
                                     void* At, float* an, int* outside) {
  const int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= m) return;
  double ss = 0.0, mx = 0.0;
  for (int c = lane; c < n; c += 32) {
    const T a = A[static_cast<size_t>(r) * n_ld + c];
    const size_t o = static_cast<size_t>(c) * m_ld + r;
    if constexpr (SCREEN) {
      static_cast<float*>(At)[o] = static_cast<float>(a);
      ss += static_cast<double>(a) * static_cast<double>(a);
      mx = fmax(mx, fabs(static_cast<double>(a)));
    } else {
      static_cast<T*>(At)[o] = a;
    }
  }
  if constexpr (SCREEN) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      ss += __shfl_xor_sync(0xffffffffu, ss, off);
      mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    }
    if (lane == 0) {
      const double k = static_cast<double>(n + 8) * 0x1p-24;
      an[r] = static_cast<float>(k / (1.0 - k) * sqrt(ss) * (1.0 + 0x1p-8));
      if (!(mx <= 0x1p50 && (mx == 0.0 || mx >= 0x1p-50) && fabs(b[r]) <= 0x1p50))
        atomicOr(outside, 1);
    }
  }
}

// FP64 bodies with more entries than this are screened: below it a row's
// serial FP64 sum is short and one row a thread covers the body.
constexpr int kDirectEntries = 1024;
constexpr size_t kSmallSmem = 200 << 10;

bool small_screened(const mhar_ctx* c) {
  return c->opts.precision == MHAR_FP64 && static_cast<long long>(c->m) * c->n > kDirectEntries;
}

// Iterations drawn ahead: one pass of the threads.
int small_ahead(const mhar_ctx* c, int G) {
  const int draws = (c->n + 1) / 2 + (c->pc_rank + 2) / 2 + 1;
  const int R = kThreadsSmall / (G * draws);
  return R < 1 ? 1 : (R > kMaxAhead ? kMaxAhead : R);
}

size_t small_bytes(const mhar_ctx* c, int G) {
  const int m_ld = (c->m + 3) / 4 * 4, R = small_ahead(c, G);
  if (c->opts.precision == MHAR_FP32) return small_layout<float, false>(c->m, m_ld, c->n, G, R).total;
  return small_screened(c) ? small_layout<double, true>(c->m, m_ld, c->n, G, R).total
                           : small_layout<double, false>(c->m, m_ld, c->n, G, R).total;
}

// Walkers per CTA: one while the walkers alone do not fill the SMs twice, then
// as many (a power of two) as leave two CTAs per SM and fit its shared memory
// twice.  FP32: at most four, so that a warp belongs to one walker.
int small_group(const mhar_ctx* c) {
  int sms = 148;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
  const int most = c->opts.precision == MHAR_FP32 ? 4 : kMaxGroup;
  int G = 1;
  while (2 * G <= most && c->z / (2 * G) >= 2 * sms && small_bytes(c, 2 * G) <= kSmallSmem / 2) G *= 2;
  return G;
}

template <typename T, bool SCREEN>
cudaError_t launch_small_t(mhar_ctx* c, const SmallRun& r, const T* A, const T* b, const T* kr,
                           const T* delta, const T* U) {
  SmallParams<T> p;
  p.A = A;
  p.At = reinterpret_cast<const float*>(c->d.small_at);
  p.b = b;
  p.an = c->d.small_an;
  p.kr = kr;
  p.sigma = c->d.sigma;
  p.delta = delta;
  p.U = U;
  p.seed = c->opts.seed;
  p.step0 = r.step;
  p.out = r.out;
  p.emit = r.emit;
  p.thin = r.thin;
  p.phase = r.phase;
  p.walker0 = c->opts.walker0;
  p.iters = r.iters;
  p.m = c->m;
  p.m_ld = (c->m + 3) / 4 * 4;
  p.n = c->n;
  p.n_ld = c->n_ld;
  p.z = c->z;
  p.pc_rank = c->pc_rank;
  p.lmin = c->d.lmin;
  p.lmax = c->d.lmax;
  p.theta = c->d.theta;
  p.status = c->d.status;
  p.counters = c->d.counters;
  p.X64 = c->d.X64;
  p.Xhi = c->d.Xhi;
  p.Xlo = c->d.Xlo;
  const int G = small_group(c);
  small_kernel<T, SCREEN><<<(c->z + G - 1) / G, kThreadsSmall, small_bytes(c, G), c->stream>>>(
      p, G, small_ahead(c, G));
  return cudaGetLastError();
}

}  // namespace

bool small_eligible(const mhar_ctx* c) {
  return simt_warp_path(c) && c->mE == 0 && small_bytes(c, 1) <= kSmallSmem;
}

size_t small_arena(mhar_ctx* c, uint8_t* base) {
  const size_t at = (sizeof(double) * static_cast<size_t>((c->m + 3) / 4 * 4) * c->n + 255) / 256 * 256;
  if (base) {
    c->d.small_at = base;
    c->d.small_an = reinterpret_cast<float*>(base + at);
  }
  return at + sizeof(float) * static_cast<size_t>(c->m);
}

cudaError_t small_prepare(mhar_ctx* c, int* outside) {
  const int blocks = (c->m + 3) / 4, m_ld = (c->m + 3) / 4 * 4;
  const int bytes = static_cast<int>(kSmallSmem);
  cudaError_t e = cudaFuncSetAttribute(small_kernel<float, false>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(small_kernel<double, false>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(small_kernel<double, true>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) return e;
  if (c->opts.precision == MHAR_FP32)
    small_prepare_kernel<float, false><<<blocks, 128, 0, c->stream>>>(
        c->m, m_ld, c->n, c->n_ld, c->d.A32, c->d.b64, c->d.small_at, c->d.small_an, outside);
  else if (small_screened(c))
    small_prepare_kernel<double, true><<<blocks, 128, 0, c->stream>>>(
        c->m, m_ld, c->n, c->n_ld, c->d.A64, c->d.b64, c->d.small_at, c->d.small_an, outside);
  else
    small_prepare_kernel<double, false><<<blocks, 128, 0, c->stream>>>(
        c->m, m_ld, c->n, c->n_ld, c->d.A64, c->d.b64, c->d.small_at, c->d.small_an, outside);
  return cudaGetLastError();
}

cudaError_t launch_small(mhar_ctx* c, const SmallRun& r) {
  mhar::DeviceBuffers& d = c->d;
  if (c->opts.precision == MHAR_FP32)
    return launch_small_t<float, false>(c, r, d.A32, d.b32, d.kr32, d.pc_delta32, d.pc_U32);
  if (small_screened(c))
    return launch_small_t<double, true>(c, r, d.A64, d.b64, nullptr, d.pc_delta64, d.pc_U64);
  return launch_small_t<double, false>(c, r, d.A64, d.b64, nullptr, d.pc_delta64, d.pc_U64);
}

}  // namespace mhar
