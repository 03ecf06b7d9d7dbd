// kernels_simt.cu -- CUDA-core kernels of the MHAR walker step.
//
// Section 4.3 (Generating D): Philox4x32-10 words -> Box-Muller N(0,1) entries
//   of H, one thread per (walker, quad of coordinates); D = P H through the
//   projector of Section 3.2 in the form P = I - Q^T Q, Q = L^{-1} A_E with
//   orthonormal rows (L the Cholesky factor of A_E A_E^T).
// Section 4.4 (Finding the line sets) in the recompute formulation of
//   Lemma 4.2: A X and A D are tiled over (64 rows x 64 walkers) blocks, the
//   slack b - A X and the ratios are formed in registers, and every block
//   folds its rows into per-walker (lambda_min, lambda_max) with ordered-key
//   atomics, so the m x z ratio matrix never reaches memory.
// Section 4.5 (Choosing samples): one warp per walker draws theta uniformly
//   on the chord and moves x += theta d.
// These kernels serve MHAR_FP64 (T = double) and MHAR_FP32 (T = float; points
// kept as FP32 pairs).  The tensor-core mode is in kernels_tc.cu.
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cuda_fp16.h>

#include "mhar_device.cuh"
#include "mhar_internal.h"
#include "normals_f64.cuh"

namespace mhar {
namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ double neg_inf() { return -__longlong_as_double(0x7ff0000000000000ll); }
__device__ __forceinline__ double pos_inf() { return __longlong_as_double(0x7ff0000000000000ll); }

// ---- Section 4.3: direction entries ----------------------------------------
// mode 0: FP64 -> D64 (one thread per Box-Muller pair: the FP64 functions are
// slow on this GPU, so the two pairs of a quad go to two threads); mode 1:
// FP32 -> D32; mode 2: FP32 -> FP16 hi/lo split (when there is no
// projection) or FP32 scratch D32 (projection follows).  One thread per quad
// in modes 1 and 2.
__global__ void directions_kernel(int mode, int split, uint64_t seed, const uint64_t* step_ptr,
                                  int j, uint32_t walker0, int z, int n, int n_ld, int k_pad,
                                  const float* sigma, double* D64, float* D32, __half* Dh,
                                  __half* Dl, __half* Dh1, __half* Dl1) {
  const int quads = (n + 3) >> 2;
  const int per_quad = mode == 0 ? 2 : 1;
  const long long idx = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx >= static_cast<long long>(z) * quads * per_quad) return;
  const long long qi = idx / per_quad;
  const int half = static_cast<int>(idx - qi * per_quad);
  const int k = static_cast<int>(qi / quads);
  const int q = static_cast<int>(qi - static_cast<long long>(k) * quads);
  const uint64_t step = *step_ptr + static_cast<uint64_t>(j);
  if (Dh1 != nullptr && (step & 1ull)) {
    Dh = Dh1;  // iteration s's pair is s % 2
    Dl = Dl1;
  }
  const U4 w = philox_block(seed, step, walker0 + static_cast<uint32_t>(k),
                            static_cast<uint32_t>(q), kStreamDirection);
  const int i0 = 4 * q;
  if (mode == 0) {
    // One call: a branch for each half ran both for every warp.
    double v[2];
    box_muller_f64(half ? w.z : w.x, half ? w.w : w.y, v[0], v[1]);
    double* dst = D64 + static_cast<size_t>(k) * n_ld + i0 + 2 * half;
#pragma unroll
    for (int e = 0; e < 2; ++e)
      if (i0 + 2 * half + e < n) dst[e] = v[e];
  } else {
    float v[4];
    box_muller_f32(w.x, w.y, v[0], v[1]);
    box_muller_f32(w.z, w.w, v[2], v[3]);
    if (mode == 2 && split) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (i0 + e < n) {
          const float vs = v[e] * pow2_recip(sigma[i0 + e]);   // d_i / sigma_i, exact
          const __half h = __float2half_rn(vs);
          const __half l = __float2half_rn(vs - __half2float(h));
          Dh[static_cast<size_t>(k) * k_pad + i0 + e] = h;
          Dl[static_cast<size_t>(k) * k_pad + i0 + e] = l;
        }
      }
    } else {
      float* dst = D32 + static_cast<size_t>(k) * n_ld + i0;
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (i0 + e < n) dst[e] = v[e];
    }
  }
}

// ---- Section 3.2: d = P h with P = I - Q^T Q (FP64 mode) -------------------
// One warp per walker.  Q (mE x n, orthonormal rows, Q = L^{-1} A_E): the
// coefficients c = Q h in FP64 (warp reductions; every lane ends with the
// sum), kept in shared memory (mE doubles per warp, dynamic), then
// d_i = h_i - sum_e c_e q_ei in place.
__global__ void projection_f64_kernel(int z, int n, int n_ld, int mE, const double* __restrict__ Q64,
                                      double* D) {
  extern __shared__ double proj_c[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k = blockIdx.x * (blockDim.x >> 5) + warp;
  if (k >= z) return;
  double* h = D + static_cast<size_t>(k) * n_ld;
  double* c = proj_c + static_cast<size_t>(warp) * mE;
  for (int e = 0; e < mE; ++e) {
    const double* q = Q64 + static_cast<size_t>(e) * n_ld;
    double acc = 0.0;
    for (int i = lane; i < n; i += 32) acc += q[i] * h[i];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (lane == 0) c[e] = acc;
  }
  __syncwarp();
  for (int i = lane; i < n; i += 32) {
    double v = h[i];
    for (int e = 0; e < mE; ++e) v -= c[e] * Q64[static_cast<size_t>(e) * n_ld + i];
    h[i] = v;
  }
}

// ---- Section 3.2 in the FP32 and tensor-core modes -------------------------
// The same projection in double-float arithmetic (unevaluated sums of two
// FP32 numbers, about 2^-46 relative; mhar_device.cuh): the FP64 units of this
// GPU run at a small fraction of the FP32 rate, and pairs of FP32 carry the
// cancellation in h - Q^T Q h all the same.  Q = Qh + Ql, Qh = fl32(Q) and
// Ql = fl32(Q - Qh).  One warp per walker; each lane takes quads of 4
// consecutive coordinates (one Philox block of Section 4.3, one 16-byte load
// of a row of Q).
// d = h - Q^T c with c = Q h, rounded once to FP32: kept in D32 (FP32 mode) or
// split into the FP16 operand pair d / sigma (tensor-core modes: split).
// The direction actually used (FP32, or sigma (d_hi + d_lo)) leaves a
// rounding residual A_E d of order 1e-7 |d|: its coordinates c' = Q d_used in
// the row space are stored per walker (corr), and the point update moves
// along d - Q^T c', so that A_E x = b_E does not drift by theta * 1e-7 per
// iteration; ||Q^T c' / sigma||_2, rounded up (corrn), enters the chord's
// error margins (walker_tail.cuh).
// draw: h is the direction kernel's draw, made here (and made again in the
// second pass rather than stored); otherwise h is read from D32 (the
// preconditioned draw).
constexpr int kProjRows = 4;   // rows of Q accumulated per pass over h

// (s, r) += (ah + al) b
__device__ __forceinline__ void ff_acc(float& s, float& r, float ah, float al, float b) {
  const float p = ah * b;
  const float pe = fmaf(al, b, fmaf(ah, b, -p));
  float t, err;
  two_sum(s, p, t, err);
  s = t;
  r += err + pe;
}
// (s, r) -= (ch + cl)(qh + ql), the cl ql term dropped (2^-48 relative)
__device__ __forceinline__ void ff_sub_prod(float& s, float& r, float ch, float cl, float qh,
                                            float ql) {
  const float p = ch * qh;
  const float pe = fmaf(cl, qh, fmaf(ch, ql, fmaf(ch, qh, -p)));
  float t, err;
  two_sum(s, -p, t, err);
  s = t;
  r += err - pe;
}
// Sum over the warp.  Lanes may differ in the last bit of r (the order of
// the low-part additions): the caller takes lane 0's.
__device__ __forceinline__ void ff_warp_sum(float& s, float& r) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float os = __shfl_xor_sync(0xffffffffu, s, off);
    const float orr = __shfl_xor_sync(0xffffffffu, r, off);
    float t, err;
    two_sum(s, os, t, err);
    s = t;
    r += orr + err;
  }
}
__device__ __forceinline__ void draw_quad(uint64_t seed, uint64_t step, uint32_t walker, int q,
                                          int n, float (&h)[4]) {
  const U4 w = philox_block(seed, step, walker, static_cast<uint32_t>(q), kStreamDirection);
  box_muller_f32(w.x, w.y, h[0], h[1]);
  box_muller_f32(w.z, w.w, h[2], h[3]);
  if (4 * q + 4 > n) {
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (4 * q + u >= n) h[u] = 0.0f;
  }
}
__device__ __forceinline__ uint2 pack4h(const __half* h) {
  return make_uint2(static_cast<uint32_t>(__half_as_ushort(h[0])) |
                        (static_cast<uint32_t>(__half_as_ushort(h[1])) << 16),
                    static_cast<uint32_t>(__half_as_ushort(h[2])) |
                        (static_cast<uint32_t>(__half_as_ushort(h[3])) << 16));
}

__global__ void __launch_bounds__(kThreads)
projection_ff_kernel(int draw, uint64_t seed, const uint64_t* step_ptr, int j, uint32_t walker0,
                     int z, int n, int n_ld, int mE, const float* __restrict__ Qh,
                     const float* __restrict__ Ql, float* D32, int split, int k_pad, int z_ld,
                     int inter, const float* __restrict__ sigma, __half* Dh, __half* Dl,
                     __half* Dh1, __half* Dl1, float* corr, float* corrn, int keep,
                     int* status) {
  extern __shared__ __align__(16) float proj_ff[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k = blockIdx.x * (blockDim.x >> 5) + warp;
  if (k >= z) return;  // whole warps: k is the warp's
  const uint64_t step = *step_ptr + static_cast<uint64_t>(j);
  if (Dh1 != nullptr && (step & 1ull)) {
    Dh = Dh1;  // recompute mode: iteration s's pair is s % 2
    Dl = Dl1;
  }
  // keep: h is kept in shared memory (keep floats per warp, first) between
  // the passes; otherwise it is drawn (or read) again.
  float* hk = proj_ff + static_cast<size_t>(warp) * keep;
  float* ch = proj_ff + static_cast<size_t>(blockDim.x >> 5) * keep +
              static_cast<size_t>(warp) * 3 * mE;  // c (hi, lo), then c'
  float* cl = ch + mE;
  float* cp = cl + mE;
  const int quads = (n + 3) >> 2;
  float* Dk = D32 + static_cast<size_t>(k) * n_ld;
  const uint32_t walker = walker0 + static_cast<uint32_t>(k);
  auto normals = [&](int q, float (&h)[4]) {
    if (draw) {
      draw_quad(seed, step, walker, q, n, h);
    } else {
      const float4 v = *reinterpret_cast<const float4*>(Dk + 4 * q);
      h[0] = v.x; h[1] = v.y; h[2] = v.z; h[3] = v.w;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (4 * q + u >= n) h[u] = 0.0f;
    }
  };
  auto qrow = [&](const float* Q, int e, int q) {
    return __ldg(reinterpret_cast<const float4*>(Q + static_cast<size_t>(e) * n_ld + 4 * q));
  };
  // The direction actually used, read back (rows of c' past the first pass).
  auto used = [&](int q, float (&du)[4]) {
    const int i0 = 4 * q;
    if (split) {
      const size_t o = op_off(k, i0, k_pad, z_ld, inter);
      const uint2 a = *reinterpret_cast<const uint2*>(Dh + o);
      const uint2 b = *reinterpret_cast<const uint2*>(Dl + o);
      const uint32_t aw[2] = {a.x, a.y}, bw[2] = {b.x, b.y};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float hh = __half2float(__ushort_as_half(static_cast<unsigned short>(aw[u >> 1] >> (16 * (u & 1)))));
        const float ll = __half2float(__ushort_as_half(static_cast<unsigned short>(bw[u >> 1] >> (16 * (u & 1)))));
        du[u] = i0 + u < n ? (hh + ll) * sigma[i0 + u] : 0.0f;
      }
    } else {
      const float4 v = *reinterpret_cast<const float4*>(Dk + i0);
      du[0] = v.x; du[1] = v.y; du[2] = v.z; du[3] = v.w;
    }
  };

  // (1) c = Q h, kProjRows rows of Q per pass over h.
  for (int e0 = 0; e0 < mE; e0 += kProjRows) {
    float s[kProjRows], r[kProjRows];
#pragma unroll
    for (int u = 0; u < kProjRows; ++u) s[u] = r[u] = 0.0f;
    for (int q = lane; q < quads; q += 32) {
      float h[4];
      if (keep && e0 > 0) {
        const float4 v = *reinterpret_cast<const float4*>(hk + 4 * q);
        h[0] = v.x; h[1] = v.y; h[2] = v.z; h[3] = v.w;
      } else {
        normals(q, h);
        if (keep) *reinterpret_cast<float4*>(hk + 4 * q) = make_float4(h[0], h[1], h[2], h[3]);
      }
#pragma unroll
      for (int u = 0; u < kProjRows; ++u) {
        if (e0 + u < mE) {
          const float4 a = qrow(Qh, e0 + u, q), b = qrow(Ql, e0 + u, q);
          ff_acc(s[u], r[u], a.x, b.x, h[0]);
          ff_acc(s[u], r[u], a.y, b.y, h[1]);
          ff_acc(s[u], r[u], a.z, b.z, h[2]);
          ff_acc(s[u], r[u], a.w, b.w, h[3]);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < kProjRows; ++u) {
      ff_warp_sum(s[u], r[u]);
      if (lane == 0 && e0 + u < mE) fast_two_sum(s[u], r[u], ch[e0 + u], cl[e0 + u]);
    }
  }
  __syncwarp();

  // (2) d = h - Q^T c, rounded once; its FP16 pair or FP32 copy; c' of the
  // first kProjRows rows on the way.
  const bool want_corr = corr != nullptr;
  float s2[kProjRows], r2[kProjRows];
#pragma unroll
  for (int u = 0; u < kProjRows; ++u) s2[u] = r2[u] = 0.0f;
  for (int q = lane; q < quads; q += 32) {
    const int i0 = 4 * q;
    float ds[4], dr[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    if (keep) {  // each lane reads back the quads it stored
      const float4 v = *reinterpret_cast<const float4*>(hk + i0);
      ds[0] = v.x; ds[1] = v.y; ds[2] = v.z; ds[3] = v.w;
    } else {
      normals(q, ds);
    }
    for (int e = 0; e < mE; ++e) {
      const float c_hi = ch[e], c_lo = cl[e];
      const float4 a = qrow(Qh, e, q), b = qrow(Ql, e, q);
      ff_sub_prod(ds[0], dr[0], c_hi, c_lo, a.x, b.x);
      ff_sub_prod(ds[1], dr[1], c_hi, c_lo, a.y, b.y);
      ff_sub_prod(ds[2], dr[2], c_hi, c_lo, a.z, b.z);
      ff_sub_prod(ds[3], dr[3], c_hi, c_lo, a.w, b.w);
    }
    // Past n, h and the padded columns of Q are 0, and so is d: no
    // per-coordinate test (sigma is 1 there).
    float du[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) du[u] = ds[u] + dr[u];
    if (split) {
      __half hh[4], ll[4];
      bool bad = false;
      const float4 sg4 = __ldg(reinterpret_cast<const float4*>(sigma + i0));
      const float sg[4] = {sg4.x, sg4.y, sg4.z, sg4.w};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float v = du[u] * pow2_recip(sg[u]);  // exact
        hh[u] = __float2half_rn(v);
        ll[u] = __float2half_rn(v - __half2float(hh[u]));
        bad |= !(fabsf(v) <= kHalfMax);
        // hi + lo is exact in FP32 (at most 24 significant bits), and so is
        // the scaling by sigma.
        du[u] = (__half2float(hh[u]) + __half2float(ll[u])) * sg[u];
      }
      const size_t o = op_off(k, i0, k_pad, z_ld, inter);
      *reinterpret_cast<uint2*>(Dh + o) = pack4h(hh);
      *reinterpret_cast<uint2*>(Dl + o) = pack4h(ll);
      if (bad) atomicOr(status, MHAR_ST_NONFINITE);
    } else {
      *reinterpret_cast<float4*>(Dk + i0) = make_float4(du[0], du[1], du[2], du[3]);
    }
    if (want_corr) {
#pragma unroll
      for (int u = 0; u < kProjRows; ++u) {
        if (u < mE) {
          const float4 a = qrow(Qh, u, q), b = qrow(Ql, u, q);
          ff_acc(s2[u], r2[u], a.x, b.x, du[0]);
          ff_acc(s2[u], r2[u], a.y, b.y, du[1]);
          ff_acc(s2[u], r2[u], a.z, b.z, du[2]);
          ff_acc(s2[u], r2[u], a.w, b.w, du[3]);
        }
      }
    }
  }
  if (!want_corr) return;
  float* ck = corr + static_cast<size_t>(k) * mE;
#pragma unroll
  for (int u = 0; u < kProjRows; ++u) {
    ff_warp_sum(s2[u], r2[u]);
    if (lane == 0 && u < mE) ck[u] = cp[u] = s2[u] + r2[u];
  }
  // (3) c' of the remaining rows, from the stored direction (each lane reads
  // back the quads it wrote).
  for (int e0 = kProjRows; e0 < mE; e0 += kProjRows) {
    float s[kProjRows], r[kProjRows];
#pragma unroll
    for (int u = 0; u < kProjRows; ++u) s[u] = r[u] = 0.0f;
    for (int q = lane; q < quads; q += 32) {
      float du[4];
      used(q, du);
#pragma unroll
      for (int u = 0; u < kProjRows; ++u) {
        if (e0 + u < mE) {
          const float4 a = qrow(Qh, e0 + u, q), b = qrow(Ql, e0 + u, q);
          ff_acc(s[u], r[u], a.x, b.x, du[0]);
          ff_acc(s[u], r[u], a.y, b.y, du[1]);
          ff_acc(s[u], r[u], a.z, b.z, du[2]);
          ff_acc(s[u], r[u], a.w, b.w, du[3]);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < kProjRows; ++u) {
      ff_warp_sum(s[u], r[u]);
      if (lane == 0 && e0 + u < mE) ck[e0 + u] = cp[e0 + u] = s[u] + r[u];
    }
  }
  __syncwarp();
  // (4) ||Q^T c' / sigma||_2 in FP32, rounded up by 2^-10 (far above the
  // FP32 rounding of these n mE products).
  float cn = 0.0f;
  for (int q = lane; q < quads; q += 32) {
    float dlt[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    for (int e = 0; e < mE; ++e) {
      const float4 a = qrow(Qh, e, q);
      const float ce = cp[e];
      dlt[0] = fmaf(a.x, ce, dlt[0]);
      dlt[1] = fmaf(a.y, ce, dlt[1]);
      dlt[2] = fmaf(a.z, ce, dlt[2]);
      dlt[3] = fmaf(a.w, ce, dlt[3]);
    }
    const float4 sg4 = __ldg(reinterpret_cast<const float4*>(sigma + 4 * q));
    const float v0 = dlt[0] * pow2_recip(sg4.x), v1 = dlt[1] * pow2_recip(sg4.y);
    const float v2 = dlt[2] * pow2_recip(sg4.z), v3 = dlt[3] * pow2_recip(sg4.w);
    cn = fmaf(v0, v0, fmaf(v1, v1, fmaf(v2, v2, fmaf(v3, v3, cn))));
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) cn += __shfl_xor_sync(0xffffffffu, cn, off);
  if (lane == 0) corrn[k] = sqrtf(cn) * 1.0009765625f;
}

// ---- preconditioned directions ---------------------------------------------
// FP64 mode: d = delta .* h + U g for a block of 32 walkers x 128 coordinates: the
// block draws the 32 walkers' low-rank normals g (Philox stream 2, Box-Muller as in
// Section 4.3) into shared memory; each thread keeps its coordinate's row of U
// in registers and walks the 32 walkers (coalesced along coordinates).
// In place on the normals.  The projection (when m_E > 0) follows on the result.
constexpr int kPcWalkers = 32;
constexpr int kPcThreads = 128;

__global__ void __launch_bounds__(kPcThreads)
precondition_kernel(uint64_t seed, const uint64_t* step_ptr, int j, uint32_t walker0, int z,
                    int n, int n_ld, int rank, const double* __restrict__ delta,
                    const double* __restrict__ U, double* D) {
  __shared__ double g[kPcWalkers][kMaxPcRank + 1];
  const int k0 = blockIdx.y * kPcWalkers;
  for (int t = threadIdx.x; t < kPcWalkers * (kMaxPcRank + 1); t += kPcThreads)
    g[t / (kMaxPcRank + 1)][t % (kMaxPcRank + 1)] = 0.0;
  __syncthreads();
  const uint64_t step = *step_ptr + static_cast<uint64_t>(j);
  const int quads = (rank + 3) >> 2;
  for (int t = threadIdx.x; t < kPcWalkers * quads; t += kPcThreads) {
    const int w = t / quads, q = t - (t / quads) * quads;
    if (k0 + w >= z) continue;
    const U4 r = philox_block(seed, step, walker0 + static_cast<uint32_t>(k0 + w),
                              static_cast<uint32_t>(q), kStreamLowRank);
    double v[4];
    box_muller_f64(r.x, r.y, v[0], v[1]);
    box_muller_f64(r.z, r.w, v[2], v[3]);
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (4 * q + e < rank) g[w][4 * q + e] = v[e];
  }
  __syncthreads();
  const int i = blockIdx.x * kPcThreads + threadIdx.x;
  if (i >= n) return;
  double u[kMaxPcRank];
#pragma unroll
  for (int c = 0; c < kMaxPcRank; ++c) u[c] = U[static_cast<size_t>(i) * kMaxPcRank + c];
  const double di = delta[i];
  const int wend = min(kPcWalkers, z - k0);
  for (int w = 0; w < wend; ++w) {
    const int k = k0 + w;
    double acc = di * D[static_cast<size_t>(k) * n_ld + i];
#pragma unroll
    for (int c = 0; c < kMaxPcRank; ++c) acc = fma(u[c], g[w][c], acc);
    D[static_cast<size_t>(k) * n_ld + i] = acc;
  }
}

// FP32 and tensor-core modes: the draw and d = delta .* h + U g in one kernel, into
// the FP16 pair as d_i / sigma_i (split), or into D32.  A block takes 64 walkers and
// a range of 64-coordinate tiles: the walkers' g once in shared memory, U
// transposed a tile at a time; a thread draws one quad of coordinates for each of
// four walkers and keeps the sixteen sums, so a step of four columns reads eight
// 16-byte words for 64 FMAs.  Bound by instruction issue (the Philox words and
// Box-Muller transforms, then the FMAs).  Two kernels, the normals through memory and a
// load for each FMA, took 21 + 76 us on illcond500x10000 (z = 16384, rank 32);
// this one 43 (three blocks an SM: 79 registers).
constexpr int kDpWalkers = 64;
constexpr int kDpTile = 64;
constexpr int kDpThreads = 256;      // 16 quads x 16 groups of four walkers

__global__ void __launch_bounds__(kDpThreads, 3)
draw_precondition_kernel(uint64_t seed, const uint64_t* step_ptr, int j, uint32_t walker0, int z,
                         int n, int n_ld, int rank, int tiles_per_block,
                         const float* __restrict__ delta, const float* __restrict__ U, float* D32,
                         int split, int k_pad, int z_ld, int inter, const float* __restrict__ sigma,
                         __half* Dh, __half* Dl, __half* Dh1, __half* Dl1, int* status) {
  __shared__ __align__(16) float g[kDpWalkers][kMaxPcRank];
  __shared__ __align__(16) float ut[kMaxPcRank][kDpTile + 4];   // U^T of the tile
  const uint64_t step = *step_ptr + static_cast<uint64_t>(j);
  if (Dh1 != nullptr && (step & 1ull)) {
    Dh = Dh1;  // recompute mode: iteration s's pair is s % 2
    Dl = Dl1;
  }
  const int tid = threadIdx.x, k0 = blockIdx.y * kDpWalkers;
  for (int t = tid; t < kDpWalkers * (kMaxPcRank / 4); t += kDpThreads) {
    const int w = t / (kMaxPcRank / 4), q = t % (kMaxPcRank / 4);
    float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    if (4 * q < rank && k0 + w < z) {
      const U4 r = philox_block(seed, step, walker0 + static_cast<uint32_t>(k0 + w),
                                static_cast<uint32_t>(q), kStreamLowRank);
      box_muller_f32(r.x, r.y, v[0], v[1]);
      box_muller_f32(r.z, r.w, v[2], v[3]);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) g[w][4 * q + e] = 4 * q + e < rank ? v[e] : 0.0f;
  }
  const int q = tid & 15, wg = 4 * (tid >> 4);
  const int t_end = min((n + kDpTile - 1) / kDpTile, static_cast<int>(blockIdx.x + 1) * tiles_per_block);
  for (int t = blockIdx.x * tiles_per_block; t < t_end; ++t) {
    const int i0 = t * kDpTile;
    __syncthreads();      // g is ready; the tile before is done with
    for (int e = tid; e < kDpTile * kMaxPcRank; e += kDpThreads) {
      const int i = i0 + (e >> 5);
      ut[e & 31][e >> 5] = i < n ? U[static_cast<size_t>(i) * kMaxPcRank + (e & 31)] : 0.0f;
    }
    __syncthreads();
    const int i = i0 + 4 * q;
    if (i >= n) continue;
    float acc[4][4], dl[4], is[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      dl[e] = i + e < n ? delta[i + e] : 0.0f;
      is[e] = split && i + e < n ? pow2_recip(sigma[i + e]) : 1.0f;
    }
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const U4 r = philox_block(seed, step, walker0 + static_cast<uint32_t>(k0 + wg + w),
                                static_cast<uint32_t>(i >> 2), kStreamDirection);
      box_muller_f32(r.x, r.y, acc[w][0], acc[w][1]);
      box_muller_f32(r.z, r.w, acc[w][2], acc[w][3]);
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[w][e] *= dl[e];
    }
#pragma unroll 2
    for (int c = 0; c < rank; c += 4) {        // g and U are 0 past the rank
      float4 gv[4];
#pragma unroll
      for (int w = 0; w < 4; ++w) gv[w] = *reinterpret_cast<const float4*>(&g[wg + w][c]);
#pragma unroll
      for (int cc = 0; cc < 4; ++cc) {
        const float4 u = *reinterpret_cast<const float4*>(&ut[c + cc][4 * q]);
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          const float gc = cc == 0 ? gv[w].x : cc == 1 ? gv[w].y : cc == 2 ? gv[w].z : gv[w].w;
          acc[w][0] = fmaf(u.x, gc, acc[w][0]);
          acc[w][1] = fmaf(u.y, gc, acc[w][1]);
          acc[w][2] = fmaf(u.z, gc, acc[w][2]);
          acc[w][3] = fmaf(u.w, gc, acc[w][3]);
        }
      }
    }
    // n_ld and k_pad are multiples of four: the quad's padding is 0 and stays so.
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const int k = k0 + wg + w;
      if (k >= z) continue;
      if (split) {
        __half2 h[2], l[2];
        bool bad = false;
#pragma unroll
        for (int e = 0; e < 4; e += 2) {
          const float a = i + e < n ? acc[w][e] * is[e] : 0.0f;
          const float b = i + e + 1 < n ? acc[w][e + 1] * is[e + 1] : 0.0f;
          h[e / 2] = __floats2half2_rn(a, b);
          l[e / 2] = __floats2half2_rn(a - __low2float(h[e / 2]), b - __high2float(h[e / 2]));
          bad |= !(fabsf(a) <= kHalfMax) || !(fabsf(b) <= kHalfMax);
        }
        if (bad) atomicOr(status, MHAR_ST_NONFINITE);
        const size_t o = op_off(k, i, k_pad, z_ld, inter);
        *reinterpret_cast<uint2*>(Dh + o) = *reinterpret_cast<const uint2*>(h);
        *reinterpret_cast<uint2*>(Dl + o) = *reinterpret_cast<const uint2*>(l);
      } else {
        *reinterpret_cast<float4*>(D32 + static_cast<size_t>(k) * n_ld + i) =
            make_float4(acc[w][0], i + 1 < n ? acc[w][1] : 0.0f, i + 2 < n ? acc[w][2] : 0.0f,
                        i + 3 < n ? acc[w][3] : 0.0f);
      }
    }
  }
}

// ---- Section 4.4: line sets, recompute formulation ---------------------------
template <typename T>
struct ChordTile;
template <>
struct ChordTile<double> { static constexpr int BK = 8; };
template <>
struct ChordTile<float> { static constexpr int BK = 16; };

// Rounding-error margins of the FP32 chord (unit roundoff u = 2^-24): with
// sigma the power-of-two column scales of A,
//   |computed - exact| of b_i - a_i . x  <=  e(x) + 3 u |b_i|
//   |computed - exact| of a_i . d        <=  e(d)
//   e(v) = min(K_i,2 ||v / sigma||_2, K_i,1 max |v_j / sigma_j|)
// where K_i,p = gamma_{nnz_i + 4} ||a_i sigma||_p (gamma_k = k u / (1 - k u):
// the roundings of A, x, the products and sums over the row's nonzeros, and
// the ratio; Hoelder on |a_i| . |v|).  The kernels take b already lowered by
// 3 u |b_i| and kr = (K_i,2, K_i,1); the per-walker norms are computed here,
// rounded up.  FP64 passes kr = NULL: its rounding (gamma ~ 1e-13 for n = 1000)
// is far inside the 1e-6 feasibility tolerance, and no margin keeps the FP64
// walk equal to the exact one to the last bits the parity tests see.
template <typename T>
struct Unit;
template <>
struct Unit<double> { static constexpr double guard = 1.0 + 1e-12; };
template <>
struct Unit<float> { static constexpr float guard = 1.0009765625f; };

template <typename T>
__global__ void __launch_bounds__(kThreads)
chord_simt_kernel(const T* __restrict__ A, const T* __restrict__ b, const T* __restrict__ kr,
                  const T* __restrict__ X, const T* __restrict__ D, const float* __restrict__ sigma,
                  const float* __restrict__ corrn, int m, int n_ld, int z,
                  unsigned long long* key_lo, unsigned long long* key_hi, int* status) {
  constexpr int BK = ChordTile<T>::BK;
  constexpr int kRowsPerThread = 64 * BK / kThreads;   // walker rows each thread loads
  __shared__ T As[BK][64];
  __shared__ T Xs[BK][64];
  __shared__ T Ds[BK][64];
  __shared__ T red_lo[16][64];
  __shared__ T red_hi[16][64];
  __shared__ T nrm[4][64];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int i0 = blockIdx.x * 64, w0 = blockIdx.y * 64;
  T accS[4][4], accG[4][4];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) { accS[r][c] = T(0); accG[r][c] = T(0); }
  // Sums of (x_i / sigma_i)^2, (d_i / sigma_i)^2 of the walker rows this
  // thread loads (column tid % BK of each tile).
  T sx[kRowsPerThread], sd[kRowsPerThread], mxx[kRowsPerThread], mxd[kRowsPerThread];
#pragma unroll
  for (int j = 0; j < kRowsPerThread; ++j) { sx[j] = T(0); sd[j] = T(0); mxx[j] = T(0); mxd[j] = T(0); }

  for (int k0 = 0; k0 < n_ld; k0 += BK) {
    const T isig = T(1) / static_cast<T>(sigma[k0 + tid % BK]);   // a power of two: exact
#pragma unroll
    for (int j = 0; j < kRowsPerThread; ++j) {
      const int e = tid + j * kThreads;
      const int r = e / BK, c = e - r * BK;
      const int gi = i0 + r, gw = w0 + r;
      As[c][r] = gi < m ? A[static_cast<size_t>(gi) * n_ld + k0 + c] : T(0);
      const T xv = gw < z ? X[static_cast<size_t>(gw) * n_ld + k0 + c] : T(0);
      const T dv = gw < z ? D[static_cast<size_t>(gw) * n_ld + k0 + c] : T(0);
      Xs[c][r] = xv;
      Ds[c][r] = dv;
      if (kr != nullptr) {
        const T xs = xv * isig, ds = dv * isig;
        sx[j] += xs * xs;
        sd[j] += ds * ds;
        mxx[j] = fmax(mxx[j], fabs(xs));
        mxd[j] = fmax(mxd[j], fabs(ds));
      }
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      T a[4], xv[4], dv[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) a[r] = As[kk][ty * 4 + r];
#pragma unroll
      for (int c = 0; c < 4; ++c) { xv[c] = Xs[kk][tx + 16 * c]; dv[c] = Ds[kk][tx + 16 * c]; }
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          accS[r][c] += a[r] * xv[c];
          accG[r][c] += a[r] * dv[c];
        }
    }
    __syncthreads();
  }
  // Each walker row's sums are spread over BK consecutive lanes: add them
  // with a butterfly (every lane gets the same bits).
#pragma unroll
  for (int j = 0; j < kRowsPerThread; ++j) {
#pragma unroll
    for (int off = BK / 2; off > 0; off >>= 1) {
      sx[j] += __shfl_xor_sync(0xffffffffu, sx[j], off);
      sd[j] += __shfl_xor_sync(0xffffffffu, sd[j], off);
      mxx[j] = fmax(mxx[j], __shfl_xor_sync(0xffffffffu, mxx[j], off));
      mxd[j] = fmax(mxd[j], __shfl_xor_sync(0xffffffffu, mxd[j], off));
    }
    if (tid % BK == 0) {
      const int r = (tid + j * kThreads) / BK;
      nrm[0][r] = sqrt(sx[j]) * Unit<T>::guard;
      nrm[1][r] = sqrt(sd[j]) * Unit<T>::guard;
      nrm[2][r] = mxx[j];
      nrm[3][r] = mxd[j];
    }
  }
  __syncthreads();

  bool bad = false;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    T lo = static_cast<T>(neg_inf()), hi = static_cast<T>(pos_inf());
    const int w = tx + 16 * c;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int gi = i0 + ty * 4 + r;
      if (gi >= m) continue;
      T s = b[gi] - accS[r][c];
      T g = accG[r][c];
      if (kr != nullptr) {
        const T k2 = kr[3 * gi], k1 = kr[3 * gi + 1];
        s -= fmin(k2 * nrm[0][w], k1 * nrm[2][w]);
        T eg = fmin(k2 * nrm[1][w], k1 * nrm[3][w]);
        if (corrn != nullptr && w0 + w < z) eg += kr[3 * gi + 2] * static_cast<T>(corrn[w0 + w]);
        g = g > T(0) ? g + eg : (g < T(0) ? g - eg : g);
      }
      if (!isfinite(s) || !isfinite(g)) { bad = true; continue; }
      if (s < T(0)) s = T(0);
      if (g > T(0)) {
        const T lam = s / g;
        hi = lam < hi ? lam : hi;
      } else if (g < T(0)) {
        const T lam = s / g;
        lo = lam > lo ? lam : lo;
      }
    }
    red_lo[ty][tx + 16 * c] = lo;
    red_hi[ty][tx + 16 * c] = hi;
  }
  __syncthreads();
  if (tid < 64) {
    T lo = red_lo[0][tid], hi = red_hi[0][tid];
#pragma unroll
    for (int t = 1; t < 16; ++t) {
      lo = red_lo[t][tid] > lo ? red_lo[t][tid] : lo;
      hi = red_hi[t][tid] < hi ? red_hi[t][tid] : hi;
    }
    const int gw = w0 + tid;
    if (gw < z) {
      if (!isinf(lo)) atomicMax(&key_lo[gw], f64_key(static_cast<double>(lo)));
      if (!isinf(hi)) atomicMin(&key_hi[gw], f64_key(static_cast<double>(hi)));
    }
  }
  if (bad) atomicOr(status, MHAR_ST_NONFINITE);
}

// ---- Section 4.5: theta on the chord, x += theta d ---------------------------
// mode 0: FP64 points; mode 1: FP32-pair points with FP32 directions.
__global__ void update_kernel(int mode, uint64_t seed, const uint64_t* step_ptr, int j,
                              uint32_t walker0, int z, int n, int n_ld,
                              unsigned long long* key_lo, unsigned long long* key_hi,
                              double* lmin, double* lmax, double* theta, int* status,
                              unsigned long long* counters, double* X64, const double* D64,
                              float* Xhi, float* Xlo, const float* D32, int mE,
                              const float* Q32, const float* corr) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k = blockIdx.x * (kThreads / 32) + warp;
  if (k >= z) return;
  double t = 0.0;
  if (lane == 0) {
    const double L = f64_unkey(key_lo[k]);
    const double H = f64_unkey(key_hi[k]);
    key_lo[k] = f64_key(neg_inf());
    key_hi[k] = f64_key(pos_inf());
    if (isinf(L) || isinf(H)) {
      atomicOr(status, MHAR_ST_UNBOUNDED);
      atomicAdd(&counters[1], 1ull);
    } else if (L > H) {
      atomicOr(status, MHAR_ST_STALL);
      atomicAdd(&counters[0], 1ull);
    } else {
      const uint64_t step = *step_ptr + static_cast<uint64_t>(j);
      const U4 w = philox_block(seed, step, walker0 + static_cast<uint32_t>(k), 0u, kStreamChord);
      const double u = open_unit_f64(w.x);
      t = L + u * (H - L);
      if (mode != 0) t = static_cast<double>(static_cast<float>(t));
    }
    lmin[k] = L;
    lmax[k] = H;
    theta[k] = t;
  }
  t = __shfl_sync(0xffffffffu, t, 0);
  const size_t row = static_cast<size_t>(k) * n_ld;
  if (mode == 0) {
    for (int i = lane; i < n; i += 32) X64[row + i] += t * D64[row + i];
  } else {
    const float tf = static_cast<float>(t);
    for (int i = lane; i < n; i += 32) df_axpy(Xhi[row + i], Xlo[row + i], tf, D32[row + i]);
    if (corr != nullptr && tf != 0.0f) {
      for (int i = lane; i < n; i += 32) {
        float dlt = 0.0f;
        for (int e = 0; e < mE; ++e)
          dlt = fmaf(Q32[static_cast<size_t>(e) * n_ld + i], corr[static_cast<size_t>(k) * mE + e], dlt);
        Xlo[row + i] = fmaf(-tf, dlt, Xlo[row + i]);
      }
    }
  }
}

// Recompute mode: the walkers' operands for iteration s = step + j, built
// from the host-visible state (after creation, set_state or a new
// preconditioner; afterwards each chord kernel leaves them in place):
//  (2) split each point into the FP16 pair of the tensor-core operand, as
//      x_i / (sigma_i 2^e) with 2^e a power of two such that
//      max_i |x_i| / sigma_i 2^-e lies in [0.5, 1);
//  (3) draw iteration s's directions (Section 4.3): into FP16 pair s % 2
//      directly when neither a projection nor a preconditioner follows, else
//      into the FP32 scratch those kernels read.
// `flags`: bit 1 split, bit 2 draw.
// Layout: 32 walkers per block, one per lane; each warp takes 8-coordinate
// chunks (warp, warp + warps, ...).  A thread reads and writes whole chunks:
// 32 B of each FP32 row and 16 B of each FP16 operand, so in the interleaved
// operand layout a warp's 32 walkers fill one contiguous 512-byte line.
constexpr int kPrepWalkers = 32;
constexpr int kPrepMaxWarps = 16;

__device__ __forceinline__ void ld8(const float* p, float* v) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  const float4 b = *reinterpret_cast<const float4*>(p + 4);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void st8(float* p, const float* v) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  *reinterpret_cast<float4*>(p + 4) = make_float4(v[4], v[5], v[6], v[7]);
}
__device__ __forceinline__ uint32_t pack2h(__half a, __half b) {
  return static_cast<uint32_t>(__half_as_ushort(a)) |
         (static_cast<uint32_t>(__half_as_ushort(b)) << 16);
}
__device__ __forceinline__ void st8h(__half* p, const __half* h) {
  *reinterpret_cast<uint4*>(p) =
      make_uint4(pack2h(h[0], h[1]), pack2h(h[2], h[3]), pack2h(h[4], h[5]), pack2h(h[6], h[7]));
}

__global__ void __launch_bounds__(kPrepMaxWarps * 32)
prep_walkers_kernel(int flags, uint64_t seed, const uint64_t* step_ptr, int j, uint32_t walker0,
                    int z, int z_ld, int n, int n_ld, int k_pad, const float* Xhi,
                    const float* Xlo, __half* Dh0, __half* Dl0, __half* Dh1, __half* Dl1,
                    float* D32, __half* Xh, __half* Xl, float* wscale, int inter,
                    const float* sigma, int draw32, int* status) {
  __shared__ float red[kPrepMaxWarps][kPrepWalkers];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarps = blockDim.x >> 5;
  const int k = blockIdx.x * kPrepWalkers + lane;
  const bool live = k < z;
  const int chunks = (n + 7) >> 3;
  const size_t xr = static_cast<size_t>(k) * n_ld;
  const uint64_t step = *step_ptr + static_cast<uint64_t>(j);
  __half* Dh = (Dh1 != nullptr && (step & 1ull)) ? Dh1 : Dh0;
  __half* Dl = (Dl1 != nullptr && (step & 1ull)) ? Dl1 : Dl0;
  auto opo = [&](int i) { return op_off(k, i, k_pad, z_ld, inter); };

  // (2) the walker's largest scaled coordinate, then its FP16 pair.
  if (flags & 2) {
    float mx = 0.0f;
    if (live)
      for (int c = warp; c < chunks; c += nwarps) {
        float hi[8];
        ld8(Xhi + xr + 8 * c, hi);
#pragma unroll
        for (int e = 0; e < 8; ++e)
          if (8 * c + e < n) mx = fmaxf(mx, fabsf(hi[e]) * pow2_recip(sigma[8 * c + e]));
      }
    red[warp][lane] = mx;
    __syncthreads();
    if (live) {
      for (int w = 0; w < nwarps; ++w) mx = fmaxf(mx, red[w][lane]);
      int ex = 0;
      if (mx > 0.0f) frexpf(mx, &ex);
      const float inv = ldexpf(1.0f, -ex);
      if (warp == 0) wscale[k] = ldexpf(1.0f, ex);
      for (int c = warp; c < chunks; c += nwarps) {
        const int i0 = 8 * c;
        float hi[8], lo[8];
        ld8(Xhi + xr + i0, hi);
        ld8(Xlo + xr + i0, lo);
        __half h8[8], l8[8];
        bool bad = false;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const int i = i0 + e;
          const float v = i < n ? (hi[e] + lo[e]) * inv * pow2_recip(sigma[i]) : 0.0f;
          h8[e] = __float2half_rn(v);
          l8[e] = __float2half_rn(v - __half2float(h8[e]));
          bad |= !(fabsf(v) <= kHalfMax);
        }
        if (bad) atomicOr(status, MHAR_ST_NONFINITE);
        st8h(Xh + opo(i0), h8);
        st8h(Xl + opo(i0), l8);
      }
    }
  }

  // (3) directions: quads 2c and 2c + 1 of each chunk.
  if ((flags & 4) && live) {
    for (int c = warp; c < chunks; c += nwarps) {
      const int i0 = 8 * c;
      float v[8];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (i0 + 4 * h < n) {
          const U4 w = philox_block(seed, step, walker0 + static_cast<uint32_t>(k),
                                    static_cast<uint32_t>(2 * c + h), kStreamDirection);
          box_muller_f32(w.x, w.y, v[4 * h], v[4 * h + 1]);
          box_muller_f32(w.z, w.w, v[4 * h + 2], v[4 * h + 3]);
        } else {
          v[4 * h] = v[4 * h + 1] = v[4 * h + 2] = v[4 * h + 3] = 0.0f;
        }
      }
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (i0 + e >= n) v[e] = 0.0f;
      if (!draw32) {
        __half h8[8], l8[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float vs = v[e] * pow2_recip(sigma[i0 + e]);   // d_i / sigma_i, exact
          h8[e] = __float2half_rn(vs);
          l8[e] = __float2half_rn(vs - __half2float(h8[e]));
        }
        st8h(Dh + opo(i0), h8);
        st8h(Dl + opo(i0), l8);
      } else {
        st8(D32 + xr + i0, v);
      }
    }
  }
}

__global__ void advance_kernel(uint64_t* step_ptr, int steps) { *step_ptr += steps; }

__global__ void advance_many_kernel(uint64_t* const* steps, int count, int by) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) *steps[i] += static_cast<uint64_t>(by);
}

__global__ void emit_kernel(int mode, int z, int n, int n_ld, const double* X64, const float* Xhi,
                            const float* Xlo, double* out) {
  const long long idx = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx >= static_cast<long long>(z) * n) return;
  const int k = static_cast<int>(idx / n), i = static_cast<int>(idx - static_cast<long long>(k) * n);
  const size_t src = static_cast<size_t>(k) * n_ld + i;
  out[idx] = mode == 0 ? X64[src] : static_cast<double>(Xhi[src]) + static_cast<double>(Xlo[src]);
}

// A batch: the samples of up to kBatchEmit problems (grid.y) in one launch, and
// every problem's status words cleared or gathered (a launch, and a copy, of its
// own for each of 48 problems took 350 us of a call).
__global__ void batch_emit_kernel(const BatchProblem* __restrict__ probs, const BatchOuts outs) {
  const BatchProblem p = probs[blockIdx.y];
  double* out = outs.out[blockIdx.y];
  if (out == nullptr) return;
  const long long count = static_cast<long long>(p.walkers) * p.n;
  for (long long idx = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; idx < count;
       idx += static_cast<long long>(gridDim.x) * blockDim.x) {
    const int k = static_cast<int>(idx / p.n), i = static_cast<int>(idx - static_cast<long long>(k) * p.n);
    const size_t src = static_cast<size_t>(k) * p.n_ld + i;
    out[idx] = static_cast<double>(p.Xhi[src]) + static_cast<double>(p.Xlo[src]);
  }
}

// Clearing also zeroes the arrival counters of cut strips: after an expired wait some
// stand part of the way.
__global__ void batch_status_kernel(const BatchProblem* __restrict__ probs, int count, int2* gather,
                                    const BatchCounters counters) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  for (int i = 0; gather == nullptr && i < counters.sets; ++i)
    for (int t = q; t < counters.count[i]; t += gridDim.x * blockDim.x) counters.at[i][t] = 0;
  if (q >= count) return;
  int* st = probs[q].status;
  if (gather != nullptr) {
    gather[q] = make_int2(st[0], st[1]);
  } else {
    st[0] = 0;
    st[1] = 0;
  }
}

__global__ void set_points_kernel(int mode, int z, int n, int n_ld, const double* Xin, double* X64,
                                  float* Xhi, float* Xlo) {
  const long long idx = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx >= static_cast<long long>(z) * n) return;
  const int k = static_cast<int>(idx / n), i = static_cast<int>(idx - static_cast<long long>(k) * n);
  const size_t dst = static_cast<size_t>(k) * n_ld + i;
  const double v = Xin[idx];
  if (mode == 0) {
    X64[dst] = v;
  } else {
    const float h = static_cast<float>(v);
    Xhi[dst] = h;
    Xlo[dst] = static_cast<float>(v - static_cast<double>(h));
  }
}

__device__ __forceinline__ double load_point(int mode, const double* X64, const float* Xhi,
                                             const float* Xlo, size_t idx) {
  return mode == 0 ? X64[idx] : static_cast<double>(Xhi[idx]) + static_cast<double>(Xlo[idx]);
}

// FP64 feasibility check: max over (walker, row) of a_i x - b_i, and
// max over walkers of |A_E x - b_E|_inf.
//
// Only one number leaves the check, so FP64 (1/64 of the FP32 rate on this
// GPU) is spent on the rows that can hold it:
//  (1) check_screen_kernel forms v = a_i . x - b_i in FP32 with a bound e on
//      its error, keeps the largest v + e of each (row tile, walker), and
//      folds v - e into the largest value some row certainly reaches;
//  (2) check_exact_kernel evaluates in FP64, row by row in index order, the
//      tiles whose v + e reaches that value -- a handful of them -- and folds
//      s - b_i into the result.  A value FP32 cannot bound (overflow, NaN)
//      counts as reaching it.
// The screen is the standard FP32 bound (Higham, Accuracy and Stability,
// Section 3.1; u = 2^-24): e = gamma_{n+10} ||a_i||_2 ||x||_2 + 4 u |b_i|,
// gamma_k = k u / (1 - k u), the truncations of A and x (2 u each), the roundings
// of the products, the sums and the comparison among its k; it takes nothing
// from the walk's own error margins, which the check is there to verify.  Squares of entries below
// 2^-75 leave the FP32 norms: kNormFloor per entry covers them.
// A thread per (row, walker) in FP64, with an atomic each, took 5.35 ms for
// 4096 walkers of a 2000 x 100 body and 1.39 ms for 1024 of them (ncu); the
// two kernels took 109 + 45 us for the 4096 while the screen's conversions from
// FP64 cost as much as its products and a warp evaluated a whole tile;
// 80 + 16 us now.
constexpr int kChkRows = 128;      // rows of a tile
constexpr int kChkWalkers = 64;    // walkers of a tile
constexpr int kChkK = 16;
constexpr float kNormFloor = 1e-22f;

__device__ __forceinline__ unsigned int f32_key(float f) {
  const unsigned int u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float f32_unkey(unsigned int k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// v truncated to FP32 in integer arithmetic (a conversion takes the FP64 pipe 16
// clocks a warp); below the normal range 0, above it as converted.
__device__ __forceinline__ float f32_truncated(double v) {
  const unsigned int hi = static_cast<unsigned int>(__double2hiint(v));
  const unsigned int lo = static_cast<unsigned int>(__double2loint(v));
  const unsigned int e = hi & 0x7ff00000u;
  if (e > 0x47e00000u) return static_cast<float>(v);
  const unsigned int f = (hi & 0x80000000u) | (((hi & 0x7fffffffu) - 0x38000000u) << 3) | (lo >> 29);
  return e >= 0x38100000u ? __uint_as_float(f) : 0.0f;
}

// blockIdx.x: group of `group` consecutive row tiles, blockIdx.y: 64 walkers.
// ub[blockIdx.x * walkers + k]; best: key of the largest certain value.
__global__ void __launch_bounds__(kThreads)
check_screen_kernel(int mode, int m, int n, int n_ld, int walkers, int group,
                    const double* __restrict__ A, const double* __restrict__ b,
                    const double* __restrict__ X64, const float* __restrict__ Xhi,
                    const float* __restrict__ Xlo, float* __restrict__ ub, unsigned int* best) {
  __shared__ __align__(16) float As[kChkK][kChkRows + 4];
  __shared__ __align__(16) float Xs[kChkK][kChkWalkers + 4];
  __shared__ float an[kChkRows], xn[kChkWalkers], red[16][kChkWalkers];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int w0 = blockIdx.y * kChkWalkers;
  const float gam = static_cast<float>(n + 10) * 0x1p-24f /
                    (1.0f - static_cast<float>(n + 10) * 0x1p-24f) * 1.0009765625f;
  const float floor_n = static_cast<float>(n) * kNormFloor;
  float up[4], low = -INFINITY;
#pragma unroll
  for (int c = 0; c < 4; ++c) up[c] = -INFINITY;
  const int xw = tid >> 2, xk = (tid & 3) * 4;   // this thread's part of a walker tile
  const bool xin = w0 + xw < walkers;
  for (int g = 0; g < group; ++g) {
    const int i0 = (blockIdx.x * group + g) * kChkRows;
    if (i0 >= m) break;
    float acc[8][4];
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[r][c] = 0.0f;
    float sa[4] = {0.0f, 0.0f, 0.0f, 0.0f}, sx = 0.0f;
    // The next K step's part of both tiles is on its way during the products.
    double2 av[4];
    double2 xd[2];
    float4 xh, xl;
    auto fetch = [&](int k0) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int r = (tid >> 3) + 32 * j, c = (tid & 7) * 2;
        av[j] = make_double2(0.0, 0.0);
        if (i0 + r < m)
          av[j] = *reinterpret_cast<const double2*>(A + static_cast<size_t>(i0 + r) * n_ld + k0 + c);
      }
      xd[0] = xd[1] = make_double2(0.0, 0.0);
      xh = xl = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (xin) {
        const size_t o = static_cast<size_t>(w0 + xw) * n_ld + k0 + xk;
        if (mode == 0) {
          xd[0] = *reinterpret_cast<const double2*>(X64 + o);
          xd[1] = *reinterpret_cast<const double2*>(X64 + o + 2);
        } else {
          xh = *reinterpret_cast<const float4*>(Xhi + o);
          xl = *reinterpret_cast<const float4*>(Xlo + o);
        }
      }
    };
    fetch(0);
    for (int k0 = 0; k0 < n_ld; k0 += kChkK) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int r = (tid >> 3) + 32 * j, c = (tid & 7) * 2;
        const float f0 = f32_truncated(av[j].x), f1 = f32_truncated(av[j].y);
        As[c][r] = f0;
        As[c + 1][r] = f1;
        sa[j] = fmaf(f0, f0, fmaf(f1, f1, sa[j]));
      }
      float xv[4];
      if (mode == 0) {
        xv[0] = f32_truncated(xd[0].x); xv[1] = f32_truncated(xd[0].y);
        xv[2] = f32_truncated(xd[1].x); xv[3] = f32_truncated(xd[1].y);
      } else {
        xv[0] = xh.x + xl.x; xv[1] = xh.y + xl.y; xv[2] = xh.z + xl.z; xv[3] = xh.w + xl.w;
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        Xs[xk + e][xw] = xv[e];
        sx = fmaf(xv[e], xv[e], sx);
      }
      if (k0 + kChkK < n_ld) fetch(k0 + kChkK);
      __syncthreads();
#pragma unroll
      for (int kk = 0; kk < kChkK; ++kk) {
        const float4 a0 = *reinterpret_cast<const float4*>(&As[kk][ty * 8]);
        const float4 a1 = *reinterpret_cast<const float4*>(&As[kk][ty * 8 + 4]);
        const float4 xq = *reinterpret_cast<const float4*>(&Xs[kk][tx * 4]);
        const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
        const float x[4] = {xq.x, xq.y, xq.z, xq.w};
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[r][c] = fmaf(a[r], x[c], acc[r][c]);
      }
      __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
      for (int off = 4; off > 0; off >>= 1) sa[j] += __shfl_xor_sync(0xffffffffu, sa[j], off);
      if ((tid & 7) == 0) an[(tid >> 3) + 32 * j] = sqrtf(sa[j]) * 1.0009765625f + floor_n;
    }
#pragma unroll
    for (int off = 2; off > 0; off >>= 1) sx += __shfl_xor_sync(0xffffffffu, sx, off);
    if ((tid & 3) == 0) xn[xw] = sqrtf(sx) * 1.0009765625f + floor_n;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int gi = i0 + ty * 8 + r;
      if (gi >= m) continue;
      const float bf = static_cast<float>(b[gi]), ga = gam * an[ty * 8 + r];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if (w0 + tx * 4 + c >= walkers) continue;
        const float v = acc[r][c] - bf;
        // 1e-36: products and b's below the normal FP32 range.
        const float e = fmaf(ga, xn[tx * 4 + c], fmaf(0x1p-22f, fabsf(bf) + fabsf(v), 1e-36f));
        const float hi = v + e, lo = v - e;
        up[c] = hi < INFINITY ? fmaxf(up[c], hi) : INFINITY;   // not below +Inf, NaN too
        if (fabsf(lo) < INFINITY) low = fmaxf(low, lo);
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) red[ty][tx * 4 + c] = up[c];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) low = fmaxf(low, __shfl_xor_sync(0xffffffffu, low, off));
  __syncthreads();
  if (tid < kChkWalkers && w0 + tid < walkers) {
    float u = red[0][tid];
#pragma unroll
    for (int t = 1; t < 16; ++t) u = fmaxf(u, red[t][tid]);
    ub[static_cast<size_t>(blockIdx.x) * walkers + w0 + tid] = u;
  }
  if ((tid & 31) == 0) atomicMax(best, f32_key(low));
}

// The FP64 values of the tiles the screen left: a block looks at kChkEntries
// entries of ub and takes those at or above the certain value one at a time, a
// thread per row, the point staged once as FP64.  (A warp an entry with four rows a
// lane, the point converted by every lane: 22 us each.  Few entries a block: sparse
// bodies with many slacks near the least leave most of them.)
constexpr int kChkEntries = 16;
constexpr int kChkStage = 512;     // columns of the point staged at once

__global__ void __launch_bounds__(kChkRows)
check_exact_kernel(int mode, int m, int n, int n_ld, int walkers, int group,
                   const double* __restrict__ A, const double* __restrict__ b,
                   const double* __restrict__ X64, const float* __restrict__ Xhi,
                   const float* __restrict__ Xlo, const float* __restrict__ ub,
                   const unsigned int* __restrict__ best, long long entries,
                   unsigned long long* out_key) {
  __shared__ __align__(16) double xs[kChkStage];
  const int lane = threadIdx.x & 31, tid = threadIdx.x;
  const long long e0 = static_cast<long long>(blockIdx.x) * kChkEntries;
  const float floor_v = f32_unkey(*best);
  const bool take = lane < kChkEntries && e0 + lane < entries && !(ub[e0 + lane] < floor_v);
  unsigned int todo = __ballot_sync(0xffffffffu, take);      // every warp the same
  while (todo) {
    const int t = __ffs(todo) - 1;
    todo &= todo - 1;
    const long long en = e0 + t;
    const int tile = static_cast<int>(en / walkers), k = static_cast<int>(en - static_cast<long long>(tile) * walkers);
    const size_t row = static_cast<size_t>(k) * n_ld;
    const int r1 = min(m, (tile + 1) * group * kChkRows);
    unsigned long long top = 0ull;
    for (int r0 = tile * group * kChkRows; r0 < r1; r0 += kChkRows) {
      const int r = r0 + tid;
      const double* a = A + static_cast<size_t>(min(r, m - 1)) * n_ld;
      double s = 0.0;                                        // in index order
      for (int c0 = 0; c0 < n; c0 += kChkStage) {
        const int c1 = min(n_ld - c0, kChkStage);            // zero past n
        __syncthreads();
        for (int i = tid; i < c1; i += kChkRows) xs[i] = load_point(mode, X64, Xhi, Xlo, row + c0 + i);
        __syncthreads();
        for (int i = 0; i < c1; i += 8) {                    // n_ld is a multiple of 32
          double2 av[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) av[q] = *reinterpret_cast<const double2*>(a + c0 + i + 2 * q);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            s += av[q].x * xs[i + 2 * q];
            s += av[q].y * xs[i + 2 * q + 1];
          }
        }
      }
      if (r < r1) top = max(top, f64_key(s - b[r]));
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, off));
    if (lane == 0) atomicMax(out_key, top);
  }
}

// Both parts in one launch, every (row, walker) in FP64: a block per (128 rows,
// walker).  Small checks (kCheckScreen products and below, or kCheckPairs rows times
// walkers; the equalities of the larger ones, with m = 0).  A call on 50 and more columns
// goes by the pairs: at 32000 of them 68 us against the screen's 68 (8000 x 50, 4 walkers),
// 71 / 73 (8000 x 100, 4), 105 / 108 (8000 x 300, 4), 192 / 210 (8000 x 1000, 4), at 64000
// 104 / 73 (8000 x 100, 8); all values equal, as before a chain's first step, 78 / 355
// (4000 x 300, 4).  On fewer columns equal values make the screen slow for longer.
constexpr long long kCheckScreen = 1ll << 22;
constexpr long long kCheckPairs = 1ll << 15;

__global__ void check_kernel(int mode, int m, int n, int n_ld, int mE, const double* A,
                             const double* b, const double* AE, const double* bE,
                             const double* X64, const float* Xhi, const float* Xlo,
                             unsigned long long* out_keys) {
  extern __shared__ double xs[];
  const int k = blockIdx.y;
  const size_t row = static_cast<size_t>(k) * n_ld;
  for (int i = threadIdx.x; i < n; i += blockDim.x) xs[i] = load_point(mode, X64, Xhi, Xlo, row + i);
  __syncthreads();
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r < m) {
    double s = 0.0;
    for (int i = 0; i < n; ++i) s += A[static_cast<size_t>(r) * n_ld + i] * xs[i];
    atomicMax(&out_keys[0], f64_key(s - b[r]));
  }
  if (blockIdx.x == 0 && r < mE) {
    double s = 0.0;
    for (int i = 0; i < n; ++i) s += AE[static_cast<size_t>(r) * n_ld + i] * xs[i];
    atomicMax(&out_keys[1], f64_key(fabs(s - bE[r])));
  }
}

// Stored-slack mode, after a refresh (one warp per walker): the bound
// ||x / sigma||_2 (1 + 2^-8) of the refreshed point, the step sum of the
// tracked slack's error reset, and the refresh's iteration recorded.
__global__ void stored_reset_kernel(int z, int n, int n_ld, const float* Xhi, const float* Xlo,
                                    const float* sigma, const uint64_t* step, float* nx_ref,
                                    float* theta_acc, uint64_t* refresh_step) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k = blockIdx.x * (blockDim.x >> 5) + warp;
  if (blockIdx.x == 0 && threadIdx.x == 0) *refresh_step = *step;
  if (k >= z) return;
  float ss = 0.0f;
  for (int i = lane; i < n; i += 32) {
    const size_t o = static_cast<size_t>(k) * n_ld + i;
    const float v = (Xhi[o] + Xlo[o]) / sigma[i];
    ss = fmaf(v, v, ss);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
  if (lane == 0) {
    nx_ref[k] = sqrtf(ss) * 1.00390625f;
    theta_acc[k] = 0.0f;
  }
}

// Mixed mode: S = b - A X recomputed in FP64 from the FP32-pair points (tiles
// of 64 rows x 64 walkers, K staged through shared memory), stored as the
// tensor-core path keeps it (divided by the row scale, blocked by 4 rows),
// and the largest change |S_old - S_new| recorded (drift).
// Small bodies: one warp per walker, lanes over the rows.  The tile kernel
// above keeps (m/64)(z/64) blocks busy, which for a body like the
// 10-dimensional cube is a couple of SMs; here every walker has its own warp,
// so the FP64 work (slow on this GPU) spreads over many SMs.  Same formulas:
// s = b - a.x, g = a.d, slack clamped at 0, rows with g == 0 skipped.  With
// `move` the warp also draws theta and moves its walker (update_kernel's
// arithmetic), so one launch does Sections 4.4 and 4.5.
constexpr int kWarpChordThreads = 128;

template <typename T>
__global__ void __launch_bounds__(kWarpChordThreads)
chord_warp_kernel(const T* __restrict__ A, const T* __restrict__ b, const T* __restrict__ kr,
                  const float* __restrict__ sigma, const float* __restrict__ corrn,
                  const T* __restrict__ X,
                  const T* __restrict__ D, int m, int n, int n_ld, int z,
                  unsigned long long* key_lo, unsigned long long* key_hi, int* status,
                  int move, uint64_t seed, const uint64_t* step_ptr, int j, uint32_t walker0,
                  double* lmin, double* lmax, double* theta, unsigned long long* counters,
                  double* X64, const double* D64, float* Xhi, float* Xlo, const float* D32,
                  int mE, const float* Q32, const float* corr) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k = blockIdx.x * (kWarpChordThreads / 32) + warp;
  if (k >= z) return;
  const T* x = X + static_cast<size_t>(k) * n_ld;
  const T* d = D + static_cast<size_t>(k) * n_ld;
  // ||x / sigma||_2 and ||d / sigma||_2 of the walker (the margins of
  // chord_simt_kernel); the butterfly gives every lane the same bits.
  T nx = T(0), nd = T(0), ix = T(0), id = T(0);
  if (kr != nullptr) {
    for (int c = lane; c < n; c += 32) {
      const T is = T(1) / static_cast<T>(sigma[c]);
      const T xs = x[c] * is, ds = d[c] * is;
      nx += xs * xs;
      nd += ds * ds;
      ix = fmax(ix, fabs(xs));
      id = fmax(id, fabs(ds));
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      nx += __shfl_xor_sync(0xffffffffu, nx, off);
      nd += __shfl_xor_sync(0xffffffffu, nd, off);
      ix = fmax(ix, __shfl_xor_sync(0xffffffffu, ix, off));
      id = fmax(id, __shfl_xor_sync(0xffffffffu, id, off));
    }
    nx = sqrt(nx) * Unit<T>::guard;
    nd = sqrt(nd) * Unit<T>::guard;
  }
  T lo = static_cast<T>(neg_inf()), hi = static_cast<T>(pos_inf());
  bool bad = false;
  for (int i = lane; i < m; i += 32) {
    const T* a = A + static_cast<size_t>(i) * n_ld;
    T ax = T(0), ad = T(0);
    for (int c = 0; c < n; ++c) {
      ax += a[c] * x[c];
      ad += a[c] * d[c];
    }
    T sv = b[i] - ax;
    if (kr != nullptr) {
      const T k2 = kr[3 * i], k1 = kr[3 * i + 1];
      sv -= fmin(k2 * nx, k1 * ix);
      T eg = fmin(k2 * nd, k1 * id);
      if (corrn != nullptr) eg += kr[3 * i + 2] * static_cast<T>(corrn[k]);
      ad = ad > T(0) ? ad + eg : (ad < T(0) ? ad - eg : ad);
    }
    if (!isfinite(sv) || !isfinite(ad)) { bad = true; continue; }
    if (sv < T(0)) sv = T(0);
    if (ad > T(0)) {
      const T lam = sv / ad;
      hi = lam < hi ? lam : hi;
    } else if (ad < T(0)) {
      const T lam = sv / ad;
      lo = lam > lo ? lam : lo;
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const T ol = __shfl_xor_sync(0xffffffffu, lo, off);
    const T oh = __shfl_xor_sync(0xffffffffu, hi, off);
    lo = ol > lo ? ol : lo;
    hi = oh < hi ? oh : hi;
  }
  if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(status, MHAR_ST_NONFINITE);
  if (!move) {
    if (lane == 0) {
      key_lo[k] = f64_key(static_cast<double>(lo));
      key_hi[k] = f64_key(static_cast<double>(hi));
    }
    return;
  }
  // Section 4.5 in the same warp (the arithmetic of update_kernel): theta on
  // the chord, x += theta d.
  double t = 0.0;
  if (lane == 0) {
    const double L = static_cast<double>(lo), H = static_cast<double>(hi);
    if (isinf(L) || isinf(H)) {
      atomicOr(status, MHAR_ST_UNBOUNDED);
      atomicAdd(&counters[1], 1ull);
    } else if (L > H) {
      atomicOr(status, MHAR_ST_STALL);
      atomicAdd(&counters[0], 1ull);
    } else {
      const uint64_t step = *step_ptr + static_cast<uint64_t>(j);
      const U4 w = philox_block(seed, step, walker0 + static_cast<uint32_t>(k), 0u, kStreamChord);
      const double u = open_unit_f64(w.x);
      t = L + u * (H - L);
      if (sizeof(T) != 8) t = static_cast<double>(static_cast<float>(t));
    }
    lmin[k] = L;
    lmax[k] = H;
    theta[k] = t;
  }
  t = __shfl_sync(0xffffffffu, t, 0);
  const size_t row = static_cast<size_t>(k) * n_ld;
  if constexpr (sizeof(T) == 8) {
    for (int i = lane; i < n; i += 32) X64[row + i] += t * D64[row + i];
  } else {
    const float tf = static_cast<float>(t);
    for (int i = lane; i < n; i += 32) df_axpy(Xhi[row + i], Xlo[row + i], tf, D32[row + i]);
    if (corr != nullptr && tf != 0.0f) {
      for (int i = lane; i < n; i += 32) {
        float dlt = 0.0f;
        for (int e = 0; e < mE; ++e)
          dlt = fmaf(Q32[static_cast<size_t>(e) * n_ld + i], corr[static_cast<size_t>(k) * mE + e], dlt);
        Xlo[row + i] = fmaf(-tf, dlt, Xlo[row + i]);
      }
    }
  }
}

__global__ void __launch_bounds__(kThreads)
refresh_simt_kernel(int m, int n_ld, int z, int z_ld, const double* __restrict__ A,
                    const double* __restrict__ b, const float* __restrict__ Xhi,
                    const float* __restrict__ Xlo, const float* __restrict__ row_scale, float* S,
                    unsigned long long* drift_key) {
  constexpr int BK = 8;
  __shared__ double As[BK][64];
  __shared__ double Xs[BK][64];
  __shared__ double red[kThreads];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int i0 = blockIdx.x * 64, w0 = blockIdx.y * 64;
  double acc[4][4];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[r][c] = 0.0;
  for (int k0 = 0; k0 < n_ld; k0 += BK) {
    for (int e = tid; e < 64 * BK; e += kThreads) {
      const int r = e / BK, c = e - r * BK;
      const int gi = i0 + r, gw = w0 + r;
      As[c][r] = gi < m ? A[static_cast<size_t>(gi) * n_ld + k0 + c] : 0.0;
      const size_t xi = static_cast<size_t>(gw) * n_ld + k0 + c;
      Xs[c][r] = gw < z ? static_cast<double>(Xhi[xi]) + static_cast<double>(Xlo[xi]) : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      double a[4], xv[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) a[r] = As[kk][ty * 4 + r];
#pragma unroll
      for (int c = 0; c < 4; ++c) xv[c] = Xs[kk][tx + 16 * c];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] += a[r] * xv[c];
    }
    __syncthreads();
  }
  double drift = 0.0;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int gi = i0 + ty * 4 + r;
    if (gi >= m) continue;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int gw = w0 + tx + 16 * c;
      if (gw >= z) continue;
      const double s = b[gi] - acc[r][c];
      const double sc = static_cast<double>(row_scale[gi]);
      float* sp = S + (static_cast<size_t>(gi >> 2) * z_ld + gw) * 4 + (gi & 3);
      drift = fmax(drift, fabs(static_cast<double>(*sp) * sc - s));
      *sp = static_cast<float>(s / sc);
    }
  }
  red[tid] = drift;
  __syncthreads();
  for (int st = kThreads / 2; st > 0; st >>= 1) {
    if (tid < st) red[tid] = fmax(red[tid], red[tid + st]);
    __syncthreads();
  }
  if (tid == 0) atomicMax(drift_key, f64_key(red[0]));
}

// Mixed mode with equalities: x <- x - A_E^T (A_E A_E^T)^{-1} (A_E x - b_E)
// = x - Q^T (Q x - w) (Section 3.2),
// in FP64 on the FP32-pair points (removes drift of the equality residual).
__global__ void reproject_kernel(int z, int n, int n_ld, int mE, const double* Q,
                                 const double* w, float* Xhi, float* Xlo) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k = blockIdx.x * (kThreads / 32) + warp;
  if (k >= z) return;
  const size_t row = static_cast<size_t>(k) * n_ld;
  // x <- x - (q_e . x - w_e) q_e, one orthonormal row at a time (the same
  // as x - Q^T (Q x - w)), on the FP64 value of the hi + lo pair.
  for (int e = 0; e < mE; ++e) {
    const double* q = Q + static_cast<size_t>(e) * n_ld;
    double acc = 0.0;
    for (int i = lane; i < n; i += 32)
      acc += q[i] * (static_cast<double>(Xhi[row + i]) + static_cast<double>(Xlo[row + i]));
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    const double r = acc - w[e];
    for (int i = lane; i < n; i += 32) {
      const double v = static_cast<double>(Xhi[row + i]) + static_cast<double>(Xlo[row + i]) -
                       r * q[i];
      const float hv = static_cast<float>(v);
      Xhi[row + i] = hv;
      Xlo[row + i] = static_cast<float>(v - static_cast<double>(hv));
    }
  }
}

// Tensor-core operands: columns multiplied by the coordinate scales sigma
// (powers of two), then a per-row power-of-two scale s_r with
// max_i |a_ri sigma_i| / s_r in [0.5, 1), then the row split into FP16 hi + lo.
// FP32 copy of b / s_r, padded.  With them, the error bounds of the chord
// epilogue (tc_common.cuh, row_block), from the row a_hat = a_r sigma / s_r in
// FP64 and its FP16 pair (hi, lo), in two forms, for the 2-norms and for the
// max-norms of the walker's operands (|.|_p below is the p-norm of a row):
//   Kg_p = |a_hat - hi - lo|_p + 2^-11 |lo|_p (1 + 2^-11)
//          + (T + 1) 2^-22 |a_hat|_p (1 + 2^-9)
//     -- |computed - exact| of a_hat . d per unit |d_hat|_q (1/p + 1/q = 1):
//     the pair's exact representation error, the dropped lo.lo product
//     (|d_lo| <= 2^-11 |d_hi|), and the FP32 accumulation of the T MMAs that
//     meet the row's nonzeros (T = `per_step` per 16-column block holding a
//     nonzero: at most (T + 1) 2^-22 of the sum of |products| on GB300,
//     Hoelder's inequality bounds that by |a_hat|_p |d_hat|_q);
//   Ks_p = Kg_p + |a_hat|_p (2^-21 + 2^-24 c_p) + 2^-22 |a_hat|_p
//     -- the same for a_hat . x_hat per unit |x_hat|_q (max |x_hat| in
//     [0.5, 1)), adding the split of the point (2^-21 relative plus 2^-25
//     absolute per coordinate: c_2 = sqrt(nonzeros), c_1 = 1) and the
//     relative rounding of the ratio and of theta (2^-22 of |a_hat . x_hat|).
// The other relative roundings (b / s_r in FP32, the slack's FMA, the ratio,
// theta) are at most 2^-21 |b / s_r| and lower bS by that much.  Every bound
// is rounded up to FP32.  rowk[4 r ..]: Ks_2, Kg_2, Ks_1, Kg_1.
__global__ void prepare_tc_kernel(int m, int n, int n_ld, int m_pad, int k_pad, int per_step,
                                  const double* A, const double* b, __half* Ah, __half* Al,
                                  float* row_scale, float* bS, float* rowk, const float* sigma) {
  const int r = blockIdx.x;
  if (r >= m_pad) return;
  __shared__ double red[7][kThreads];
  __shared__ unsigned int blocks[4];   // nonzero 16-column blocks (k_pad <= 2048)
  if (threadIdx.x < 4) blocks[threadIdx.x] = 0u;
  double mx = 0.0;
  if (r < m)
    for (int i = threadIdx.x; i < n; i += blockDim.x)
      mx = fmax(mx, fabs(A[static_cast<size_t>(r) * n_ld + i] * static_cast<double>(sigma[i])));
  red[0][threadIdx.x] = mx;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[0][threadIdx.x] = fmax(red[0][threadIdx.x], red[0][threadIdx.x + s]);
    __syncthreads();
  }
  mx = red[0][0];
  __syncthreads();
  int e = 0;
  if (mx > 0.0) frexp(mx, &e);  // mx = f 2^e, f in [0.5, 1)
  const double scale = ldexp(1.0, e);
  const bool near_one = e >= -1000 && e <= 1000;
  const double inv = near_one ? ldexp(1.0, -e) : 0.0;
  double q[7] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};   // |a|_2^2 |a|_1 |rep|_2^2 |rep|_1 |lo|_2^2 |lo|_1 nnz
  for (int i = threadIdx.x; i < k_pad; i += blockDim.x) {
    double a = 0.0;
    if (r < m && i < n) {
      a = A[static_cast<size_t>(r) * n_ld + i] * static_cast<double>(sigma[i]);
      a = near_one ? a * inv : a / scale;      // the same bits
    }
    const float v = static_cast<float>(a);
    const __half h = __float2half_rn(v);
    const __half l = __float2half_rn(v - __half2float(h));
    Ah[static_cast<size_t>(r) * k_pad + i] = h;
    Al[static_cast<size_t>(r) * k_pad + i] = l;
    const double hl = static_cast<double>(__half2float(h));
    const double ll = static_cast<double>(__half2float(l));
    const double rep = a - hl - ll;
    q[0] += a * a;
    q[1] += fabs(a);
    q[2] += rep * rep;
    q[3] += fabs(rep);
    q[4] += ll * ll;
    q[5] += fabs(ll);
    if (a != 0.0) {
      q[6] += 1.0;
      atomicOr(&blocks[(i >> 4) >> 5], 1u << ((i >> 4) & 31));
    }
  }
  for (int t = 0; t < 7; ++t) red[t][threadIdx.x] = q[t];
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s)
      for (int t = 0; t < 7; ++t) red[t][threadIdx.x] += red[t][threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const int nblk = __popc(blocks[0]) + __popc(blocks[1]) + __popc(blocks[2]) + __popc(blocks[3]);
    const double g = static_cast<double>(per_step * nblk + 1) * 0x1p-22 * (1.0 + 0x1p-9);
    const double up = 1.0 + 1e-12;   // the FP64 sums and square roots
    const double na2 = sqrt(red[0][0]) * up, na1 = red[1][0] * up;
    const double rp2 = sqrt(red[2][0]) * up, rp1 = red[3][0] * up;
    const double lo2 = sqrt(red[4][0]) * up, lo1 = red[5][0] * up;
    const double nnz = red[6][0];
    const double kg2 = rp2 + 0x1p-11 * lo2 * (1.0 + 0x1p-11) + g * na2;
    const double ks2 = kg2 + na2 * (0x1p-21 + 0x1p-24 * sqrt(nnz)) + 0x1p-22 * na2;
    const double kg1 = rp1 + 0x1p-11 * lo1 * (1.0 + 0x1p-11) + g * na1;
    const double ks1 = kg1 + na1 * (0x1p-21 + 0x1p-24) + 0x1p-22 * na1;
    const double bs = r < m ? b[r] / scale : 0.0;
    float bf = static_cast<float>(bs);
    bf = bf - 0x1p-21f * fabsf(bf);           // the relative roundings (see above)
    if (static_cast<double>(bf) > bs) bf = nextafterf(bf, -INFINITY);
    const double kk[4] = {ks2, kg2, ks1, kg1};
    for (int t = 0; t < 4; ++t) {
      float f = static_cast<float>(kk[t]);
      if (static_cast<double>(f) < kk[t]) f = nextafterf(f, INFINITY);
      rowk[4 * r + t] = r < m ? f : 0.0f;
    }
    row_scale[r] = r < m ? static_cast<float>(scale) : 1.0f;
    bS[r] = r < m ? bf : 0.0f;
  }
}

// The per-32-row blocks of the chord epilogue (tc_common.cuh, row_block): each
// group of 32 rows takes the bound form (2-norms or max-norms of the walker's
// operands) whose sum of Kg over the group, times the typical norm of the
// scaled direction (d2, dinf), is smaller -- the max-norm form wins for rows
// with few nonzeros, the 2-norm form for dense ones.
__global__ void row_blocks_kernel(int groups, const float* bS, const float* rowk, float d2,
                                  float dinf, float* rows) {
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= groups) return;
  double s2 = 0.0, s1 = 0.0;
  for (int t = 0; t < 32; ++t) {
    s2 += rowk[4 * (32 * g + t) + 1];
    s1 += rowk[4 * (32 * g + t) + 3];
  }
  const int inf = s1 * dinf < s2 * d2 ? 1 : 0;
  float* blk = rows + g * 128;
  for (int t = 0; t < 32; ++t) {
    const int r = 32 * g + t;
    blk[t] = bS[r];
    blk[32 + t] = rowk[4 * r + (inf ? 2 : 0)];
    blk[64 + t] = rowk[4 * r + (inf ? 3 : 1)];
    blk[96 + t] = inf ? 1.0f : 0.0f;
  }
}

__global__ void init_keys_kernel(int z, unsigned long long* key_lo, unsigned long long* key_hi) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < z) {
    key_lo[k] = f64_key(neg_inf());
    key_hi[k] = f64_key(pos_inf());
  }
}

inline int blocks_for(long long count, int per_block) {
  return static_cast<int>((count + per_block - 1) / per_block);
}

}  // namespace

cudaError_t launch_directions(mhar_ctx* c, int j) {
  const int mode = c->opts.precision == MHAR_FP64 ? 0 : (c->opts.precision == MHAR_FP32 ? 1 : 2);
  const long long threads =
      static_cast<long long>(c->z) * ((c->n + 3) / 4) * (mode == 0 ? 2 : 1);
  // Few threads (small bodies): small blocks, so that the draws (FP64
  // transcendental functions in FP64 mode) spread over many SMs.
  int sms = 148;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
  int block = static_cast<int>((threads + sms - 1) / sms);
  block = block < 32 ? 32 : (block > kThreads ? kThreads : (block + 31) / 32 * 32);
  directions_kernel<<<blocks_for(threads, block), block, 0, c->stream>>>(
      mode, (c->mE == 0 && c->pc_rank < 0) ? 1 : 0, c->opts.seed, c->d.step, j, c->opts.walker0,
      c->z, c->n, c->n_ld,
      c->k_pad, c->d.sigma, c->d.D64, c->d.D32, c->d.Dh, c->d.Dl, c->d.Dh2, c->d.Dl2);
  return cudaGetLastError();
}

// Walkers (warps) per block of the projections: eight, fewer when their
// shared coefficient vectors (mE doubles, or 3 mE floats, per walker) would
// pass 150 KB (with the kept h below: 198 KB at most).
int projection_warps(int mE) {
  const int w = static_cast<int>((150u << 10) / (3 * sizeof(float) * (mE > 0 ? mE : 1)));
  return w < 1 ? 1 : (w > kThreads / 32 ? kThreads / 32 : w);
}

// Floats of h a walker keeps in shared memory between the passes of the
// FP32 / tensor-core projection: all of it up to n = 1536 (6 KB a warp),
// else none (drawn again).
int projection_keep(int n) {
  const int q = (n + 3) / 4;
  return q <= 384 ? 4 * q : 0;
}

// The limit is a per-function attribute shared by every context, so it is
// set to the most any context uses (198 KB: 150 KB of coefficients and 48 KB
// of kept h), not to this context's need.
cudaError_t projection_smem_attr(int mE, int n) {
  (void)mE;
  (void)n;
  const int bytes = 200 << 10;
  cudaError_t e = cudaFuncSetAttribute(projection_f64_kernel,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(projection_ff_kernel,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  return e;
}

cudaError_t launch_projection(mhar_ctx* c, int j, int draw) {
  const int warps = projection_warps(c->mE);
  const int grid = blocks_for(c->z, warps);
  if (c->opts.precision == MHAR_FP64) {
    const size_t smem = sizeof(double) * static_cast<size_t>(warps) * c->mE;
    projection_f64_kernel<<<grid, warps * 32, smem, c->stream>>>(c->z, c->n, c->n_ld, c->mE,
                                                                 c->d.Q64, c->d.D64);
  } else {
    const int split =
        (c->opts.precision == MHAR_MIXED_F16X3 || c->opts.precision == MHAR_MIXED_RECOMPUTE) ? 1 : 0;
    const int keep = projection_keep(c->n);
    const size_t smem = sizeof(float) * static_cast<size_t>(warps) * (3 * c->mE + keep);
    projection_ff_kernel<<<grid, warps * 32, smem, c->stream>>>(
        draw, c->opts.seed, c->d.step, j, c->opts.walker0, c->z, c->n, c->n_ld, c->mE,
        c->d.Q32, c->d.Q32lo, c->d.D32, split, c->k_pad, (c->z + 127) / 128 * 128,
        c->use_ts ? 1 : 0, c->d.sigma, c->d.Dh, c->d.Dl, c->d.Dh2, c->d.Dl2, c->d.corr,
        c->d.corrn, keep, c->d.status);
  }
  return cudaGetLastError();
}

cudaError_t launch_precondition(mhar_ctx* c, int j) {
  dim3 grid(blocks_for(c->n, kPcThreads), blocks_for(c->z, kPcWalkers));
  precondition_kernel<<<grid, kPcThreads, 0, c->stream>>>(
      c->opts.seed, c->d.step, j, c->opts.walker0, c->z, c->n, c->n_ld, c->pc_rank,
      c->d.pc_delta64, c->d.pc_U64, c->d.D64);
  return cudaGetLastError();
}

cudaError_t launch_draw_precondition(mhar_ctx* c, int j, int split) {
  const int z_ld = (c->z + 127) / 128 * 128;
  int sms = 148;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
  // A block's g is drawn again by each block beside it along the coordinates (as
  // much work as half a tile), so only as many as give an SM four blocks.
  const int tiles = blocks_for(c->n, kDpTile), rows = blocks_for(c->z, kDpWalkers);
  int across = blocks_for(4 * sms, rows);
  across = across > tiles ? tiles : across;
  const int per = blocks_for(tiles, across);
  draw_precondition_kernel<<<dim3(blocks_for(tiles, per), rows), kDpThreads, 0, c->stream>>>(
      c->opts.seed, c->d.step, j, c->opts.walker0, c->z, c->n, c->n_ld, c->pc_rank, per,
      c->d.pc_delta32, c->d.pc_U32, c->d.D32, split, c->k_pad, z_ld, c->use_ts ? 1 : 0, c->d.sigma,
      c->d.Dh, c->d.Dl, c->d.Dh2, c->d.Dl2, c->d.status);
  return cudaGetLastError();
}

bool simt_warp_path(const mhar_ctx* c) {
  int sms = 148;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
  return static_cast<long long>(blocks_for(c->m, 64)) * blocks_for(c->z, 64) < sms &&
         c->m <= 2048;
}

cudaError_t launch_chord_update_warp(mhar_ctx* c, int j) {
  const int g = blocks_for(c->z, kWarpChordThreads / 32);
  if (c->opts.precision == MHAR_FP64)
    chord_warp_kernel<double><<<g, kWarpChordThreads, 0, c->stream>>>(
        c->d.A64, c->d.b64, static_cast<const double*>(nullptr), c->d.sigma, nullptr, c->d.X64,
        c->d.D64, c->m, c->n, c->n_ld, c->z, c->d.key_lo,
        c->d.key_hi, c->d.status, 1, c->opts.seed, c->d.step, j, c->opts.walker0, c->d.lmin,
        c->d.lmax, c->d.theta, c->d.counters, c->d.X64, c->d.D64, nullptr, nullptr, nullptr,
        c->mE, nullptr, nullptr);
  else
    chord_warp_kernel<float><<<g, kWarpChordThreads, 0, c->stream>>>(
        c->d.A32, c->d.b32, c->d.kr32, c->d.sigma, c->d.corrn, c->d.Xhi, c->d.D32, c->m, c->n, c->n_ld, c->z, c->d.key_lo,
        c->d.key_hi, c->d.status, 1, c->opts.seed, c->d.step, j, c->opts.walker0, c->d.lmin,
        c->d.lmax, c->d.theta, c->d.counters, nullptr, nullptr, c->d.Xhi, c->d.Xlo, c->d.D32,
        c->mE, c->d.Q32, c->d.corr);
  return cudaGetLastError();
}

cudaError_t launch_chord_simt(mhar_ctx* c) {
  dim3 grid(blocks_for(c->m, 64), blocks_for(c->z, 64));
  if (c->opts.precision == MHAR_FP64) {
    chord_simt_kernel<double><<<grid, kThreads, 0, c->stream>>>(
        c->d.A64, c->d.b64, static_cast<const double*>(nullptr), c->d.X64, c->d.D64, c->d.sigma,
        nullptr, c->m, c->n_ld, c->z,
        c->d.key_lo, c->d.key_hi, c->d.status);
  } else {
    chord_simt_kernel<float><<<grid, kThreads, 0, c->stream>>>(
        c->d.A32, c->d.b32, c->d.kr32, c->d.Xhi, c->d.D32, c->d.sigma, c->d.corrn, c->m, c->n_ld,
        c->z,
        c->d.key_lo, c->d.key_hi, c->d.status);
  }
  return cudaGetLastError();
}

cudaError_t launch_update_simt(mhar_ctx* c, int j) {
  const int mode = c->opts.precision == MHAR_FP64 ? 0 : 1;
  update_kernel<<<blocks_for(c->z, kThreads / 32), kThreads, 0, c->stream>>>(
      mode, c->opts.seed, c->d.step, j, c->opts.walker0, c->z, c->n, c->n_ld, c->d.key_lo,
      c->d.key_hi, c->d.lmin, c->d.lmax, c->d.theta, c->d.status, c->d.counters, c->d.X64,
      c->d.D64, c->d.Xhi, c->d.Xlo, c->d.D32, c->mE, c->d.Q32, c->d.corr);
  return cudaGetLastError();
}

cudaError_t launch_prep_walkers(mhar_ctx* c, int j, int flags) {
  const int z_ld = (c->z + 127) / 128 * 128;
  const int chunks = (c->n + 7) / 8;
  const int warps = chunks < kPrepMaxWarps ? chunks : kPrepMaxWarps;
  prep_walkers_kernel<<<blocks_for(c->z, kPrepWalkers), warps * 32, 0, c->stream>>>(
      flags, c->opts.seed, c->d.step, j, c->opts.walker0, c->z, z_ld, c->n, c->n_ld, c->k_pad,
      c->d.Xhi, c->d.Xlo, c->d.Dh, c->d.Dl, c->d.Dh2, c->d.Dl2, c->d.D32, c->d.Xh, c->d.Xl,
      c->d.wscale, c->use_ts ? 1 : 0, c->d.sigma, (c->mE > 0 || c->pc_rank >= 0) ? 1 : 0,
      c->d.status);
  return cudaGetLastError();
}

cudaError_t launch_advance_many(uint64_t* const* steps, int count, int by, cudaStream_t stream) {
  advance_many_kernel<<<blocks_for(count, kThreads), kThreads, 0, stream>>>(steps, count, by);
  return cudaGetLastError();
}

cudaError_t launch_advance(mhar_ctx* c, int steps) {
  advance_kernel<<<1, 1, 0, c->stream>>>(c->d.step, steps);
  return cudaGetLastError();
}

cudaError_t launch_emit(mhar_ctx* c, double* out_device, int walkers) {
  const int mode = c->opts.precision == MHAR_FP64 ? 0 : 1;
  const long long count = static_cast<long long>(walkers) * c->n;
  emit_kernel<<<blocks_for(count, kThreads), kThreads, 0, c->stream>>>(
      mode, walkers, c->n, c->n_ld, c->d.X64, c->d.Xhi, c->d.Xlo, out_device);
  return cudaGetLastError();
}

cudaError_t launch_batch_emit(const BatchProblem* probs, int count, long long most,
                              const BatchOuts& outs, cudaStream_t stream) {
  const int bx = std::min(64, blocks_for(most, 4 * kThreads));
  batch_emit_kernel<<<dim3(bx, count), kThreads, 0, stream>>>(probs, outs);
  return cudaGetLastError();
}

cudaError_t launch_batch_status(const BatchProblem* probs, int count, int2* gather,
                                const BatchCounters& counters, cudaStream_t stream) {
  batch_status_kernel<<<blocks_for(count, kThreads), kThreads, 0, stream>>>(probs, count, gather,
                                                                            counters);
  return cudaGetLastError();
}

cudaError_t launch_set_points(mhar_ctx* c, const double* X_dev) {
  const int mode = c->opts.precision == MHAR_FP64 ? 0 : 1;
  const long long count = static_cast<long long>(c->z) * c->n;
  if (X_dev)
    set_points_kernel<<<blocks_for(count, kThreads), kThreads, 0, c->stream>>>(
        mode, c->z, c->n, c->n_ld, X_dev, c->d.X64, c->d.Xhi, c->d.Xlo);
  init_keys_kernel<<<blocks_for(c->z, kThreads), kThreads, 0, c->stream>>>(c->z, c->d.key_lo,
                                                                         c->d.key_hi);
  return cudaGetLastError();
}

bool check_direct(const mhar_ctx* c, int walkers) {
  const long long pairs = static_cast<long long>(c->m) * walkers;
  return pairs <= kCheckPairs || pairs * c->n <= kCheckScreen;
}

int check_launches(const mhar_ctx* c, int walkers) {
  return check_direct(c, walkers) ? 1 : (c->mE > 0 ? 3 : 2);
}

cudaError_t launch_check(mhar_ctx* c, int walkers, unsigned long long* out_keys) {
  const int mode = c->opts.precision == MHAR_FP64 ? 0 : 1;
  const int block = 128;
  auto direct = [&](int m) {
    const int rows = m > c->mE ? m : c->mE;
    check_kernel<<<dim3(blocks_for(rows, block), walkers), block, sizeof(double) * c->n, c->stream>>>(
        mode, m, c->n, c->n_ld, c->mE, c->d.A64, c->d.b64, c->d.AE64, c->d.bE64, c->d.X64,
        c->d.Xhi, c->d.Xlo, out_keys);
  };
  if (check_direct(c, walkers)) {
    direct(c->m);
    return cudaGetLastError();
  }
  // The screen's ub array lives in the emission buffer (z n doubles; every
  // use of it is ordered on the context's stream): 2 n floats per walker, so
  // row tiles are grouped when there are more of them than that.
  const int tiles = blocks_for(c->m, kChkRows);
  const int group = blocks_for(tiles, 2 * c->n);
  const int groups = blocks_for(tiles, group);
  float* ub = reinterpret_cast<float*>(c->d.emit);
  unsigned int* best = reinterpret_cast<unsigned int*>(c->d.check + 5);
  cudaError_t e = cudaMemsetAsync(best, 0, sizeof(*best), c->stream);
  if (e != cudaSuccess) return e;
  check_screen_kernel<<<dim3(groups, blocks_for(walkers, kChkWalkers)), kThreads, 0, c->stream>>>(
      mode, c->m, c->n, c->n_ld, walkers, group, c->d.A64, c->d.b64, c->d.X64, c->d.Xhi,
      c->d.Xlo, ub, best);
  const long long entries = static_cast<long long>(groups) * walkers;
  check_exact_kernel<<<blocks_for(entries, kChkEntries), kChkRows, 0, c->stream>>>(
      mode, c->m, c->n, c->n_ld, walkers, group, c->d.A64, c->d.b64, c->d.X64, c->d.Xhi,
      c->d.Xlo, ub, best, entries, out_keys);
  if (c->mE > 0) direct(0);
  return cudaGetLastError();
}

cudaError_t launch_stored_reset(mhar_ctx* c) {
  stored_reset_kernel<<<blocks_for(c->z, kThreads / 32), kThreads, 0, c->stream>>>(
      c->z, c->n, c->n_ld, c->d.Xhi, c->d.Xlo, c->d.sigma, c->d.step, c->d.nx_ref,
      c->d.theta_acc, c->d.refresh_step);
  return cudaGetLastError();
}

cudaError_t launch_refresh_simt(mhar_ctx* c) {
  const int z_ld = (c->z + 127) / 128 * 128;
  dim3 grid(blocks_for(c->m, 64), blocks_for(c->z, 64));
  refresh_simt_kernel<<<grid, kThreads, 0, c->stream>>>(
      c->m, c->n_ld, c->z, z_ld, c->d.A64, c->d.b64, c->d.Xhi, c->d.Xlo, c->d.row_scale, c->d.S,
      reinterpret_cast<unsigned long long*>(c->d.check) + 2);
  return cudaGetLastError();
}

cudaError_t launch_reproject(mhar_ctx* c) {
  reproject_kernel<<<blocks_for(c->z, kThreads / 32), kThreads, 0, c->stream>>>(
      c->z, c->n, c->n_ld, c->mE, c->d.Q64, c->d.wE64, c->d.Xhi, c->d.Xlo);
  return cudaGetLastError();
}

cudaError_t launch_prepare_tc_operands(mhar_ctx* c, bool blocks) {
  // No more threads than columns: the sums' tree over a block is FP64 work, most of it on
  // zeros for short rows (the same bits without them; 3072 rows of 31 columns 89 -> 39 us).
  const int block = c->k_pad <= 64 ? 64 : c->k_pad <= 128 ? 128 : kThreads;
  prepare_tc_kernel<<<c->m_pad, block, 0, c->stream>>>(
      c->m, c->n, c->n_ld, c->m_pad, c->k_pad, mma_per_step(c), c->d.A64, c->d.b64, c->d.Ah,
      c->d.Al, c->d.row_scale, c->d.bS, c->d.rowk, c->d.sigma);
  if (!blocks) return cudaGetLastError();
  const int groups = c->m_pad / 32;
  row_blocks_kernel<<<blocks_for(groups, 128), 128, 0, c->stream>>>(
      groups, c->d.bS, c->d.rowk, static_cast<float>(c->dir_norm2), static_cast<float>(c->dir_norminf),
      c->d.rows);
  return cudaGetLastError();
}

}  // namespace mhar
