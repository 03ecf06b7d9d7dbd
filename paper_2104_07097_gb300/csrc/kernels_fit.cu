// kernels_fit.cu -- learned direction preconditioner: covariance of warm-up
// points and the rank-r plus diagonal fit, in FP64 on CUDA cores.
//
// The paper draws isotropic directions and assumes the body was brought to
// near-isotropic position beforehand (Sections 1.2 and 3.1).  The fit learns
// that position from the chain itself:
//   1. Sigma = sum_k (x_k - mu)(x_k - mu)^T / (N - 1) over the N warm-up
//      points (all walkers at every snapshot), accumulated about a shift c
//      (walker 0's first snapshot) as S1 = sum (x - c), S2 = sum (x - c)(x - c)^T,
//      Sigma = (S2 - S1 S1^T / N) / (N - 1);
//   2. randomized subspace iteration: Y = Sigma Omega (Omega's column c is
//      Philox stream 3 for walker c at step 0), then power_iters times
//      Q = orth(Y), Y = Sigma Q, and finally Q = orth(Y);
//      orth is the Q factor with a positive diagonal in R, computed by
//      classical Gram-Schmidt with re-orthogonalisation;
//   3. Rayleigh-Ritz: T = Q^T Sigma Q, T = V Lambda V^T by cyclic Jacobi
//      rotations (Golub & Van Loan, Matrix Computations, Section 8.5),
//      U = Q V Lambda_+^{1/2}, largest eigenvalue first;
//   4. delta_i^2 = max(Sigma_ii - (U U^T)_ii, 1e-2 Sigma_ii, 1e-9 tr(Sigma) / n).
// The host then sets the coordinate scales of the tensor-core operands from
// the fitted (delta, U), as for a preconditioner given by the caller.
// None of this is on the per-iteration path; it runs once, then the
// preconditioner is frozen.
#include <cmath>

#include "jacobi_angle.cuh"
#include "mhar_device.cuh"
#include "mhar_internal.h"
#include "normals_f64.cuh"
#include "tc_common.cuh"

namespace mhar {
namespace {

constexpr int kCovTile = 64;     // Sigma tile edge
constexpr int kCovChunk = 1024;  // walkers per block
constexpr int kCovStage = 16;    // walkers staged in shared memory at once
constexpr int kFitThreads = 1024;
constexpr double kEpsRel = 1e-2;
constexpr double kEpsAbs = 1e-9;

__device__ __forceinline__ double point(int mode, const double* X64, const float* Xhi,
                                        const float* Xlo, size_t idx) {
  return mode == 0 ? X64[idx] : static_cast<double>(Xhi[idx]) + static_cast<double>(Xlo[idx]);
}

__global__ void fit_shift_kernel(int mode, int n, const double* X64, const float* Xhi,
                                 const float* Xlo, double* shift) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    shift[i] = point(mode, X64, Xhi, Xlo, static_cast<size_t>(i));
}

// One (row tile ti, column tile tj >= ti) of S2 and, on diagonal tiles, the
// matching part of S1, over one chunk of walkers.  16 x 16 threads, 4 x 4
// outputs each.
__global__ void __launch_bounds__(256)
cov_accumulate_kernel(int mode, int z, int n, int n_ld, int tiles, const double* X64,
                      const float* Xhi, const float* Xlo, const double* shift, double* s1,
                      double* s2) {
  int t = blockIdx.x, ti = 0;
  while (t >= tiles - ti) {
    t -= tiles - ti;
    ++ti;
  }
  const int tj = ti + t;
  // Centred values (x - shift, formed in FP64) are staged as FP32; the
  // products of one stage of kCovStage walkers are summed in FP32 and each
  // stage's sum is added to an FP64 total, so FP64 work is 1 / kCovStage of
  // the products (FP64 runs at a small fraction of the FP32 rate on GB300).
  __shared__ float xa[kCovStage][kCovTile];
  __shared__ float xb[kCovStage][kCovTile];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double acc[4][4];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[r][q] = 0.0;
  double col_sum = 0.0;
  const int kbeg = blockIdx.y * kCovChunk;
  const int kend = min(z, kbeg + kCovChunk);
  for (int kb = kbeg; kb < kend; kb += kCovStage) {
    for (int e = threadIdx.x; e < kCovStage * kCovTile; e += blockDim.x) {
      const int w = e / kCovTile, q = e % kCovTile, k = kb + w;
      const int ia = ti * kCovTile + q, ib = tj * kCovTile + q;
      double va = 0.0, vb = 0.0;
      if (k < kend) {
        const size_t row = static_cast<size_t>(k) * n_ld;
        if (ia < n) va = point(mode, X64, Xhi, Xlo, row + ia) - shift[ia];
        if (ib < n) vb = point(mode, X64, Xhi, Xlo, row + ib) - shift[ib];
      }
      xa[w][q] = static_cast<float>(va);
      xb[w][q] = static_cast<float>(vb);
    }
    __syncthreads();
    float part[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int q = 0; q < 4; ++q) part[r][q] = 0.0f;
#pragma unroll 4
    for (int w = 0; w < kCovStage; ++w) {
      float a[4], bb[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) a[r] = xa[w][ty * 4 + r];
#pragma unroll
      for (int q = 0; q < 4; ++q) bb[q] = xb[w][tx * 4 + q];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q) part[r][q] = fmaf(a[r], bb[q], part[r][q]);
      if (ti == tj && threadIdx.x < kCovTile) col_sum += static_cast<double>(xa[w][threadIdx.x]);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[r][q] += static_cast<double>(part[r][q]);
    __syncthreads();
  }
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = ti * kCovTile + ty * 4 + r, jj = tj * kCovTile + tx * 4 + q;
      if (i < n && jj < n) atomicAdd(&s2[static_cast<size_t>(i) * n + jj], acc[r][q]);
    }
  if (ti == tj && threadIdx.x < kCovTile) {
    const int i = ti * kCovTile + threadIdx.x;
    if (i < n) atomicAdd(&s1[i], col_sum);
  }
}

// Sigma (full, symmetric) from S1 and the upper tiles of S2.
__global__ void cov_finalize_kernel(int n, double N, const double* s1, const double* s2,
                                    double* sigma, int* flag, int* expo) {
  const long long idx = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx >= static_cast<long long>(n) * n) return;
  const int i = static_cast<int>(idx / n), jj = static_cast<int>(idx % n);
  const int lo = min(i, jj), hi = max(i, jj);
  const double v = (s2[static_cast<size_t>(lo) * n + hi] - s1[i] * s1[jj] / N) / (N - 1.0);
  if (!isfinite(v)) atomicOr(flag, 1);
  else if (i == jj) atomicMax(expo, (__double2hiint(v) >> 20) & 0x7ff);
  sigma[idx] = v;
}

// Omega: column c < rank holds stream 3's normals of walker c at step 0.
__global__ void omega_kernel(uint64_t seed, int n, int rank, double* Q) {
  const int quads = (n + 3) >> 2;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= kMaxPcRank * quads) return;
  const int c = idx / quads, q = idx % quads;
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  if (c < rank) {
    const U4 w = philox_block(seed, 0ull, static_cast<uint32_t>(c), static_cast<uint32_t>(q),
                              kStreamFit);
    box_muller_f64(w.x, w.y, v[0], v[1]);
    box_muller_f64(w.z, w.w, v[2], v[3]);
  }
#pragma unroll
  for (int e = 0; e < 4; ++e)
    if (4 * q + e < n) Q[static_cast<size_t>(4 * q + e) * kMaxPcRank + c] = v[e];
}

// Y = Sigma Q (n x n times n x 32): a lane per column; a block's eight warps
// split the sum over k for kSymmRows rows and their partial sums are added in
// warp order.  Bound by the FP64 rate (2 FMAs a clock and SM: 13 us for n = 500
// on the whole chip); a warp per row, 63 blocks for n = 500, left it to the
// latency of 500 dependent steps: 79 us, now 22.
constexpr int kSymmRows = 4;
constexpr int kSymmWarps = 8;

__global__ void __launch_bounds__(kSymmWarps * 32)
symm_block_kernel(int n, const double* __restrict__ sigma, const double* __restrict__ Q,
                  double* __restrict__ Y) {
  __shared__ double part[kSymmWarps][kSymmRows][kMaxPcRank];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i0 = blockIdx.x * kSymmRows;
  const int per = (n + kSymmWarps - 1) / kSymmWarps;
  const int k0 = warp * per, k1 = min(n, k0 + per);
  double acc[kSymmRows] = {};
  const double* row[kSymmRows];
#pragma unroll
  for (int r = 0; r < kSymmRows; ++r)
    row[r] = sigma + static_cast<size_t>(min(i0 + r, n - 1)) * n;
#pragma unroll 4
  for (int k = k0; k < k1; ++k) {
    const double q = Q[static_cast<size_t>(k) * kMaxPcRank + lane];
#pragma unroll
    for (int r = 0; r < kSymmRows; ++r) acc[r] = fma(row[r][k], q, acc[r]);
  }
#pragma unroll
  for (int r = 0; r < kSymmRows; ++r) part[warp][r][lane] = acc[r];
  __syncthreads();
  if (warp < kSymmRows && i0 + warp < n) {
    double s = part[0][warp][lane];
#pragma unroll
    for (int w = 1; w < kSymmWarps; ++w) s += part[w][warp][lane];
    Y[static_cast<size_t>(i0 + warp) * kMaxPcRank + lane] = s;
  }
}

__device__ double block_sum(double v, double* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  double s = 0.0;
  if (warp == 0) {
    s = lane < static_cast<int>(blockDim.x >> 5) ? red[lane] : 0.0;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) red[32] = s;
  }
  __syncthreads();
  return red[32];
}

// A power of two that brings Y = Sigma Q near 1, so that squares of covariances past
// 2^+-511 stay in range (Q has the same bits); expo: the largest biased exponent of
// Sigma's diagonal.
__device__ __forceinline__ double orth_scale(const int* expo) {
  const int k = max(-1000, min(1000, __ldg(expo) - 1022));
  return __hiloint2double((1023 - k) << 20, 0);              // 2^-k
}

// Q = orth(Y) for the first `rank` columns (zero beyond): classical
// Gram-Schmidt, each column projected out twice, then normalised.  One block:
// the general form, for n past what the cluster keeps in shared memory.
__global__ void __launch_bounds__(kFitThreads)
orth_kernel(int n, int rank, const int* expo, const double* __restrict__ Y,
            double* __restrict__ Q) {
  const double scale = orth_scale(expo);
  __shared__ double dots[kMaxPcRank];
  __shared__ double red[33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int c = 0; c < kMaxPcRank; ++c) {
    for (int i = threadIdx.x; i < n; i += blockDim.x)
      Q[static_cast<size_t>(i) * kMaxPcRank + c] = c < rank ? Y[static_cast<size_t>(i) * kMaxPcRank + c] * scale : 0.0;
    if (c >= rank) continue;
    for (int pass = 0; pass < 2; ++pass) {
      __syncthreads();
      if (warp < c) {
        double acc = 0.0;
        for (int i = lane; i < n; i += 32)
          acc = fma(Q[static_cast<size_t>(i) * kMaxPcRank + warp],
                    Q[static_cast<size_t>(i) * kMaxPcRank + c], acc);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if (lane == 0) dots[warp] = acc;
      }
      __syncthreads();
      for (int i = threadIdx.x; i < n; i += blockDim.x) {
        double v = Q[static_cast<size_t>(i) * kMaxPcRank + c];
        for (int p = 0; p < c; ++p) v = fma(-dots[p], Q[static_cast<size_t>(i) * kMaxPcRank + p], v);
        Q[static_cast<size_t>(i) * kMaxPcRank + c] = v;
      }
    }
    __syncthreads();
    double part = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const double v = Q[static_cast<size_t>(i) * kMaxPcRank + c];
      part = fma(v, v, part);
    }
    const double nrm2 = block_sum(part, red);
    const double inv = nrm2 > 0.0 ? 1.0 / sqrt(nrm2) : 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x)
      Q[static_cast<size_t>(i) * kMaxPcRank + c] *= inv;
    __syncthreads();
  }
}

__device__ __forceinline__ uint32_t cluster_addr(const void* local, uint32_t cta) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
               : "=r"(remote)
               : "r"(tc::smem_u32(local)), "r"(cta));
  return remote;
}
__device__ __forceinline__ void st_cluster_f64(double* local, uint32_t cta, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(cluster_addr(local, cta)), "d"(v)
               : "memory");
}
__device__ __forceinline__ void st_cluster_u32(int* local, uint32_t cta, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr(local, cta)), "r"(v)
               : "memory");
}

// Q = orth(Y) by a cluster of kOrthCtas CTAs, each with a share of the rows in
// shared memory (column-major, unnormalised until the end).  Column c is
// projected out of the earlier ones; one exchange over distributed shared
// memory brings every CTA the products with them and |v|^2, so |v - proj|^2
// follows without another.  A second (third) projection only while one took
// away more than half of |v|^2 -- "twice is enough" (Parlett, The Symmetric
// Eigenvalue Problem, Section 6.9): with less taken the rounding left along
// the earlier columns is of the order of the unit roundoff already.
// Bound by the latency of the chain (products, exchange, update) and by the FP64
// rate of the SMs, which one CTA alone used on one SM: n = 500, rank 32 took 1064
// us in orth_kernel, 89 here.
constexpr int kOrthCtas = 16;             // 8 (a portable size): 98 us
constexpr int kOrthThreads = 9 * 32;      // eight warps of products, one that sums
constexpr int kOrthPasses = 3;
constexpr int kOrthMaxLd = 856;           // 32 columns of 856 rows: 219136 bytes

__host__ __device__ constexpr int orth_ld(int n) {   // 8 mod 16: spreads the banks
  return ((n + kOrthCtas - 1) / kOrthCtas + 7) / 16 * 16 + 8;
}

__global__ void __cluster_dims__(kOrthCtas, 1, 1) __launch_bounds__(kOrthThreads)
orth_cluster_kernel(int n, int rank, const int* expo, const double* __restrict__ Y,
                    double* __restrict__ Q) {
  extern __shared__ double col[];                      // [32][ld]
  __shared__ double recv[2][kOrthCtas][kMaxPcRank];    // products of each CTA's rows
  __shared__ double coef[kMaxPcRank];                  // products / |q_p|^2
  __shared__ double inv2[kMaxPcRank];                  // 1 / |q_p|^2
  __shared__ int again;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int cta = static_cast<int>(blockIdx.x);
  const int ld = orth_ld(n), per = (n + kOrthCtas - 1) / kOrthCtas;
  const int r0 = cta * per, rows = max(0, min(per, n - r0));
  const double scale = orth_scale(expo);
  for (int e = tid; e < rows * kMaxPcRank; e += kOrthThreads)
    col[(e & 31) * ld + (e >> 5)] = Y[static_cast<size_t>(r0) * kMaxPcRank + e] * scale;
  // No CTA writes into another before that one runs.
  tc::cluster_sync_all();

  int turn = 0;
  for (int c = 0; c < rank; ++c) {
    double* v = col + c * ld;
    for (int pass = 0; pass < kOrthPasses; ++pass) {
      // Written for pass t + 2 only when every CTA has read it in pass t.
      auto& got = recv[turn];
      turn ^= 1;
      // Products of columns 0 .. c with v: 8 lanes a column, which then send
      // the sum to two CTAs each.
      const int p = tid >> 3, g = tid & 7;
      if ((tid & ~31) >> 3 <= c && warp < 8) {
        double acc = 0.0;
        if (p <= c)
          for (int i = g; i < rows; i += 8) acc = fma(col[p * ld + i], v[i], acc);
#pragma unroll
        for (int off = 1; off < 8; off <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        for (int to = g; to < kOrthCtas; to += 8)
          st_cluster_f64(&got[cta][p], static_cast<uint32_t>(to), acc);
      }
      tc::cluster_sync_all();
      double nrm2 = 0.0, vv = 0.0;
      if (warp == 8) {
        double s[kOrthCtas];
#pragma unroll
        for (int r = 0; r < kOrthCtas; ++r) s[r] = lane <= c ? got[r][lane] : 0.0;
        // The same order in every CTA: every CTA decides alike.
#pragma unroll
        for (int w = kOrthCtas / 2; w > 0; w >>= 1)
#pragma unroll
          for (int r = 0; r < w; ++r) s[r] += s[r + w];
        const double dot = s[0];
        const double cf = lane < c ? dot * inv2[lane] : 0.0;
        coef[lane] = cf;
        nrm2 = lane < c ? -dot * cf : dot;     // dot = 0 past c
        vv = dot;
      }
      __syncthreads();
      if (warp < 8) {
        // v -= sum_p coef_p q_p: four lanes a row.
        const int h = tid & 3;
        for (int ib = 0; ib < rows; ib += 64) {
          const int i = ib + (tid >> 2);
          double acc = 0.0;
          if (i < rows)
            for (int q = h; q < c; q += 4) acc = fma(coef[q], col[q * ld + i], acc);
          acc += __shfl_xor_sync(0xffffffffu, acc, 1);
          acc += __shfl_xor_sync(0xffffffffu, acc, 2);
          if (h == 0 && i < rows) v[i] -= acc;
        }
      } else {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) nrm2 += __shfl_xor_sync(0xffffffffu, nrm2, off);
        vv = __shfl_sync(0xffffffffu, vv, c);
        if (lane == 0) {
          again = !(nrm2 >= 0.5 * vv);
          inv2[c] = nrm2 > 0.0 ? 1.0 / nrm2 : 0.0;
        }
      }
      __syncthreads();
      if (!again) break;
    }
  }
  for (int e = tid; e < rows * kMaxPcRank; e += kOrthThreads) {
    const int c = e & 31;
    Q[static_cast<size_t>(r0) * kMaxPcRank + e] =
        c < rank ? col[c * ld + (e >> 5)] * sqrt(inv2[c]) : 0.0;
  }
}

// T = Q^T (Sigma Q): a block per row of T, a lane per column, the sum over the
// coordinates split over the warps and added in their order.
__global__ void __launch_bounds__(256)
ritz_matrix_kernel(int n, int rank, const double* __restrict__ Q, const double* __restrict__ SQ,
                   double* __restrict__ T) {
  __shared__ double part[8][kMaxPcRank];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, a = blockIdx.x;
  double acc = 0.0;
  if (a < rank && lane < rank)
#pragma unroll 4
    for (int i = warp; i < n; i += 8)
      acc = fma(Q[static_cast<size_t>(i) * kMaxPcRank + a],
                SQ[static_cast<size_t>(i) * kMaxPcRank + lane], acc);
  part[warp][lane] = acc;
  __syncthreads();
  if (warp == 0) {
    double s = part[0][lane];
#pragma unroll
    for (int w = 1; w < 8; ++w) s += part[w][lane];
    T[a * kMaxPcRank + lane] = s;
  }
}

// T = V Lambda V^T by Jacobi rotations in cyclic row order, all rotations of
// one antidiagonal p + q at once: (p, q) shares an index only with rotations
// of smaller p + q before it in that order and of larger p + q after it, so
// the result is the row-cyclic one with 2 rank - 3 steps a sweep instead of
// rank (rank - 1) / 2.  Two CTAs: the first rotates T (a warp per pair), the
// second V, one step behind, so V's half of the FP64 work is off the chain.
// The angle comes from FP32's approximate functions (jacobi_angle.cuh: a relative error
// of 1e-6 in tan leaves that share of the entry to the next sweep); cos and sin are
// normalised in FP64, so the rotations are orthogonal to the FP64 roundoff.
// Bound by the chain of steps and one SM's FP64 rate; rank 32 with one warp and
// one rotation at a time took most of 8018 us, 573 to 669 (by the input) here.
constexpr int kJacobiThreads = 512;

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kJacobiThreads)
jacobi_kernel(int rank, const double* __restrict__ Tin, double* __restrict__ lam,
              double* __restrict__ Vout) {
  __shared__ double M[kMaxPcRank][kMaxPcRank + 1];     // T, or V
  __shared__ double2 rot[2][kMaxPcRank / 2];           // (cos, sin) of a step's pairs
  __shared__ double red[2][kJacobiThreads / 32];
  __shared__ int go;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool t_side = blockIdx.x == 0;
  // Scaled by a power of two to a trace near 1 (the angles are formed in FP32).
  double tr = 0.0;
  for (int a = 0; a < rank; ++a) tr += fabs(Tin[a * kMaxPcRank + a]);
  int e = 0;
  if (tr > 0.0 && isfinite(tr)) frexp(tr, &e);
  e = max(-1000, min(1000, e));
  const double down = ldexp(1.0, -e), up = ldexp(1.0, e);
  for (int idx = tid; idx < kMaxPcRank * kMaxPcRank; idx += kJacobiThreads) {
    const int a = idx >> 5, b = idx & 31;
    M[a][b] = t_side ? 0.5 * (Tin[a * kMaxPcRank + b] + Tin[b * kMaxPcRank + a]) * down
                     : (a == b ? 1.0 : 0.0);
  }
  tc::cluster_sync_all();
  for (int sweep = 0; sweep < 60; ++sweep) {
    if (t_side) {
      double off = 0.0, tot = 0.0;
      for (int a = warp; a < kMaxPcRank; a += kJacobiThreads / 32) {
        const double v = M[a][lane], v2 = v * v;
        tot += v2;
        if (lane != a) off += v2;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        off += __shfl_xor_sync(0xffffffffu, off, o);
        tot += __shfl_xor_sync(0xffffffffu, tot, o);
      }
      if (lane == 0) { red[0][warp] = off; red[1][warp] = tot; }
      __syncthreads();
      if (tid == 0) {
        off = tot = 0.0;
        for (int w = 0; w < kJacobiThreads / 32; ++w) { off += red[0][w]; tot += red[1][w]; }
        go = off > 1e-30 * tot;
        st_cluster_u32(&go, 1u, static_cast<uint32_t>(go));
      }
      __syncwarp();
    }
    tc::cluster_sync_all();
    if (!go) break;
    for (int t = 1; t <= 2 * rank - 3; ++t) {
      const int p0 = max(0, t - rank + 1), pairs = (t - 1) / 2 - p0 + 1;
      const int p = p0 + warp, q = t - p;
      double2* const cs = rot[t & 1];
      if (t_side) {
        if (warp == 0 && lane < pairs) {
          const int pp = p0 + lane, qq = t - pp;
          const double2 r = jacobi_rotation(static_cast<float>(M[pp][qq]),
                                            static_cast<float>(M[qq][qq] - M[pp][pp]));
          cs[lane] = r;
          st_cluster_f64(&cs[lane].x, 1u, r.x);
          st_cluster_f64(&cs[lane].y, 1u, r.y);
        }
        __syncthreads();
        tc::cluster_arrive();
        if (warp < pairs) {      // T <- T J
          const double c = cs[warp].x, s = cs[warp].y;
          const double a = M[lane][p], b = M[lane][q];
          M[lane][p] = c * a - s * b;
          M[lane][q] = s * a + c * b;
        }
        __syncthreads();
        if (warp < pairs) {      // T <- J^T T
          const double c = cs[warp].x, s = cs[warp].y;
          const double a = M[p][lane], b = M[q][lane];
          M[p][lane] = c * a - s * b;
          M[q][lane] = s * a + c * b;
        }
        __syncthreads();
        tc::cluster_wait();      // the step before is done with the other buffer
      } else {
        tc::cluster_arrive();
        tc::cluster_wait();
        if (warp < pairs) {      // V <- V J
          const double c = cs[warp].x, s = cs[warp].y;
          const double a = M[lane][p], b = M[lane][q];
          M[lane][p] = c * a - s * b;
          M[lane][q] = s * a + c * b;
        }
      }
    }
  }
  __syncthreads();
  if (t_side) {
    if (tid < kMaxPcRank) lam[tid] = tid < rank ? M[tid][tid] * up : 0.0;
  } else {
    for (int idx = tid; idx < kMaxPcRank * kMaxPcRank; idx += kJacobiThreads)
      Vout[idx] = M[idx >> 5][idx & 31];
  }
}

// U = Q V Lambda_+^{1/2} (largest eigenvalue first), the diagonal floor and the
// outputs: a warp per coordinate.  (Rank 0: the diagonal alone.)
__global__ void __launch_bounds__(256)
ritz_finish_kernel(int n, int n_ld, int rank, const double* __restrict__ Q,
                   const double* __restrict__ lam_in, const double* __restrict__ V_in,
                   const double* __restrict__ sigma_mat, double* delta64, double* U64,
                   float* delta32, float* U32, int* flag) {
  __shared__ double V[kMaxPcRank][kMaxPcRank + 1];
  __shared__ double lam[kMaxPcRank];
  __shared__ int perm[kMaxPcRank];
  __shared__ double red[33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (rank > 0)
    for (int idx = threadIdx.x; idx < kMaxPcRank * kMaxPcRank; idx += blockDim.x)
      V[idx >> 5][idx & 31] = V_in[idx];
  if (warp == 0 && lane < rank) {
    // NaN counts as -Inf, ties go by the index: perm is a permutation whatever the values.
    auto key = [&](int q) { const double v = lam_in[q]; return isnan(v) ? -INFINITY : v; };
    const double mine = key(lane);
    int at = 0;
    for (int q = 0; q < rank; ++q) at += key(q) > mine || (key(q) == mine && q < lane);
    perm[at] = lane;
    lam[at] = fmax(mine, 0.0);
    if (!isfinite(lam_in[lane])) atomicOr(flag, 1);
  }
  // Trace of Sigma for the absolute floor.
  double part = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) part += sigma_mat[static_cast<size_t>(i) * n + i];
  const double tr = block_sum(part, red);
  const int i = blockIdx.x * (blockDim.x >> 5) + warp;
  if (i >= n_ld) return;
  double u = 0.0;
  if (i < n && lane < rank) {
    const int c = perm[lane];
    for (int b = 0; b < rank; ++b) u = fma(Q[static_cast<size_t>(i) * kMaxPcRank + b], V[b][c], u);
    u *= sqrt(lam[lane]);
  }
  double u2 = u * u;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) u2 += __shfl_xor_sync(0xffffffffu, u2, o);
  double d2 = 0.0;
  if (i < n) {
    const double sii = sigma_mat[static_cast<size_t>(i) * n + i];
    d2 = fmax(sii - u2, fmax(kEpsRel * sii, kEpsAbs * tr / n));
    if (!isfinite(d2 + u2) || !isfinite(u)) atomicOr(flag, 1);
  }
  U64[static_cast<size_t>(i) * kMaxPcRank + lane] = u;
  U32[static_cast<size_t>(i) * kMaxPcRank + lane] = static_cast<float>(u);
  if (lane == 0) {
    delta64[i] = sqrt(d2);
    delta32[i] = static_cast<float>(sqrt(d2));
  }
}

inline int blocks_for(long long count, int per_block) {
  return static_cast<int>((count + per_block - 1) / per_block);
}

}  // namespace

cudaError_t launch_fit_shift(mhar_ctx* c, FitScratch* f) {
  const int mode = c->opts.precision == MHAR_FP64 ? 0 : 1;
  fit_shift_kernel<<<blocks_for(c->n, 256), 256, 0, c->stream>>>(mode, c->n, c->d.X64, c->d.Xhi,
                                                                c->d.Xlo, f->shift);
  return cudaGetLastError();
}

cudaError_t launch_fit_accumulate(mhar_ctx* c, FitScratch* f) {
  const int mode = c->opts.precision == MHAR_FP64 ? 0 : 1;
  const int tiles = blocks_for(c->n, kCovTile);
  dim3 grid(tiles * (tiles + 1) / 2, blocks_for(c->z, kCovChunk));
  cov_accumulate_kernel<<<grid, 256, 0, c->stream>>>(mode, c->z, c->n, c->n_ld, tiles, c->d.X64,
                                                     c->d.Xhi, c->d.Xlo, f->shift, f->s1, f->s2);
  return cudaGetLastError();
}

cudaError_t launch_fit_factor(mhar_ctx* c, FitScratch* f, long long samples, int rank,
                              int power_iters) {
  const int n = c->n;
  cov_finalize_kernel<<<blocks_for(static_cast<long long>(n) * n, 256), 256, 0, c->stream>>>(
      n, static_cast<double>(samples), f->s1, f->s2, f->sigma, f->flag, f->flag + 1);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (rank > 0) {
    omega_kernel<<<blocks_for(static_cast<long long>(kMaxPcRank) * ((n + 3) / 4), 256), 256, 0,
                   c->stream>>>(c->opts.seed, n, rank, f->Q);
    const size_t smem = sizeof(double) * kMaxPcRank * orth_ld(n);
    bool cluster = orth_ld(n) <= kOrthMaxLd;
    if (cluster) {
      // The largest any call needs: the attribute belongs to the function.
      e = cudaFuncSetAttribute(orth_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               static_cast<int>(sizeof(double) * kMaxPcRank * kOrthMaxLd));
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(orth_cluster_kernel,
                                 cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (e != cudaSuccess) return e;
    }
    for (int it = 0; it <= power_iters; ++it) {
      symm_block_kernel<<<blocks_for(n, kSymmRows), kSymmWarps * 32, 0, c->stream>>>(
          n, f->sigma, f->Q, f->Y);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      if (cluster) {
        orth_cluster_kernel<<<kOrthCtas, kOrthThreads, smem, c->stream>>>(n, rank, f->flag + 1,
                                                                           f->Y, f->Q);
        // A device part without room for sixteen CTAs side by side refuses the launch.
        cluster = cudaGetLastError() == cudaSuccess;
      }
      if (!cluster) orth_kernel<<<1, kFitThreads, 0, c->stream>>>(n, rank, f->flag + 1, f->Y, f->Q);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    symm_block_kernel<<<blocks_for(n, kSymmRows), kSymmWarps * 32, 0, c->stream>>>(
        n, f->sigma, f->Q, f->Y);
    ritz_matrix_kernel<<<kMaxPcRank, 256, 0, c->stream>>>(n, rank, f->Q, f->Y, f->T);
    jacobi_kernel<<<2, kJacobiThreads, 0, c->stream>>>(rank, f->T, f->lam, f->V);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  ritz_finish_kernel<<<blocks_for(c->n_ld, 8), 256, 0, c->stream>>>(
      n, c->n_ld, rank, f->Q, f->lam, f->V, f->sigma, c->d.pc_delta64, c->d.pc_U64,
      c->d.pc_delta32, c->d.pc_U32, f->flag);
  return cudaGetLastError();
}

}  // namespace mhar
