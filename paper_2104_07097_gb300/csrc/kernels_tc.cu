// kernels_tc.cu -- the fused tensor-core walker step (MHAR_MIXED_F16X3 mode).
//
// One launch performs, for every walker, Sections 4.4 and 4.5 of the paper on
// the stored slack S = b - A X:
//   G = D A^T           tcgen05.mma kind::f16 (FP16 hi/lo split operands,
//                       3 products hi.hi + hi.lo + lo.hi, FP32 accumulation
//                       in tensor memory; TMA-staged 128B-swizzled tiles)
//   lambda_max = min{ s_i / g_i : g_i > 0 },  lambda_min = max{ s_i / g_i : g_i < 0 }
//                       folded in registers straight out of tensor memory --
//                       the m x z ratio matrix never reaches memory
//   theta = lambda_min + u (lambda_max - lambda_min),  u from Philox stream 1
//   S -= G diag(theta),  X += D diag(theta)   (X as FP32 pairs)
//
// Work decomposition.  The MMA's M dimension is the walkers (128 per CTA, one
// walker per tensor-memory lane, so every thread owns one walker and reduces
// its chord sequentially), N is the constraint rows (128 per tile), K is the
// dimension n.  The rows of A are split over the CTAs of a thread-block
// cluster (up to 4 tiles = 512 tensor-memory columns per CTA); the partial
// chords are combined through distributed shared memory, so each CTA can
// update its own slack rows while G is still in tensor memory.
//
// Warp roles (640 threads): warp 0 = TMA producer, warp 1 = MMA issuer and
// tensor-memory owner, warps 2..17 = epilogue (four warps per 32-lane quarter,
// each taking a quarter of every tile's columns), warps 18 and 19 draw the next
// directions into the other pair.
//
// A strip's walkers concern its cluster alone, so without equalities and a
// preconditioner one launch runs many iterations: the draw, two launches and
// the set-up of each iteration (33.7 us an iteration for 4096 walkers of a 2000 x
// 100 body) go, the rows of A for the next iteration arrive while the points
// move, and the walker operands of up to two K chunks stay in shared memory for
// all row tiles; 22.8 us now, bound by the slack's trips to L2 (three a row:
// 96 MB) and the latency of the steps between the MMAs.  (The last tile's slack
// kept in registers between the passes: 26.6 us, from spills.)
//
// Every mbarrier wait is bounded (about 2 s of clock); on expiry the kernel
// records a timeout in the error word, stops waiting and still runs
// through every cluster barrier, so no peer is left waiting.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_fp16.h>

#include <cstdio>
#include <cstring>

#include "mhar_device.cuh"
#include "mhar_internal.h"
#include "tc_common.cuh"
#include "walker_tail.cuh"

namespace mhar {
namespace {

using namespace tc;

constexpr int kStages = 3;                            // A and walker chunk together, or
constexpr int kStagesRes = 4;                         // A alone, walker operands resident
constexpr int kMaxTilesPerCta = 4;                    // 512 TMEM columns
constexpr int kStageBytes = 4 * kOperandBytes;        // A hi, A lo, W hi, W lo
constexpr int kEpiWarps = 16;                         // 4 per TMEM lane quarter
constexpr int kEpiThreads = kEpiWarps * 32;
constexpr int kDrawWarp = 2 + kEpiWarps;
constexpr int kDrawThreads = 64;
constexpr int kThreadsTc = kDrawWarp * 32 + kDrawThreads;
constexpr int kThreadsOne = kDrawWarp * 32;           // a single iteration draws nothing
constexpr int kMaxClusterTc = 16;
static_assert(kStagesRes * 2 * kOperandBytes + 4 * kOperandBytes <= kStages * kStageBytes,
              "the resident layout fits the streamed one's space");

enum : int { kModeChord = 0, kModeRefresh = 1 };

struct TcParams {
  int mode;                 // kModeChord | kModeRefresh
  const float* row_scale;   // m_pad: A[i,:] = row_scale[i] (Ah + Al)[i,:]
  const float* bS;          // m_pad: b[i] / row_scale[i] in FP32 (refresh)
  const float* wscale;      // z_ld: X[k,:] = wscale[k] (Xh + Xl)[k,:] (refresh)
  float* S;                 // slack / row_scale, blocked: [(i/4) z_ld + k] * 4 + i%4
  float* Xhi;               // z x n_ld
  float* Xlo;
  const float* rowk;        // 4 m_pad: Ks_2, Kg_2, Ks_1, Kg_1 of every row (prepare_tc_kernel)
  const __half* Xh;         // z_ld x k_pad: FP16 hi of the points split at the last refresh
  const float* corrn;       // z or null: ||Q^T corr / sigma||_2 (see add_correction)
  // The tracked slack's error since the last refresh, per walker: bounded by
  // Ks_i E_k + k 2^-24 |b_i / scale_i| after k updates, with
  //   E_k = (||x_r / sigma|| + sum_t |theta_t| ||d_hat_t||) (1 + k / (4 T + 4)),
  // x_r the point at the refresh and T the MMAs of one product chain.
  const float* nx_ref;      // z: ||x_r / sigma||_2 bound, set by every refresh
  float* theta_acc;         // z: sum_t |theta_t| ||d_hat_t||_2 since the refresh
  const uint64_t* refresh_step;  // iteration counter at the last refresh
  float growth;             // 1 / (4 T + 4)
  int check_drift;          // refresh: compare the tracked slack with its bound
  WalkerTail wt;            // direction pairs, coordinate scales, the draw's arguments
  const float* sigma;       // n_ld: coordinate scales (operands hold x / sigma, d / sigma)
  const float* Q32;         // mE x n_ld (orthonormal rows of the equalities) or null
  const float* corr;        // z x mE residual corrections or null
  double* lmin;
  double* lmax;
  double* theta;
  int* status;
  unsigned long long* counters;
  int* err;
  unsigned long long* drift_key;
  const uint64_t* step_ptr; // the iteration is *step_ptr + j, or (null) step0
  uint64_t* step_out;       // null, or where the next iteration's number goes
  uint64_t seed, step0;
  int j, iters;             // iterations of this launch
  double* out;              // samples, SmallRun's layout, or null
  int emit, thin, phase;
  int draw_items;           // of the next directions: the draw warps' share
  uint32_t walker0;
  int m, n, n_ld, z, z_ld, kdim, k_chunks, tiles_per_cta, m_tiles, mE;
};

struct alignas(16) SmemTail {
  uint64_t full[kStagesRes];
  uint64_t empty[kStagesRes];
  uint64_t tfull[kMaxTilesPerCta];
  uint64_t w_full;                         // resident walker operands
  uint64_t c_full;                         // every CTA's partial chords
  uint32_t tmem_base;
  int timed_out;
  float part_lo[4][kWalkers];
  float part_hi[4][kWalkers];
  float2 recv[kMaxClusterTc][kWalkers];    // (lambda_min, lambda_max) of each CTA's rows
  float theta[kWalkers];
  alignas(16) float scale[kMaxTilesPerCta * kRowsTile];
  alignas(16) float brow[kMaxTilesPerCta * kRowsTile];
  alignas(16) float ks[kMaxTilesPerCta * kRowsTile];   // Ks_i of this CTA's rows
  alignas(16) float kg[kMaxTilesPerCta * kRowsTile];   // Kg_i
  alignas(16) float jk[kMaxTilesPerCta * kRowsTile];   // k 2^-24 |b_i / scale_i|, k updates since the refresh
  float nrm[kWalkers];                     // sums of squares of the directions' FP16 hi rows
  float nd[kWalkers];                      // ||d_hat||_2 bound of each walker's direction
};

constexpr size_t kSmemBytes = 1024 + static_cast<size_t>(kStages) * kStageBytes + sizeof(SmemTail);
static_assert(kSmemBytes <= 232448, "walker_tc_kernel exceeds the shared memory of a CTA");

// The slack is stored blocked by 4 rows: element (i, k) sits at
// ((i / 4) z_ld + k) 4 + i % 4, so one 16-byte access gives a walker four
// consecutive rows and a warp's 32 consecutive walkers read 512 contiguous
// bytes.  32 rows of one walker = eight such accesses, z_ld * 16 bytes apart.
__device__ __forceinline__ float* s_block(const TcParams& p, int row, int k) {
  return p.S + (static_cast<size_t>(row >> 2) * p.z_ld + k) * 4;
}
__device__ __forceinline__ void load_s32(const TcParams& p, const float* src, float (&v)[32]) {
  const float4* q = reinterpret_cast<const float4*>(src);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float4 t = __ldcg(q + static_cast<size_t>(i) * p.z_ld);
    v[4 * i] = t.x; v[4 * i + 1] = t.y; v[4 * i + 2] = t.z; v[4 * i + 3] = t.w;
  }
}
__device__ __forceinline__ void store_s32(const TcParams& p, float* dst, const float (&v)[32]) {
  float4* q = reinterpret_cast<float4*>(dst);
#pragma unroll
  for (int i = 0; i < 8; ++i)
    __stcg(q + static_cast<size_t>(i) * p.z_ld, make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]));
}

// Sum of squares of walker k's FP16 hi row (chunk order), by its cg == 0 thread,
// for the walker's four threads.  Run by the epilogue threads.
__device__ __forceinline__ float hi_sumsq(const TcParams& p, const __half* rows, int k, int wl,
                                          int cg, float* scr) {
  if (cg == 0) {
    const uint4* r4 = reinterpret_cast<const uint4*>(rows + static_cast<size_t>(k) * p.wt.k_pad);
    float ss = 0.0f;
#pragma unroll 4
    for (int c = 0; c < (p.wt.k_pad >> 3); ++c) ss += sumsq8(__ldcg(r4 + c));
    scr[wl] = ss;
  }
  named_bar<kEpiThreads>();
  return scr[wl];
}

// The rounding of b in `since` updates, for this CTA's rows (a barrier of the
// epilogue follows before their use).
__device__ __forceinline__ void fill_jk(const TcParams& p, SmemTail* tail, int row_base, int ntiles,
                                        float since, int tid) {
  for (int r = tid; r < p.tiles_per_cta * kRowsTile; r += kEpiThreads)
    tail->jk[r] = r < ntiles * kRowsTile ? since * 5.9604645e-8f * fabsf(tail->brow[r]) * 1.0001f : 0.0f;
}

// (x, y) into CTA `rank`'s copy of *local; counts on its barrier *bar.
__device__ __forceinline__ void push_chord(float2* local, uint64_t* bar, uint32_t rank, float x,
                                           float y) {
  uint32_t dst, rbar;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"(smem_u32(local)), "r"(rank));
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rbar) : "r"(smem_u32(bar)), "r"(rank));
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(
                   dst), "f"(x), "f"(y), "r"(rbar)
               : "memory");
}

// The four products of KS K steps of one chunk, in the order hi.hi, hi.lo, lo.hi,
// lo.lo a step (a runtime trip count starves the tensor pipe, tc_common.cuh).
template <int KS>
__device__ __forceinline__ void four_products(uint32_t d, uint64_t wh, uint64_t wl, uint64_t ah,
                                              uint64_t al, uint32_t idesc, uint32_t acc_first) {
#pragma unroll
  for (int ks = 0; ks < KS; ++ks) {
    const uint64_t o = static_cast<uint64_t>(2 * ks);
    mma_f16(d, wh + o, ah + o, idesc, ks > 0 ? 1u : acc_first);
    mma_f16(d, wh + o, al + o, idesc, 1u);
    mma_f16(d, wl + o, ah + o, idesc, 1u);
    mma_f16(d, wl + o, al + o, idesc, 1u);
  }
}

// RUN: many iterations, and the draws; else a refresh, or one iteration whose directions a
// kernel before it drew (equalities, a preconditioner), without what only the loop needs and
// without its two cluster barriers: with an equality 16.6 -> 14.9 us on 2 walkers of a
// 60 x 5 body, 36.8 -> 35.6 on 4096 of a 2000 x 100 body.  (The loop's form keeps the
// refresh's branch: compiled out, 64 iterations of rand100x2000 took 0.6 % longer.)
template <bool RUN>
__global__ void __launch_bounds__(RUN ? kThreadsTc : kThreadsOne, 1)
walker_tc_kernel(const __grid_constant__ CUtensorMap tm_ah, const __grid_constant__ CUtensorMap tm_al,
                 const __grid_constant__ CUtensorMap tm_wh, const __grid_constant__ CUtensorMap tm_wl,
                 const __grid_constant__ CUtensorMap tm_wh2, const __grid_constant__ CUtensorMap tm_wl2,
                 const __grid_constant__ TcParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  SmemTail* tail = reinterpret_cast<SmemTail*>(base + kStages * kStageBytes);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = blockIdx.x;       // cluster rank: the cluster spans grid.x
  const int csize = static_cast<int>(gridDim.x);
  const int strip = blockIdx.y;
  const int tile0 = static_cast<int>(rank) * p.tiles_per_cta;
  int ntiles = p.m_tiles - tile0;
  ntiles = ntiles < 0 ? 0 : (ntiles > p.tiles_per_cta ? p.tiles_per_cta : ntiles);
  const int row_base = tile0 * kRowsTile;
  const bool refresh = p.mode == kModeRefresh;
  // Shared memory: the walker operands of up to two K chunks, then stages of A's
  // chunks; or stages of both.
  const bool resident = p.k_chunks <= 2;
  const int stages = resident ? kStagesRes : kStages;
  uint8_t* const a_base = base + (resident ? 4 * kOperandBytes : 0);
  const int a_stage = resident ? 2 * kOperandBytes : kStageBytes;

  // ---- set-up -------------------------------------------------------------
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStagesRes; ++s) {
      mbar_init(&tail->full[s], 1);
      mbar_init(&tail->empty[s], 1);
    }
    for (int t = 0; t < kMaxTilesPerCta; ++t) mbar_init(&tail->tfull[t], 1);
    mbar_init(&tail->w_full, 1);
    mbar_init(&tail->c_full, 1);
    tail->timed_out = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    const uint32_t cols = p.tiles_per_cta <= 1 ? 128u : (p.tiles_per_cta == 2 ? 256u : 512u);
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tail->tmem_base)),
                 "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  for (int r = threadIdx.x; r < p.tiles_per_cta * kRowsTile; r += blockDim.x) {
    const bool in = r < ntiles * kRowsTile;
    tail->scale[r] = in ? p.row_scale[row_base + r] : 1.0f;
    tail->brow[r] = in ? p.bS[row_base + r] : 0.0f;
    tail->ks[r] = in ? p.rowk[4 * (row_base + r)] : 0.0f;
    tail->kg[r] = in ? p.rowk[4 * (row_base + r) + 1] : 0.0f;
  }
  tc_fence_before();
  __syncwarp();
  if constexpr (RUN) {
    cluster_sync_all();      // every CTA's barriers are ready
  } else {
    cluster_arrive();        // waited for before the first message to one of them
    __syncthreads();
  }
  tc_fence_after();
  const uint32_t tmem = tail->tmem_base;
  volatile int* timed_out = &tail->timed_out;
  const uint64_t step0 = p.step_ptr != nullptr ? *p.step_ptr + static_cast<uint64_t>(p.j) : p.step0;
  const uint64_t since0 = step0 - *p.refresh_step;
  const int tid = static_cast<int>(threadIdx.x) - 64;   // of the epilogue, then the draw threads
  // This CTA's share of the strip's draws (walkers) and moves (chunks of 8).
  const int share = (kWalkers + csize - 1) / csize;
  const int w_begin = static_cast<int>(rank) * share;
  const int w_count = max(0, min(share, kWalkers - w_begin));
  const int chunks = (p.n + 7) >> 3;
  const int draw_all = RUN && p.wt.draw && !refresh ? w_count * chunks : 0;
  const int iters = RUN ? p.iters : 1;
  int a_it = 0, m_it = 0;
#pragma unroll 1
  for (int it = 0; it < iters; ++it) {
    const uint64_t step = step0 + static_cast<uint64_t>(it);
    const int cur = static_cast<int>(step & 1ull);
    // Updates of the tracked slack since the last refresh.
    const float since = static_cast<float>(since0 + static_cast<uint64_t>(it));

    if (warp == 0) {
      // ---- TMA producer -------------------------------------------------------
      if (lane == 0) {
        const bool second = !refresh && cur != 0;
        const CUtensorMap* wh = second ? &tm_wh2 : &tm_wh;
        const CUtensorMap* wl = second ? &tm_wl2 : &tm_wl;
        const int yw = strip * kWalkers, per = ntiles * p.k_chunks;
        // The pair was written with ordinary stores by the cluster's threads.
        if (it > 0) asm volatile("fence.proxy.async;" ::: "memory");
        if (resident && ntiles > 0) {
          mbar_expect_tx(&tail->w_full, static_cast<uint32_t>(p.k_chunks) * 2u * kOperandBytes);
          for (int kc = 0; kc < p.k_chunks; ++kc) {
            tma_load_2d(base + 2 * kc * kOperandBytes, wh, &tail->w_full, kc * kTcKChunk, yw);
            tma_load_2d(base + (2 * kc + 1) * kOperandBytes, wl, &tail->w_full, kc * kTcKChunk, yw);
          }
        }
        // This iteration's stages; those of A alone also the first of the next.
        const int end = min(iters * per, (it + 1) * per + (resident ? stages : 0));
        for (; a_it < end; ++a_it) {
          const int s = a_it % stages, nt = (a_it / p.k_chunks) % ntiles, kc = a_it % p.k_chunks;
          if (a_it >= stages) mbar_wait(&tail->empty[s], ((a_it / stages) - 1) & 1, timed_out, p.err);
          uint8_t* st = a_base + s * a_stage;
          mbar_expect_tx(&tail->full[s], static_cast<uint32_t>(a_stage));
          const int x = kc * kTcKChunk;
          const int yr = row_base + nt * kRowsTile;
          tma_load_2d(st, &tm_ah, &tail->full[s], x, yr);
          tma_load_2d(st + kOperandBytes, &tm_al, &tail->full[s], x, yr);
          if (!resident) {
            tma_load_2d(st + 2 * kOperandBytes, wh, &tail->full[s], x, yw);
            tma_load_2d(st + 3 * kOperandBytes, wl, &tail->full[s], x, yw);
          }
        }
      }
      __syncwarp();
    } else if (warp == 1) {
      // ---- MMA issuer: G = (Wh + Wl)(Ah + Al)^T, four FP16 products ------------
      if (lane == 0) {
        constexpr uint32_t idesc = make_idesc(kWalkers, kRowsTile);
        if (resident && ntiles > 0) mbar_wait(&tail->w_full, it & 1, timed_out, p.err);
        for (int nt = 0; nt < ntiles; ++nt) {
          const uint32_t d_tmem = tmem + static_cast<uint32_t>(nt * kRowsTile);
          for (int kc = 0; kc < p.k_chunks; ++kc, ++m_it) {
            const int s = m_it % stages;
            mbar_wait(&tail->full[s], (m_it / stages) & 1, timed_out, p.err);
            tc_fence_after();
            const uint32_t a0 = smem_u32(a_base + s * a_stage);
            const uint32_t w0 = resident ? smem_u32(base + 2 * kc * kOperandBytes) : a0 + 2u * kOperandBytes;
            const uint64_t ah = sw128_desc(a0), al = sw128_desc(a0 + kOperandBytes);
            const uint64_t wh = sw128_desc(w0), wl = sw128_desc(w0 + kOperandBytes);
            const uint32_t acc = kc > 0 ? 1u : 0u;
            switch (min(kTcKChunk / kTcK, (p.kdim - kc * kTcKChunk) / kTcK)) {
              case 4: four_products<4>(d_tmem, wh, wl, ah, al, idesc, acc); break;
              case 3: four_products<3>(d_tmem, wh, wl, ah, al, idesc, acc); break;
              case 2: four_products<2>(d_tmem, wh, wl, ah, al, idesc, acc); break;
              default: four_products<1>(d_tmem, wh, wl, ah, al, idesc, acc); break;
            }
            mma_commit(&tail->empty[s]);
          }
          mma_commit(&tail->tfull[nt]);
        }
      }
      __syncwarp();
    } else if (warp >= kDrawWarp) {
      // ---- iteration s+1's directions into the other pair ------------------------
      walker_draw_items(p.wt, cur, p.seed, step + 1ull, p.walker0, strip, p.z, w_begin, w_count,
                        tid - kEpiThreads, min(p.draw_items, draw_all), kDrawThreads);
    } else if (refresh) {
      // ---- refresh epilogue: S = b - A X from tensor memory ----------------------
      const int e = warp - 2;
      const int q = warp & 3;
      const int cg = e >> 2;
      const int wl = q * 32 + lane;
      fill_jk(p, tail, row_base, ntiles, since, tid);
      const int k = strip * kWalkers + wl;
      const float ws = p.wscale[k];
      float drift = 0.0f;
      // Bound on |tracked - recomputed| per unit Ks_i: the tracked slack's bound
      // (see TcParams) plus the recomputation's own (ws ||x_hat||_2).
      const float nxw = ws * norm_bound(hi_sumsq(p, p.Xh, k, wl, cg, tail->nrm));
      const float Eb = (k < p.z && p.check_drift)
                           ? (p.nx_ref[k] + p.theta_acc[k]) *
                                     (1.0f + since * (p.growth + 2.384185791e-7f)) * 1.0001f +
                                 nxw
                           : INFINITY;
      bool off = false;
      for (int nt = 0; nt < ntiles; ++nt) {
        const int col = nt * kRowsTile + cg * 32;
        float* Sb = s_block(p, row_base + col, k);
        float sv[32];
        load_s32(p, Sb, sv);
        mbar_wait(&tail->tfull[nt], 0, timed_out, p.err, true);
        tc_fence_after();
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          float g[16];
          tmem_ld16(tmem + (static_cast<uint32_t>(q * 32) << 16) + static_cast<uint32_t>(col + 16 * half), g);
#pragma unroll
          for (int c = 0; c < 16; ++c) {
            const int cc = 16 * half + c;
            const float sn = fmaf(-g[c], ws, tail->brow[col + cc]);
            // drift in the units of the constraint: |change| * row scale
            drift = fmaxf(drift, fabsf(sn - sv[cc]) * tail->scale[col + cc]);
            off = off || fabsf(sn - sv[cc]) > fmaf(tail->ks[col + cc], Eb, tail->jk[col + cc]);
            sv[cc] = sn;
          }
        }
        if (k < p.z) store_s32(p, Sb, sv);
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) drift = fmaxf(drift, __shfl_xor_sync(0xffffffffu, drift, off));
      if (lane == 0 && drift > 0.0f) atomicMax(p.drift_key, f64_key(static_cast<double>(drift)));
      if (off && k < p.z) atomicOr(p.status, MHAR_ST_DRIFT);
    } else {
      // ---- chord epilogue, pass 1: partial (lambda_min, lambda_max) ---------------
      const int e = warp - 2;
      const int q = warp & 3;       // TMEM lane quarter this warp may access
      const int cg = e >> 2;        // which 32-column group of each tile
      const int wl = q * 32 + lane; // walker within the strip
      const int k = strip * kWalkers + wl;
      if (tid == 0)
        mbar_expect_tx(&tail->c_full, static_cast<uint32_t>(csize * kWalkers * sizeof(float2)));
      fill_jk(p, tail, row_base, ntiles, since, tid);
      walker_draw_items(p.wt, cur, p.seed, step + 1ull, p.walker0, strip, p.z, w_begin, w_count,
                        p.draw_items + tid, draw_all, kEpiThreads);
      const float nd = norm_bound(hi_sumsq(p, p.wt.Dh[cur], k, wl, cg, tail->nrm)) +
                       ((p.corrn != nullptr && k < p.z) ? 4194304.0f * p.corrn[k] : 0.0f);
      // Error bound of this walker's tracked slack, in units of Ks_i (see TcParams).
      // (The last factors cover the FP32 sums of theta_acc and E itself.)
      const float E = k < p.z ? (p.nx_ref[k] + __ldcg(p.theta_acc + k)) *
                                    (1.0f + since * (p.growth + 2.384185791e-7f)) * 1.0001f
                              : 0.0f;
      if (cg == 0) tail->nd[wl] = nd;
      ChordAcc acc;
      acc.init();
      float s_cur[32] = {};
      if (ntiles > 0) load_s32(p, s_block(p, row_base + cg * 32, k), s_cur);
      for (int nt = 0; nt < ntiles; ++nt) {
        const int col = nt * kRowsTile + cg * 32;
        float s_nxt[32] = {};   // (defined: else it would be kept round the iterations)
        if (nt + 1 < ntiles) load_s32(p, s_block(p, row_base + col + kRowsTile, k), s_nxt);
        mbar_wait(&tail->tfull[nt], it & 1, timed_out, p.err, true);
        tc_fence_after();
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          float g[16];
          tmem_ld16(tmem + (static_cast<uint32_t>(q * 32) << 16) +
                        static_cast<uint32_t>(col + 16 * half), g);
#pragma unroll
          for (int c = 0; c < 16; ++c) {
            // Both the slack and G are in units of the row's power-of-two
            // scale, so their ratio is the paper's lambda_i unchanged.  The
            // slack is lowered by its error bound and g pushed away from zero
            // by its own (the margins of tc_common.cuh's slack32 / scan32).
            const int r = col + 16 * half + c;
            const float gg = g[c];
            const float ss = clamp_slack(s_cur[16 * half + c] - fmaf(tail->ks[r], E, tail->jk[r]));
            const float sd = __int_as_float(__float_as_int(nd) | (__float_as_int(gg) & 0x80000000));
            acc.add(ss, fmaf(tail->kg[r], sd, gg));
          }
        }
#pragma unroll
        for (int c = 0; c < 32; ++c) s_cur[c] = s_nxt[c];
      }
      const float lo = acc.lo_all(), hi = acc.hi_all();
      tail->part_lo[cg][wl] = lo;
      tail->part_hi[cg][wl] = hi;
      named_bar<kEpiThreads>();
      if constexpr (!RUN) cluster_wait();
      if (cg == 0) {
        // This CTA's partial chord to every CTA of the cluster, data and arrival in
        // one message.
        const float cl = fmaxf(fmaxf(lo, tail->part_lo[1][wl]), fmaxf(tail->part_lo[2][wl], tail->part_lo[3][wl]));
        const float ch = fminf(fminf(hi, tail->part_hi[1][wl]), fminf(tail->part_hi[2][wl], tail->part_hi[3][wl]));
        for (int r = 0; r < csize; ++r)
          push_chord(&tail->recv[rank][wl], &tail->c_full, static_cast<uint32_t>(r), cl, ch);
        const U4 w = philox_block(p.seed, step, p.walker0 + static_cast<uint32_t>(k), 0u, kStreamChord);
        mbar_wait(&tail->c_full, it & 1, timed_out, p.err);
        float L = -INFINITY, H = INFINITY;
        for (int r = 0; r < csize; ++r) {
          const float2 v = tail->recv[r][wl];
          L = fmaxf(L, v.x);
          H = fminf(H, v.y);
        }
        float t = 0.0f;
        int flag = 0;
        if (k < p.z) {
          if (isinf(L) || isinf(H)) {
            flag = MHAR_ST_UNBOUNDED;
          } else if (L > H) {
            flag = MHAR_ST_STALL;
          } else {
            const double u = open_unit_f64(w.x);
            t = static_cast<float>(static_cast<double>(L) +
                                   u * (static_cast<double>(H) - static_cast<double>(L)));
          }
          if (rank == 0) {
            if (it + 1 == iters) {
              p.lmin[k] = L;
              p.lmax[k] = H;
              p.theta[k] = t;
            }
            p.theta_acc[k] = __ldcg(p.theta_acc + k) + fabsf(t) * tail->nd[wl];
            if (flag) {
              atomicOr(p.status, flag);
              atomicAdd(&p.counters[flag == MHAR_ST_STALL ? 0 : 1], 1ull);
            }
          }
        }
        tail->theta[wl] = t;
      }
      named_bar<kEpiThreads>();
      // ---- chord epilogue, pass 2: S -= G diag(theta) -----------------------------
      const float t = tail->theta[wl];
      if (__any_sync(0xffffffffu, t != 0.0f)) {
        float s_up[32] = {};
        if (ntiles > 0) load_s32(p, s_block(p, row_base + cg * 32, k), s_up);
        for (int nt = 0; nt < ntiles; ++nt) {
          const int col = nt * kRowsTile + cg * 32;
          float s_nxt[32] = {};
          if (nt + 1 < ntiles) load_s32(p, s_block(p, row_base + col + kRowsTile, k), s_nxt);
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            float g[16];
            // tcgen05.ld is warp-collective: every lane joins, lanes with theta == 0 skip the update.
            tmem_ld16(tmem + (static_cast<uint32_t>(q * 32) << 16) +
                          static_cast<uint32_t>(col + 16 * half), g);
#pragma unroll
            for (int c = 0; c < 16; ++c) s_up[16 * half + c] = fmaf(-t, g[c], s_up[16 * half + c]);
          }
          if (t != 0.0f) store_s32(p, s_block(p, row_base + col, k), s_up);
#pragma unroll
          for (int c = 0; c < 32; ++c) s_up[c] = s_nxt[c];
        }
      }
      // ---- X += D diag(theta) on this CTA's slice of coordinates ---------------
      // Items are (walker, 4 coordinates), the coordinates fastest: whole lines of
      // the rows (a lane per walker took a line for every lane, 3 us).
      const int slice = (chunks + csize - 1) / csize;
      const int c0 = static_cast<int>(rank) * slice;
      const int pieces = 2 * max(0, min(chunks, c0 + slice) - c0);
      const int done = p.phase + it + 1;
      double* const out = RUN && p.out != nullptr && done % p.thin == 0
                              ? p.out + static_cast<size_t>(done / p.thin - 1) * p.emit * p.n
                              : nullptr;
#pragma unroll 2
      for (int i = tid; i < pieces * kWalkers; i += kEpiThreads) {
        const int w = i / pieces, i0 = 8 * c0 + 4 * (i - w * pieces);
        const int kk = strip * kWalkers + w;
        const float tw = tail->theta[w];
        if (kk >= p.z || (tw == 0.0f && out == nullptr)) continue;
        const size_t xr = static_cast<size_t>(kk) * p.n_ld + i0;
        const float4 h4 = *reinterpret_cast<const float4*>(p.Xhi + xr);
        const float4 l4 = *reinterpret_cast<const float4*>(p.Xlo + xr);
        float hi4[4] = {h4.x, h4.y, h4.z, h4.w}, lo4[4] = {l4.x, l4.y, l4.z, l4.w};
        if (tw != 0.0f) {
          const size_t dr = static_cast<size_t>(kk) * p.wt.k_pad + i0;
          const uint2 dh = __ldcg(reinterpret_cast<const uint2*>(p.wt.Dh[cur] + dr));
          const uint2 dl = __ldcg(reinterpret_cast<const uint2*>(p.wt.Dl[cur] + dr));
          const float4 sg4 = __ldg(reinterpret_cast<const float4*>(p.sigma + i0));
          const float2 a0 = __half22float2(*reinterpret_cast<const __half2*>(&dh.x));
          const float2 a1 = __half22float2(*reinterpret_cast<const __half2*>(&dh.y));
          const float2 b0 = __half22float2(*reinterpret_cast<const __half2*>(&dl.x));
          const float2 b1 = __half22float2(*reinterpret_cast<const __half2*>(&dl.y));
          const float dv[4] = {(a0.x + b0.x) * sg4.x, (a0.y + b0.y) * sg4.y, (a1.x + b1.x) * sg4.z,
                               (a1.y + b1.y) * sg4.w};
#pragma unroll
          for (int u = 0; u < 4; ++u)       // x = d = 0 past n
            df_axpy(hi4[u], lo4[u], tw, i0 + u < p.n ? dv[u] : 0.0f);
          if (p.corr != nullptr) {
            // Exact null-space correction of the rounded direction (see projection).
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              if (i0 + u >= p.n) continue;
              float dlt = 0.0f;
              for (int q2 = 0; q2 < p.mE; ++q2)
                dlt = fmaf(p.Q32[static_cast<size_t>(q2) * p.n_ld + i0 + u],
                           p.corr[static_cast<size_t>(kk) * p.mE + q2], dlt);
              lo4[u] = fmaf(-tw, dlt, lo4[u]);
            }
          }
          *reinterpret_cast<float4*>(p.Xhi + xr) = make_float4(hi4[0], hi4[1], hi4[2], hi4[3]);
          *reinterpret_cast<float4*>(p.Xlo + xr) = make_float4(lo4[0], lo4[1], lo4[2], lo4[3]);
        }
        if (out != nullptr && kk < p.emit) {
          double* row = out + static_cast<size_t>(kk) * p.n + i0;
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (i0 + u < p.n) row[u] = static_cast<double>(hi4[u]) + static_cast<double>(lo4[u]);
        }
      }
    }

    // Every CTA is done with the pairs, the points and its tensor memory, and no
    // message is under way.
    tc_fence_before();
    __syncwarp();
    if constexpr (RUN) {
      cluster_sync_all();
    } else {
      // Every message to this CTA has arrived (c_full), and no other reads of it: nothing
      // to wait for but its own warps.
      if (warp < 2 || refresh) cluster_wait();
      __syncthreads();
      if (*timed_out && !refresh) {
        // An expired wait: messages may still be on their way.  Until the other CTAs are
        // here or have ended, and a bounded while for the messages.
        cluster_sync_all();
        if (threadIdx.x == 0)
          for (int i = 0; i < (1 << 14) && !mbar_try_wait(smem_u32(&tail->c_full), 0u); ++i) {}
        __syncthreads();
      }
    }
    tc_fence_after();
  }
  if (warp == 1) {
    const uint32_t cols = p.tiles_per_cta <= 1 ? 128u : (p.tiles_per_cta == 2 ? 256u : 512u);
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols)
                 : "memory");
  }
  if (p.step_out != nullptr && threadIdx.x == 0 && rank == 0 && strip == 0)
    *p.step_out = step0 + static_cast<uint64_t>(iters);
}

// Refresh operands: each walker's point x = hi + lo scaled by a power of two
// 2^e (max |x_i| 2^-e in [0.5, 1)) and split into FP16 hi + lo.
__global__ void split_points_kernel(int z, int z_ld, int n, int n_ld, int k_pad, const float* Xhi,
                                    const float* Xlo, __half* Xh, __half* Xl, float* wscale,
                                    const float* sigma) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k = blockIdx.x * (blockDim.x >> 5) + warp;
  if (k >= z_ld) return;
  float mx = 0.0f;
  if (k < z)
    for (int i = lane; i < n; i += 32)
      mx = fmaxf(mx, fabsf(Xhi[static_cast<size_t>(k) * n_ld + i]) / sigma[i]);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
  int ex = 0;
  if (mx > 0.0f) frexpf(mx, &ex);
  const float inv = ldexpf(1.0f, -ex);
  if (lane == 0) wscale[k] = ldexpf(1.0f, ex);
  for (int i = lane; i < k_pad; i += 32) {
    float v = 0.0f;
    if (k < z && i < n)
      v = (Xhi[static_cast<size_t>(k) * n_ld + i] + Xlo[static_cast<size_t>(k) * n_ld + i]) * inv /
          sigma[i];
    const __half h = __float2half_rn(v);
    Xh[static_cast<size_t>(k) * k_pad + i] = h;
    Xl[static_cast<size_t>(k) * k_pad + i] = __float2half_rn(v - __half2float(h));
  }
}

TcParams make_params(const mhar_ctx* c, const TcPlan* plan, int mode, int j, bool check_drift) {
  TcParams p;
  p.mode = mode;
  p.check_drift = check_drift ? 1 : 0;
  p.row_scale = c->d.row_scale;
  p.bS = c->d.bS;
  p.wscale = c->d.wscale;
  p.S = c->d.S;
  p.Xhi = c->d.Xhi;
  p.Xlo = c->d.Xlo;
  p.rowk = c->d.rowk;
  p.Xh = c->d.Xh;
  p.corrn = c->d.corrn;
  p.nx_ref = c->d.nx_ref;
  p.theta_acc = c->d.theta_acc;
  p.refresh_step = c->d.refresh_step;
  p.growth = 1.0f / static_cast<float>(4 * mma_chain(c) + 4);
  p.wt = make_walker_tail(c, 0);
  p.sigma = c->d.sigma;
  p.Q32 = c->d.Q32;
  p.corr = c->d.corr;
  p.lmin = c->d.lmin;
  p.lmax = c->d.lmax;
  p.theta = c->d.theta;
  p.status = c->d.status;
  p.counters = c->d.counters;
  p.err = c->d.status + 1;
  p.drift_key = reinterpret_cast<unsigned long long*>(c->d.check) + 2;
  p.seed = c->opts.seed;
  p.j = j;
  p.walker0 = c->opts.walker0;
  p.m = c->m;
  p.n = c->n;
  p.n_ld = c->n_ld;
  p.z = c->z;
  p.z_ld = plan->strips * kWalkers;
  p.kdim = c->kdim;
  p.k_chunks = c->k_pad / kTcKChunk;
  p.tiles_per_cta = plan->tiles_per_cta;
  p.m_tiles = plan->m_tiles;
  p.mE = c->mE;
  return p;
}

cudaError_t launch_walker_tc(mhar_ctx* c, int mode, int j, bool check_drift, const SmallRun* r) {
  const TcPlan* plan = static_cast<const TcPlan*>(c->tc);
  TcParams p = make_params(c, plan, mode, j, check_drift);
  p.step_ptr = r ? nullptr : c->d.step;
  p.step_out = r ? c->d.step : nullptr;
  p.step0 = r ? r->step : 0;
  p.iters = r ? r->iters : 1;
  p.out = r ? r->out : nullptr;
  p.emit = r ? r->emit : 0;
  p.thin = r ? r->thin : 1;
  p.phase = r ? r->phase : 0;
  p.wt.draw = r ? 1 : 0;       // a single iteration's directions were drawn before it
  // What the draw warps get done in an iteration, of 85 cycles an MMA, 3000 a row
  // tile for the slack and 9000 of the rest: a round of 64 items takes 3400.  The
  // epilogue warps draw the others while the first tile is on its way.
  const int cycles = p.tiles_per_cta * (4 * 85 * (p.kdim / kTcK) + 3000) + 9000;
  p.draw_items = cycles / 3400 * kDrawThreads;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(plan->C, plan->strips, 1);
  cfg.blockDim = dim3(r ? kThreadsTc : kThreadsOne, 1, 1);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = c->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = plan->C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (mode == kModeRefresh)
    return cudaLaunchKernelEx(&cfg, walker_tc_kernel<false>, plan->ah, plan->al, plan->xh, plan->xl,
                              plan->xh, plan->xl, p);
  const bool two = c->d.Dh2 != nullptr;      // pairs of even and odd iterations
  return cudaLaunchKernelEx(&cfg, r ? walker_tc_kernel<true> : walker_tc_kernel<false>, plan->ah, plan->al, plan->dh, plan->dl,
                            two ? plan->dh2 : plan->dh, two ? plan->dl2 : plan->dl, p);
}

}  // namespace

int tc_plan_create(mhar_ctx* c) {
  auto* plan = new TcPlan();
  plan->m_tiles = c->m_pad / kRowsTile;
  plan->tiles_per_cta = plan->m_tiles < kMaxTilesPerCta ? plan->m_tiles : kMaxTilesPerCta;
  plan->C = (plan->m_tiles + plan->tiles_per_cta - 1) / plan->tiles_per_cta;
  const int z_ld = (c->z + kWalkers - 1) / kWalkers * kWalkers;
  plan->strips = z_ld / kWalkers;
  if (plan->C > 16 && c->opts.precision == MHAR_MIXED_F16X3) {
    delete plan;
    snprintf(c->err, sizeof(c->err),
             "tensor-core mode covers m <= 8192 inequality rows (got m=%d)", c->m);
    return MHAR_E_UNSUPPORTED;
  }
  if (!make_map(&plan->ah, c->d.Ah, c->k_pad, c->m_pad) ||
      !make_map(&plan->al, c->d.Al, c->k_pad, c->m_pad) ||
      !make_map(&plan->dh, c->d.Dh, c->k_pad, z_ld) || !make_map(&plan->dl, c->d.Dl, c->k_pad, z_ld) ||
      (c->d.Dh2 && (!make_map(&plan->dh2, c->d.Dh2, c->k_pad, z_ld) ||
                    !make_map(&plan->dl2, c->d.Dl2, c->k_pad, z_ld))) ||
      !make_map(&plan->xh, c->d.Xh, c->k_pad, z_ld) || !make_map(&plan->xl, c->d.Xl, c->k_pad, z_ld)) {
    delete plan;
    snprintf(c->err, sizeof(c->err), "cuTensorMapEncodeTiled failed");
    return MHAR_E_CUDA;
  }
  cudaError_t e = cudaSuccess;
  for (auto k : {walker_tc_kernel<false>, walker_tc_kernel<true>}) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               static_cast<int>(kSmemBytes));
    if (e == cudaSuccess && plan->C > 8)
      e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  }
  if (e != cudaSuccess) {
    delete plan;
    snprintf(c->err, sizeof(c->err), "tensor-core kernel attributes: %s", cudaGetErrorString(e));
    return MHAR_E_CUDA;
  }
  c->tc = plan;
  return MHAR_OK;
}

void tc_plan_destroy(mhar_ctx* c) {
  delete static_cast<TcPlan*>(c->tc);
  c->tc = nullptr;
}

cudaError_t launch_chord_tc(mhar_ctx* c, int j) {
  return launch_walker_tc(c, kModeChord, j, false, nullptr);
}

cudaError_t launch_chord_tc_run(mhar_ctx* c, const SmallRun& r) {
  return launch_walker_tc(c, kModeChord, 0, false, &r);
}

cudaError_t launch_split_points(mhar_ctx* c) {
  const int z_ld = (c->z + kWalkers - 1) / kWalkers * kWalkers;
  split_points_kernel<<<(z_ld + 7) / 8, 256, 0, c->stream>>>(c->z, z_ld, c->n, c->n_ld, c->k_pad,
                                                          c->d.Xhi, c->d.Xlo, c->d.Xh, c->d.Xl,
                                                          c->d.wscale, c->d.sigma);
  return cudaGetLastError();
}

cudaError_t launch_refresh_tc(mhar_ctx* c, bool check_drift) {
  cudaError_t e = launch_split_points(c);
  if (e != cudaSuccess) return e;
  return launch_walker_tc(c, kModeRefresh, 0, check_drift, nullptr);
}

int tc_plan_strips(const mhar_ctx* c) { return static_cast<const TcPlan*>(c->tc)->strips; }
int tc_plan_m_tiles(const mhar_ctx* c) { return static_cast<const TcPlan*>(c->tc)->m_tiles; }

}  // namespace mhar
