// kernels_ts.cu -- the recompute-slack walker step with the walker operands
// resident in tensor memory (MHAR_MIXED_RECOMPUTE mode, n <= 128).
//
// Same arithmetic as kernels_rc.cu (Lemma 4.2 on the tensor cores: P = X A^T
// and G = D A^T from FP16 pairs, three products each, FP32 accumulation;
// s = b - p; the chord; theta), organised for the case where one walker's
// operands fit in tensor memory:
//   * the four walker operands (D hi/lo, X hi/lo: 128 walkers x k_pad FP16,
//     stored interleaved by 8-element chunks so the loads are coalesced)
//     are written once into tensor memory (256 columns) and serve as the A
//     operand of every MMA (tcgen05.mma with A in TMEM), so shared memory
//     only feeds the rows of A -- half the operand bytes per MMA of the
//     shared-memory form, which is what limited that form;
//   * the rows of A stream in 128-row tiles (MMA N = 128) through eight
//     16 KB slots, the hi and lo halves of one K chunk behind one barrier, up
//     to two tiles ahead;
//   * the G and P accumulators of a tile (128 + 128 columns) take the other
//     256 TMEM columns.  A tile's MMAs run as two passes, P first, then G,
//     each with its own full / empty barrier pair: the epilogue copies P to
//     registers while the G pass runs and releases it, so the next tile's P
//     pass follows the G pass without draining the tensor pipe, and likewise
//     for G.  The epilogue's ratio work on a tile overlaps the next tile's
//     MMAs.
// Measured on GB300: an MMA whose operands both come from shared memory needs
// the SM's whole shared-memory bandwidth at full rate, so the loads of the
// other warps and the TMA writes slow it; with A in tensor memory it needs
// half.
//   * one launch runs many iterations (SmallRun): a strip's walkers concern its
//     cluster alone.  The CTA's walkers' points stay in shared memory (TsParams::
//     resident) where they fit an item a thread, else every epilogue thread copies
//     its item in beside the tiles (cp.async); the rows of A for the next
//     iteration's first tiles arrive while the points move;
//   * two more warps draw the next directions beside the tiles, the epilogue warps
//     what those do not get done, between their last tile and theta;
//   * a partial chord goes from each epilogue warp to the CTA that holds the
//     walker as one message (st.async), theta needs no cluster barrier; one
//     barrier an iteration remains, behind which the moved points' FP16 pairs and
//     the next directions are read back from L2.
// An iteration of n = 100, m = 2000, z = 4096 takes 13.7 us (17.3 with one launch an
// iteration), n = 40, m = 400 with a rank-32 preconditioner 7.6 (25.7).  Of the 13.7
// (clock64): operands into tensor memory 1.1, four tiles 8.0 (100 cycles an MMA), the
// exchange and theta 1.0, the move 1.7, the barrier 1.0.  Drawing the directions
// before the tiles cost 2.4 us, 8 with the preconditioner; a barrier of the
// directions' own, so that a tile's G products could start before the points
// arrive, cost 1.2 us more than it hid.
// The cluster layout (C CTAs along the rows, 128 walkers per CTA), the arithmetic
// of the walker-side work (walker_tail.cuh) and the bounded waits are those of
// kernels_rc.cu.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <array>
#include <cstdio>
#include <type_traits>

#include "mhar_device.cuh"
#include "mhar_internal.h"
#include "tc_common.cuh"
#include "walker_tail.cuh"

namespace mhar {
namespace {

using namespace tc;

constexpr int kTile = 128;                           // MMA N: rows of A per tile
constexpr int kSlotBytes = kTile * kTcKChunk * 2;    // 128 x 64 FP16 = 16 KB
constexpr int kSlots = 8;                            // two tiles of A (hi, lo) ahead
constexpr int kPairs = kSlots / 2;                   // hi + lo of one K chunk per barrier
constexpr int kEpiWarps = 16;
constexpr int kEpiThreads = kEpiWarps * 32;
// Warps 18 and 19 draw the next directions beside the tiles.  Twenty warps are
// five on each sub-partition, as eighteen are on two: 96 registers either way.
constexpr int kDrawWarp = 2 + kEpiWarps;
constexpr int kDrawThreads = 64;
constexpr int kThreadsTs = kDrawWarp * 32 + kDrawThreads;
constexpr int kThreadsOne = kDrawWarp * 32;          // a single iteration draws nothing
constexpr int kMaxCluster = 8;
constexpr uint32_t kOpCol = 256;                     // first TMEM column of the walker operands

struct TsParams {
  const float* rows;        // 3 m_pad: b_i / row_scale_i and the error bounds (row_block)
  const float* wscale;      // z_ld
  const __half* Xh;         // z_ld x k_pad (operands copied into TMEM at start)
  const __half* Xl;
  double* lmin;
  double* lmax;
  double* theta;
  int* status;
  unsigned long long* counters;
  int* err;
  const uint64_t* step_ptr; // the iteration is *step_ptr + j, or (null) step0
  uint64_t* step_out;       // null, or where the next iteration's number goes
  uint64_t seed, step0;
  int j, iters;             // iterations of this launch
  double* out;              // samples, SmallRun's layout, or null
  int emit, thin, phase;
  uint32_t walker0;
  int resident;             // the walkers' points stay in shared memory (TsState)
  int draw_chunks;          // 8-coordinate chunks that the draw warps take; the epilogue warps the rest
  int n, z, z_ld, kdim, k_chunks, k_pad, tiles_per_cta, m_tiles;
  WalkerTail wt;            // walker-side work (walker_tail.cuh)
};

// Floats between two walkers' low-rank normals: 16-byte rows, and the rows that a
// quarter warp reads at once lie on different banks.
constexpr int kGStride = kMaxPcRank + 4;

struct alignas(16) TsTail {
  uint64_t a_full[kSlots];
  uint64_t a_empty[kSlots];
  uint64_t p_full, p_empty;    // P accumulator: MMAs done / copied out
  uint64_t g_full, g_empty;    // G accumulator
  uint64_t c_full;             // partial chords of this CTA's walkers
  uint32_t tmem_base;
  int timed_out;
  // (lambda_min, lambda_max) of a walker of this CTA from each epilogue warp
  // group of each CTA: [4 rank + group] [walker], rows of `share` walkers.
  float2 recv[4 * (kWalkers + kMaxCluster)];
  float theta_s[kWalkers];            // of the strip's walkers; this CTA's share is set
  double theta_u[kWalkers];           // the chord's uniform u (Philox stream 1), drawn early
  unsigned int red[kWalkers];         // this CTA's walkers: largest |x / sigma| (bits)
  float nrm[3][kWalkers];             // each walker's ||d_hat||_2, ||x_hat||_2, max |d_hat|
  alignas(16) float sigma[kWalkers];  // coordinate scales, and delta of a preconditioner
  alignas(16) float delta[kWalkers];
  alignas(16) float gs[kWalkers * kGStride];   // low-rank normals of a preconditioned draw
};

// The walker-side items.  Either (TsParams::resident) the points of the CTA's
// walkers for the whole launch: part p of item i, 16 bytes, at (512 p + i) 16, the
// parts X hi (2), X lo (2), D hi and D lo of pair 0, then of pair 1; or one slot
// per epilogue thread for its first item, staged in each iteration.
constexpr int kStateParts = 8;
constexpr size_t kStageBytes = static_cast<size_t>(kEpiThreads) * 16 * kStateParts;
static_assert(kStageBytes >= static_cast<size_t>(kEpiThreads) * kTailStageBytes, "stage slots");
constexpr size_t kSmemTs =
    1024 + static_cast<size_t>(kSlots) * kSlotBytes + sizeof(TsTail) + kStageBytes;
static_assert(kSmemTs <= 232448, "recompute_ts_kernel exceeds the shared memory of a CTA");

// A pair of floats into CTA `rank`'s copy of *local; counts on its barrier *bar.
__device__ __forceinline__ void push2(float2* local, uint64_t* bar, uint32_t rank, float x, float y) {
  uint32_t dst, rbar;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"(smem_u32(local)), "r"(rank));
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rbar) : "r"(smem_u32(bar)), "r"(rank));
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(
                   dst), "f"(x), "f"(y), "r"(rbar)
               : "memory");
}

__device__ __forceinline__ void arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// One 64-column K chunk of a tile's P pass (X hi, X lo times A hi; X hi
// times A lo) with KS K steps; pair use pu = p0 + kc holds A hi in half-slot
// 2 (pu % kPairs) and A lo in the next, behind one barrier (every wait, fence
// and commit on the issuing thread's path costs issue time).
template <int KS>
__device__ __forceinline__ void ts_p_chunk(TsTail* tail, uint8_t* base, int p0, int kc,
                                           uint32_t p_tmem, uint32_t op_xh, uint32_t op_xl,
                                           uint32_t idesc, volatile int* timed_out, int* err) {
  const int pu = p0 + kc, ps = pu % kPairs;
  const uint32_t ac0 = static_cast<uint32_t>(kc * 32);   // 2 FP16 per column
  mbar_wait(&tail->a_full[ps], (pu / kPairs) & 1, timed_out, err);
  tc_fence_after();
  // A slot's descriptor is built once; a K step of 16 FP16 adds 2 to it (32 bytes).
  const uint64_t bh = sw128_desc(smem_u32(base + (2 * ps) * kSlotBytes));
  const uint64_t bl = sw128_desc(smem_u32(base + (2 * ps + 1) * kSlotBytes));
  mma_ts_run2<KS>(p_tmem, op_xh + ac0, op_xl + ac0, bh, idesc, kc > 0 ? 1u : 0u);
  mma_ts_run1<KS>(p_tmem, op_xh + ac0, bl, idesc);
}

// The same chunk of the G pass (D hi, D lo times A hi; D hi times A lo); the
// pair was waited for by the P pass and is released here.
template <int KS>
__device__ __forceinline__ void ts_g_chunk(TsTail* tail, uint8_t* base, int p0, int kc,
                                           uint32_t g_tmem, uint32_t op_dh, uint32_t op_dl,
                                           uint32_t idesc) {
  const int pu = p0 + kc, ps = pu % kPairs;
  const uint32_t ac0 = static_cast<uint32_t>(kc * 32);
  const uint64_t bh = sw128_desc(smem_u32(base + (2 * ps) * kSlotBytes));
  const uint64_t bl = sw128_desc(smem_u32(base + (2 * ps + 1) * kSlotBytes));
  mma_ts_run2<KS>(g_tmem, op_dh + ac0, op_dl + ac0, bh, idesc, kc > 0 ? 1u : 0u);
  mma_ts_run1<KS>(g_tmem, op_dh + ac0, bl, idesc);
  mma_commit(&tail->a_empty[ps]);
}

// ---- walker-side work ---------------------------------------------------------
// The arithmetic is that of walker_tail.cuh.  Items are (8-coordinate chunk,
// walker), the walker fastest.

// Iteration `step`'s directions into pair `to`: the items (group of 4 Q
// coordinates, walker), the walker fastest, first, first + stride, ... < last; with
// a preconditioner the low-rank normals are in gs.
template <int Q>
__device__ __forceinline__ void ts_draw(const WalkerTail& t, int to, uint64_t seed, uint64_t step,
                                        uint32_t walker0, int strip, int z, int w_begin,
                                        int w_count, int first, int last, int stride,
                                        const TsTail* tail, uint4* state) {
  using namespace tail_detail;
  using Vec = std::conditional_t<Q == 2, uint4, uint2>;
#pragma unroll 1
  for (int it = first; it < last; it += stride) {
    const int c = it / w_count, wo = it - c * w_count;
    const int k = strip * kWalkers + w_begin + wo;
    if (k >= z) continue;
    const int i0 = 4 * Q * c;
    float v[4 * Q] = {};
#pragma unroll
    for (int h = 0; h < Q; ++h)
      if (i0 + 4 * h < t.n) {
        const U4 w = philox_block(seed, step, walker0 + static_cast<uint32_t>(k),
                                  static_cast<uint32_t>(Q * c + h), kStreamDirection);
        box_muller_f32(w.x, w.y, v[4 * h], v[4 * h + 1]);
        box_muller_f32(w.z, w.w, v[4 * h + 2], v[4 * h + 3]);
      }
    if (t.pc_rank >= 0) {
      // Rows of U four columns at a time, the sums side by side (scalar loads,
      // one sum after the other, took 14500 cycles for eight).
      const float* g = tail->gs + wo * kGStride;
      const float4* u4 = reinterpret_cast<const float4*>(t.pc_U + static_cast<size_t>(i0) * kMaxPcRank);
#pragma unroll
      for (int e = 0; e < 4 * Q; ++e) v[e] *= tail->delta[i0 + e];
#pragma unroll 2
      for (int c4 = 0; c4 < kMaxPcRank / 4; ++c4) {
        const float4 g4 = *reinterpret_cast<const float4*>(g + 4 * c4);
#pragma unroll
        for (int e = 0; e < 4 * Q; ++e) {      // rows of U up to n_ld, zero past n
          const float4 u = __ldg(u4 + e * (kMaxPcRank / 4) + c4);
          v[e] = fmaf(u.w, g4.w, fmaf(u.z, g4.z, fmaf(u.y, g4.y, fmaf(u.x, g4.x, v[e]))));
        }
      }
    }
    // The FP16 pair holds d_i / sigma_i (sigma a power of two: exact).
    alignas(16) __half2 h[2 * Q];
    alignas(16) __half2 l[2 * Q];
    bool bad = false;
#pragma unroll
    for (int e = 0; e < 4 * Q; e += 2) {
      const float a = i0 + e < t.n ? v[e] * pow2_recip(tail->sigma[i0 + e]) : 0.0f;
      const float b = i0 + e + 1 < t.n ? v[e + 1] * pow2_recip(tail->sigma[i0 + e + 1]) : 0.0f;
      h[e / 2] = __floats2half2_rn(a, b);
      l[e / 2] = __floats2half2_rn(a - __low2float(h[e / 2]), b - __high2float(h[e / 2]));
      bad |= !(fabsf(a) <= kHalfMax) || !(fabsf(b) <= kHalfMax);
    }
    if (bad) atomicOr(t.status, MHAR_ST_NONFINITE);
    const Vec hv = *reinterpret_cast<const Vec*>(h), lv = *reinterpret_cast<const Vec*>(l);
    const size_t o = op_off(k, i0, t.k_pad, t.z_ld, 1);
    *reinterpret_cast<Vec*>(t.Dh[to] + o) = hv;
    *reinterpret_cast<Vec*>(t.Dl[to] + o) = lv;
    if (state != nullptr) {
      Vec* part = reinterpret_cast<Vec*>(state + (4 + 2 * to) * kEpiThreads + (i0 >> 3) * w_count + wo);
      const int half = Q == 2 ? 0 : c & 1;
      part[half] = hv;
      part[(2 / Q) * kEpiThreads + half] = lv;
    }
  }
}

// The low-rank normals of the CTA's walkers (Philox stream 2), by `threads` threads.
__device__ __forceinline__ void ts_lowrank(const WalkerTail& t, uint64_t seed, uint64_t step,
                                           uint32_t walker0, int strip, int z, int w_begin,
                                           int w_count, int tid, int threads, float* gs) {
  const int quads = (t.pc_rank + 3) >> 2;
  for (int idx = tid; idx < w_count * (kMaxPcRank / 4); idx += threads) {
    const int w = idx / (kMaxPcRank / 4), q = idx - w * (kMaxPcRank / 4);
    const int k = strip * kWalkers + w_begin + w;
    float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    if (q < quads && k < z) {
      const U4 r = philox_block(seed, step, walker0 + static_cast<uint32_t>(k),
                                static_cast<uint32_t>(q), kStreamLowRank);
      box_muller_f32(r.x, r.y, v[0], v[1]);
      box_muller_f32(r.z, r.w, v[2], v[3]);
    }
    float4 o;
    o.x = 4 * q < t.pc_rank ? v[0] : 0.0f;
    o.y = 4 * q + 1 < t.pc_rank ? v[1] : 0.0f;
    o.z = 4 * q + 2 < t.pc_rank ? v[2] : 0.0f;
    o.w = 4 * q + 3 < t.pc_rank ? v[3] : 0.0f;
    *reinterpret_cast<float4*>(gs + w * kGStride + 4 * q) = o;
  }
}

// Resident points: thread `tid`'s item into shared memory at the start, and
// its direction of pair `cur`.
__device__ __forceinline__ void ts_load_state(const WalkerTail& t, int cur, int strip, int z,
                                              int w_begin, int w_count, int tid, uint4* state) {
  const int c = tid / w_count, wo = tid - c * w_count, i0 = 8 * c;
  const int k = strip * kWalkers + w_begin + wo;
  if (i0 >= t.n || k >= z) return;
  const size_t xr = static_cast<size_t>(k) * t.n_ld + i0;
  const size_t o = op_off(k, i0, t.k_pad, t.z_ld, 1);
  const uint4* hi = reinterpret_cast<const uint4*>(t.Xhi + xr);
  const uint4* lo = reinterpret_cast<const uint4*>(t.Xlo + xr);
  state[tid] = hi[0];
  state[kEpiThreads + tid] = hi[1];
  state[2 * kEpiThreads + tid] = lo[0];
  state[3 * kEpiThreads + tid] = lo[1];
  state[(4 + 2 * cur) * kEpiThreads + tid] = *reinterpret_cast<const uint4*>(t.Dh[cur] + o);
  state[(5 + 2 * cur) * kEpiThreads + tid] = *reinterpret_cast<const uint4*>(t.Dl[cur] + o);
}

// The move and the split of resident points; `red` is zero at the start.
// out: where the walker's sample goes (null: none).  save: the points go back
// to global memory.
__device__ __forceinline__ void ts_move_resident(const WalkerTail& t, int cur, int strip, int z,
                                                 int w_begin, int c, int wo, int tid,
                                                 TsTail* tail, uint4* state, double* out, int emit,
                                                 bool save) {
  using namespace tail_detail;
  const int i0 = 8 * c;
  unsigned int* red = tail->red;
  const int k = strip * kWalkers + w_begin + wo;
  const bool mine = i0 < t.n && k < z;
  float v[8] = {};
  float hi[8] = {}, lo[8] = {};
  if (mine) {
    float sg[8];
    ld8(tail->sigma + i0, sg);
    const float th = tail->theta_s[w_begin + wo];
    ld8(reinterpret_cast<const float*>(state + tid), hi, kEpiThreads);
    ld8(reinterpret_cast<const float*>(state + 2 * kEpiThreads + tid), lo, kEpiThreads);
    if (th != 0.0f) {
      float dh[8], dl[8];
      ld8h(reinterpret_cast<const __half*>(state + (4 + 2 * cur) * kEpiThreads + tid), dh);
      ld8h(reinterpret_cast<const __half*>(state + (5 + 2 * cur) * kEpiThreads + tid), dl);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        df_axpy(hi[e], lo[e], th, i0 + e < t.n ? (dh[e] + dl[e]) * sg[e] : 0.0f);
      }
      st8(reinterpret_cast<float*>(state + tid), hi, kEpiThreads);
      st8(reinterpret_cast<float*>(state + 2 * kEpiThreads + tid), lo, kEpiThreads);
    }
    float mx = 0.0f;
#pragma unroll
    for (int e = 0; e < 8; ++e) {   // x = 0 and sigma = 1 past n
      v[e] = pow2_recip(sg[e]);
      mx = fmaxf(mx, fabsf(hi[e]) * v[e]);
    }
    atomicMax(red + wo, __float_as_uint(mx));  // non-negative floats order as their bits
  }
  named_bar<kEpiThreads>();
  if (!mine) return;
  const unsigned int mb = red[wo];
  float inv, ws;
  const int ex = static_cast<int>(mb >> 23) - 126;     // frexp's exponent of a normal value
  if (mb >= 0x00800000u && ex >= -126 && ex <= 126) {
    inv = __int_as_float((127 - ex) << 23);
    ws = __int_as_float((127 + ex) << 23);
  } else {
    int e2 = 0;
    if (mb > 0u) frexpf(__uint_as_float(mb), &e2);
    inv = ldexpf(1.0f, -e2);
    ws = ldexpf(1.0f, e2);
  }
  if (c == 0) t.wscale[k] = ws;
#pragma unroll
  for (int e = 0; e < 8; ++e) v[e] = (hi[e] + lo[e]) * inv * v[e];
  const size_t o = op_off(k, i0, t.k_pad, t.z_ld, 1);
  if (split_store8(v, t.Xh + o, t.Xl + o)) atomicOr(t.status, MHAR_ST_NONFINITE);
  if (out != nullptr && k < emit) {
    double* row = out + static_cast<size_t>(k) * t.n + i0;
#pragma unroll
    for (int e = 0; e < 8; ++e)
      if (i0 + e < t.n) row[e] = static_cast<double>(hi[e]) + static_cast<double>(lo[e]);
  }
  if (save) {
    const size_t xr = static_cast<size_t>(k) * t.n_ld + i0;
    st8(t.Xhi + xr, hi);
    st8(t.Xlo + xr, lo);
  }
}

// Points too many for shared memory, and iterations with equalities:
// walker_tail on the points in global memory.
__device__ __forceinline__ void ts_move(const WalkerTail& wt, int cur, int strip, int z, int w_begin,
                                        int w_count, int tid, TsTail* tail, uint8_t* stage) {
  // Initialised: in the loop over the iterations an item that a thread does not
  // have would be kept from one to the next (444 bytes of spills, with the
  // like of it in the operands' second chunk).
  TailItem item = {};   // this thread's first tail item
  walker_tail_unstage<kEpiThreads>(wt, strip, z, w_begin, w_count, tid,
                                   stage + tid * kTailStageBytes, item);
  // The stage is free after the tail's first barrier: route the moved rows
  // through it when they fit.
  const bool rows_fit =
      static_cast<size_t>(2 * w_count) * tail_row_stride(wt.n_ld) * sizeof(float) <= kStageBytes;
  walker_tail<kEpiThreads>(wt, cur, strip, z, w_begin, w_count, tail->theta_s, tail->red, tid, item,
                           rows_fit ? reinterpret_cast<float*>(stage) : nullptr);
}

// KCH: 64-column K chunks of A's rows (1 or 2: n <= 128); LAST: K steps (16
// FP16 each) in the last chunk, 1..4, the other chunk having 4.  A
// compile-time K structure makes each pass one straight run of MMAs (the
// issuing thread's stream between MMAs is the limiter).
// RUN: many iterations, and the draws; else one iteration whose directions a kernel
// before it drew and projected (equalities), without what only the loop needs and without
// its two cluster barriers.  One kernel for both took an iteration with an equality 22.5 us
// on 294 walkers of a 2229 x 51 body, 18.1 now, 30.5 and 27.3 on 4096 of a 2000 x 100 body;
// the loop gains too (illcond40x400 with rank 32, 100 iterations: 785 -> 764 us).
template <int KCH, int LAST, bool RUN>
__global__ void __launch_bounds__(RUN ? kThreadsTs : kThreadsOne, 1)
recompute_ts_kernel(const __grid_constant__ CUtensorMap tm_ah, const __grid_constant__ CUtensorMap tm_al,
                    const __grid_constant__ TsParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  TsTail* tail = reinterpret_cast<TsTail*>(base + kSlots * kSlotBytes);
  uint8_t* stage = reinterpret_cast<uint8_t*>(tail + 1);   // 16-byte aligned

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int csz_i = static_cast<int>(gridDim.x);
  const int share = (kWalkers + csz_i - 1) / csz_i;   // walkers of this CTA's walker-side work
  const int w_begin = static_cast<int>(blockIdx.x) * share;
  const int w_count = max(0, min(share, kWalkers - w_begin));
  const uint32_t rank = blockIdx.x;
  const int strip = blockIdx.y;
  const int tile0 = static_cast<int>(rank) * p.tiles_per_cta;
  int ntiles = p.m_tiles - tile0;
  ntiles = ntiles < 0 ? 0 : (ntiles > p.tiles_per_cta ? p.tiles_per_cta : ntiles);
  const int row_base = tile0 * kTile;

  if (threadIdx.x == 32) {
    prefetch_tmap(&tm_ah);
    prefetch_tmap(&tm_al);
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < kSlots; ++s) { mbar_init(&tail->a_full[s], 1); mbar_init(&tail->a_empty[s], 1); }
    mbar_init(&tail->p_full, 1);
    mbar_init(&tail->p_empty, kEpiWarps);
    mbar_init(&tail->g_full, 1);
    mbar_init(&tail->g_empty, kEpiWarps);
    mbar_init(&tail->c_full, 1);
    tail->timed_out = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tail->tmem_base)), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncwarp();
  if constexpr (RUN) {
    cluster_sync_all();   // every CTA's barriers are ready
  } else {
    cluster_arrive();     // waited for before the first message to one of them
    __syncthreads();
  }
  tc_fence_after();
  const uint32_t tmem = tail->tmem_base;
  volatile int* timed_out = &tail->timed_out;
  // Launched as a programmatic dependent of the previous iteration's kernel:
  // the set-up above overlaps its end; nothing it wrote is read before this.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (threadIdx.x == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const uint64_t step0 = p.step_ptr != nullptr ? *p.step_ptr + static_cast<uint64_t>(p.j) : p.step0;
  const int tid = static_cast<int>(threadIdx.x) - 64;   // of the epilogue, then the draw threads
  const int my_c = tid / w_count, my_w = tid - my_c * w_count;   // a resident thread's item
  const int theta_threads = (w_count + 31) & ~31;
  const int quads = RUN && p.wt.draw ? ((p.wt.n + 7) >> 3) * 2 * w_count : 0;
  const int epi_draws = kEpiThreads - theta_threads;             // threads that draw after the tiles
  uint4* state = RUN && p.resident ? reinterpret_cast<uint4*>(stage) : nullptr;
  const int iters = RUN ? p.iters : 1;
  if constexpr (RUN) {
    if (tid >= 0 && tid < kWalkers) {
      const bool in = tid < p.wt.n_ld;
      tail->sigma[tid] = in ? p.wt.sigma[tid] : 1.0f;
      tail->delta[tid] = in && p.wt.pc_rank >= 0 ? p.wt.pc_delta[tid] : 0.0f;
    }
    __syncthreads();
  }
  if (state != nullptr && warp >= 2 && warp < kDrawWarp)
    ts_load_state(p.wt, static_cast<int>(step0 & 1ull), strip, p.z, w_begin, w_count, tid, state);
  int pu = 0;                // producer: pair uses issued
  int p0 = 0;                // MMA thread: first pair use of the tile
  int g = 0;                 // tiles of the iterations before
#pragma unroll 1
  for (int it = 0; it < iters; ++it, g += ntiles) {
    const uint64_t step = step0 + static_cast<uint64_t>(it);
    const int cur = static_cast<int>(step & 1ull);  // this iteration's direction pair

    // ---- walker operands into tensor memory: warp (quarter q, operand op) ------
    // writes its 32 walkers' row of operand op, 2 FP16 per 32-bit column.
    if (warp >= 2 && warp < kDrawWarp) {
      const int e = warp - 2;
      const int q = warp & 3;
      const int op = e >> 2;
      const int k = strip * kWalkers + q * 32 + lane;
      const __half* src = op == 0 ? p.wt.Dh[cur] : op == 1 ? p.wt.Dl[cur] : op == 2 ? p.Xh : p.Xl;
      // Operands are interleaved by 8-element chunks: chunk c of walker k is the
      // 16 bytes at (c z_ld + k) 16, so each load below is one contiguous
      // 512-byte line for the warp.
      const uint4* ops = reinterpret_cast<const uint4*>(src);
      const uint32_t col0 = kOpCol + static_cast<uint32_t>(op * 64);
      const uint32_t lane_off = static_cast<uint32_t>(q * 32) << 16;
      uint32_t r0[32], r1[32];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const uint4 v = __ldcg(ops + static_cast<size_t>(i) * p.z_ld + k);
        r0[4 * i] = v.x; r0[4 * i + 1] = v.y; r0[4 * i + 2] = v.z; r0[4 * i + 3] = v.w;
      }
      if constexpr (KCH == 2) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const uint4 v = __ldcg(ops + static_cast<size_t>(8 + i) * p.z_ld + k);
          r1[4 * i] = v.x; r1[4 * i + 1] = v.y; r1[4 * i + 2] = v.z; r1[4 * i + 3] = v.w;
        }
      }
      tmem_st32(tmem + lane_off + col0, r0);
      if constexpr (KCH == 2) tmem_st32(tmem + lane_off + col0 + 32u, r1);
      tmem_st_wait();
      tc_fence_before();
      // Operands ready: release the MMA warp (the producer never waits on this).
      asm volatile("bar.arrive 2, %0;" ::"n"((kEpiWarps + 1) * 32) : "memory");
      if (op == 0 || op == 2) {
        // The 2-norm bound of the walker's direction (op 0) or scaled point
        // (op 2) from its FP16 hi row, for the chord's error margins.
        // Sums of squares in chunk order: the same bits as operand_norms in the
        // shared-memory-operand kernels.
        float ss = 0.0f, mx = 0.0f;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const uint4 u = make_uint4(r0[4 * i], r0[4 * i + 1], r0[4 * i + 2], r0[4 * i + 3]);
          ss += sumsq8(u);
          mx = fmaxf(mx, absmax8(u));
        }
        if constexpr (KCH == 2) {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const uint4 u = make_uint4(r1[4 * i], r1[4 * i + 1], r1[4 * i + 2], r1[4 * i + 3]);
            ss += sumsq8(u);
            mx = fmaxf(mx, absmax8(u));
          }
        }
        tail->nrm[op >> 1][q * 32 + lane] = norm_bound(ss);
        if (op == 0) tail->nrm[2][q * 32 + lane] = mx * 1.00390625f;
      }
    }

    if (warp == 0) {
      // ---- TMA producer: A rows, 64-row tiles, hi and lo in separate slots ------
      if (lane == 0) {
        // This iteration's tiles and the first of the next one's, which then
        // arrive while the walkers move.
        const int per = ntiles * KCH;
        const int end = min(iters * per, (it + 1) * per + kPairs);
        for (; pu < end; ++pu) {
          const int s = pu % kPairs, nt = (pu / KCH) % ntiles, kc = pu % KCH;
          const int yr = row_base + nt * kTile;
          if (pu >= kPairs) mbar_wait(&tail->a_empty[s], ((pu / kPairs) - 1) & 1, timed_out, p.err);
          mbar_expect_tx(&tail->a_full[s], 2 * kSlotBytes);
          tma_load_2d(base + (2 * s) * kSlotBytes, &tm_ah, &tail->a_full[s], kc * kTcKChunk, yr);
          tma_load_2d(base + (2 * s + 1) * kSlotBytes, &tm_al, &tail->a_full[s], kc * kTcKChunk, yr);
        }
      }
      __syncwarp();
    } else if (warp == 1) {
      // ---- MMA issuer ------------------------------------------------------------
      asm volatile("bar.sync 2, %0;" ::"n"((kEpiWarps + 1) * 32) : "memory");
      tc_fence_after();
      if (lane == 0) {
        constexpr uint32_t idesc = make_idesc(kWalkers, kTile);
        const uint32_t op_dh = tmem + kOpCol, op_dl = op_dh + 64u, op_xh = op_dh + 128u,
                       op_xl = op_dh + 192u;
        const uint32_t g_tmem = tmem;
        const uint32_t p_tmem = tmem + 128u;
        for (int nt = 0; nt < ntiles; ++nt, p0 += KCH) {
          // P pass: X hi, X lo times A hi; X hi times A lo.  The accumulator is
          // free once the epilogue has copied the previous tile's P out.
          if (g + nt >= 1) mbar_wait(&tail->p_empty, (g + nt - 1) & 1, timed_out, p.err);
          tc_fence_after();
          if constexpr (KCH == 2)
            ts_p_chunk<4>(tail, base, p0, 0, p_tmem, op_xh, op_xl, idesc, timed_out, p.err);
          ts_p_chunk<LAST>(tail, base, p0, KCH - 1, p_tmem, op_xh, op_xl, idesc, timed_out, p.err);
          mma_commit(&tail->p_full);
          // G pass: D hi, D lo times A hi; D hi times A lo.  Each slot is
          // released after its last use here.
          if (g + nt >= 1) mbar_wait(&tail->g_empty, (g + nt - 1) & 1, timed_out, p.err);
          tc_fence_after();
          if constexpr (KCH == 2) ts_g_chunk<4>(tail, base, p0, 0, g_tmem, op_dh, op_dl, idesc);
          ts_g_chunk<LAST>(tail, base, p0, KCH - 1, g_tmem, op_dh, op_dl, idesc);
          mma_commit(&tail->g_full);
        }
      }
      __syncwarp();
    } else if (warp >= kDrawWarp) {
      // ---- iteration s+1's directions into the other pair ------------------------
      const int dt = tid - kEpiThreads;
      if (quads > 0 && p.wt.pc_rank >= 0) {
        ts_lowrank(p.wt, p.seed, step + 1ull, p.walker0, strip, p.z, w_begin, w_count, dt,
                   kDrawThreads, tail->gs);
        asm volatile("bar.sync 4, %0;" ::"n"(kDrawThreads) : "memory");
        if (2 * p.draw_chunks * w_count < quads)
          asm volatile("bar.arrive 3, %0;" ::"r"(epi_draws + kDrawThreads) : "memory");
      }
      ts_draw<2>(p.wt, cur ^ 1, p.seed, step + 1ull, p.walker0, strip, p.z, w_begin, w_count, dt,
                 min(p.draw_chunks * w_count, quads / 2), kDrawThreads, tail, state);
    } else {
      // ---- epilogue: s = b - p, ratios, per-walker partial chord ------------------
      const int e = warp - 2;
      const int q = warp & 3;
      const int cg = e >> 2;              // 32-column group of each 128-column tile
      const int row0 = row_base + cg * 32;
      if (lane < 4 && ntiles > 0) prefetch_l1(row_block(p.rows, row0) + 32 * lane);
      if (tid == 0)
        mbar_expect_tx(&tail->c_full, static_cast<uint32_t>(4 * csz_i * w_count * sizeof(float2)));
      // This thread's walker-side item, copied to shared memory in the background.
      if (state == nullptr)
        walker_tail_stage<kEpiThreads>(p.wt, cur, strip, p.z, w_begin, w_count, tid,
                                       stage + tid * kTailStageBytes);
      if (tid < w_count) {
        // The chord's uniform does not depend on the chord: draw it now.
        const int kk = strip * kWalkers + w_begin + tid;
        const U4 w = philox_block(p.seed, step, p.walker0 + static_cast<uint32_t>(kk), 0u,
                                  kStreamChord);
        tail->theta_u[tid] = open_unit_f64(w.x);
        tail->red[tid] = 0u;
      }
      const int wl = q * 32 + lane;
      const int k = strip * kWalkers + wl;
      const float ws = __ldcg(p.wscale + k);
      // The operand norms of this thread's walker (written by the warps that
      // loaded the operands into tensor memory).
      named_bar<kEpiWarps * 32>();
      WalkerNorms wn;
      wn.nd2 = tail->nrm[0][wl];
      wn.nxw2 = ws * tail->nrm[1][wl];
      wn.ws = ws;
      wn.ndinf = tail->nrm[2][wl];
      if (k < p.z) add_correction(p.wt, k, wn);
      ChordAcc acc;
      acc.init();
      const uint32_t lane_off = static_cast<uint32_t>(q * 32) << 16;
      const uint32_t gcol = tmem + lane_off + static_cast<uint32_t>(cg * 32);
#pragma unroll 1
      for (int nt = 0; nt < ntiles; ++nt) {
        // P first (its pass ends first), then G; each accumulator is released
        // as soon as it is in registers.
        if (lane < 4 && nt + 1 < ntiles) prefetch_l1(row_block(p.rows, row0 + (nt + 1) * kTile) + 32 * lane);
        float sv[32], gv[32];
        mbar_wait(&tail->p_full, (g + nt) & 1, timed_out, p.err);
        tc_fence_after();
        tmem_ld32(gcol + 128u, sv);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) arrive(&tail->p_empty);
        // The slacks while the G pass finishes.
        float fx, fd;
        wn.pick(p.rows, row0 + nt * kTile, fx, fd);
        slack32(sv, p.rows, row0 + nt * kTile, ws, fx);
        mbar_wait(&tail->g_full, (g + nt) & 1, timed_out, p.err);
        tc_fence_after();
        tmem_ld32(gcol, gv);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) arrive(&tail->g_empty);
        scan32(sv, gv, p.rows, row0 + nt * kTile, fd, acc);
      }
      // The partial chord to the CTA that holds the walker: the data and its
      // arrival in one message (a cluster barrier took 1500 cycles here).
      if constexpr (!RUN) {
        __syncwarp();
        cluster_wait();
      }
      {
        const int owner = wl / share;
        push2(&tail->recv[(4 * static_cast<int>(rank) + cg) * share + wl - owner * share],
              &tail->c_full, static_cast<uint32_t>(owner), acc.lo_all(), acc.hi_all());
      }
      if (tid < w_count) {
        mbar_wait(&tail->c_full, it & 1, timed_out, p.err);
        const int kk = strip * kWalkers + w_begin + tid;
        float L = -INFINITY, H = INFINITY;
        for (int r = 0; r < 4 * csz_i; ++r) {
          const float2 v = tail->recv[r * share + tid];
          L = fmaxf(L, v.x);
          H = fminf(H, v.y);
        }
        float t = 0.0f;
        if (kk < p.z) {
          int flag = 0;
          if (isinf(L) || isinf(H)) {
            flag = MHAR_ST_UNBOUNDED;
          } else if (L > H) {
            flag = MHAR_ST_STALL;
          } else {
            const double u = tail->theta_u[tid];
            t = static_cast<float>(static_cast<double>(L) +
                                   u * (static_cast<double>(H) - static_cast<double>(L)));
          }
          if (it + 1 == iters) {
            p.lmin[kk] = L;
            p.lmax[kk] = H;
            p.theta[kk] = t;
          }
          if (flag) {
            atomicOr(p.status, flag);
            atomicAdd(&p.counters[flag == MHAR_ST_STALL ? 0 : 1], 1ull);
          }
        }
        tail->theta_s[w_begin + tid] = t;
      } else if (tid >= theta_threads && 2 * p.draw_chunks * w_count < quads) {
        // The other warps draw their quads of iteration s+1's directions while
        // the chords are on their way.
        if (p.wt.pc_rank >= 0)
          asm volatile("bar.sync 3, %0;" ::"r"(epi_draws + kDrawThreads) : "memory");
        ts_draw<1>(p.wt, cur ^ 1, p.seed, step + 1ull, p.walker0, strip, p.z, w_begin, w_count,
                   2 * p.draw_chunks * w_count + tid - theta_threads, quads, epi_draws, tail, state);
      }
      named_bar<kEpiThreads>();
      // Algorithm 2's thinning: a sample after this iteration?
      const int done = p.phase + it + 1;
      double* out = RUN && p.out != nullptr && done % p.thin == 0
                        ? p.out + static_cast<size_t>(done / p.thin - 1) * p.emit * p.n
                        : nullptr;
      if (state != nullptr) {
        ts_move_resident(p.wt, cur, strip, p.z, w_begin, my_c, my_w, tid, tail, state, out, p.emit,
                         it + 1 == iters);
      } else {
        ts_move(p.wt, cur, strip, p.z, w_begin, w_count, tid, tail, stage);
        if (out != nullptr) {   // this CTA's walkers, a warp per row
          named_bar<kEpiThreads>();
          for (int w = warp - 2; w < w_count; w += kEpiWarps) {
            const int kk = strip * kWalkers + w_begin + w;
            if (kk >= p.emit) break;
            const float* hi = p.wt.Xhi + static_cast<size_t>(kk) * p.wt.n_ld;
            const float* lo = p.wt.Xlo + static_cast<size_t>(kk) * p.wt.n_ld;
            for (int i = lane; i < p.n; i += 32)
              out[static_cast<size_t>(kk) * p.n + i] =
                  static_cast<double>(hi[i]) + static_cast<double>(lo[i]);
          }
        }
      }
    }
    // The cluster's points and directions, and this CTA's shared memory, are
    // ready for the next iteration (at the end: no message is still under way).
    tc_fence_before();
    __syncwarp();
    if constexpr (RUN) {
      cluster_sync_all();
    } else {
      // Every message to this CTA has arrived (c_full), and no other reads of it: nothing
      // to wait for but its own warps.
      if (warp < 2) cluster_wait();
      __syncthreads();
      if (*timed_out) {
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
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u)
                 : "memory");
  }
  if (p.step_out != nullptr && threadIdx.x == 0 && rank == 0 && strip == 0)
    *p.step_out = step0 + static_cast<uint64_t>(iters);
}

struct TsShape {
  int C = 1;
  int tiles_per_cta = 1;
  int m_tiles = 1;
};

TsShape ts_shape(const mhar_ctx* c, const TcPlan* plan) {
  int sms = 148;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
  TsShape s;
  s.m_tiles = c->m_pad / kTile;
  int C = sms / plan->strips;
  C = C < 1 ? 1 : (C > kMaxCluster ? kMaxCluster : C);
  C = C > s.m_tiles ? s.m_tiles : C;
  s.tiles_per_cta = (s.m_tiles + C - 1) / C;
  s.C = (s.m_tiles + s.tiles_per_cta - 1) / s.tiles_per_cta;
  return s;
}

// Instantiations by (one iteration, many), then by (chunks, last-chunk K steps): index
// 4 (KCH - 1) + LAST - 1.
using TsKernel = void (*)(CUtensorMap, CUtensorMap, TsParams);
template <bool RUN>
constexpr std::array<TsKernel, 8> ts_kernels() {
  return {recompute_ts_kernel<1, 1, RUN>, recompute_ts_kernel<1, 2, RUN>,
          recompute_ts_kernel<1, 3, RUN>, recompute_ts_kernel<1, 4, RUN>,
          recompute_ts_kernel<2, 1, RUN>, recompute_ts_kernel<2, 2, RUN>,
          recompute_ts_kernel<2, 3, RUN>, recompute_ts_kernel<2, 4, RUN>};
}
constexpr std::array<TsKernel, 8> kTsKernels[2] = {ts_kernels<false>(), ts_kernels<true>()};

}  // namespace

bool ts_eligible(const mhar_ctx* c) { return c->k_pad <= 128; }

int ts_prepare(mhar_ctx* c) {
  auto* plan = static_cast<TcPlan*>(c->tc);
  if (!make_map_rows(&plan->ah64, c->d.Ah, c->k_pad, c->m_pad, kTile) ||
      !make_map_rows(&plan->al64, c->d.Al, c->k_pad, c->m_pad, kTile)) {
    snprintf(c->err, sizeof(c->err), "cuTensorMapEncodeTiled failed (64-row maps)");
    return MHAR_E_CUDA;
  }
  cudaError_t e = cudaSuccess;
  for (const auto& form : kTsKernels)
    for (TsKernel k : form)
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               static_cast<int>(kSmemTs));
  if (e != cudaSuccess) {
    snprintf(c->err, sizeof(c->err), "recompute (TMEM operand) kernel attributes: %s",
             cudaGetErrorString(e));
    cudaGetLastError();
    return MHAR_E_CUDA;
  }
  return MHAR_OK;
}

namespace {

cudaError_t launch_ts(mhar_ctx* c, int j, const SmallRun* r) {
  const TcPlan* plan = static_cast<const TcPlan*>(c->tc);
  const TsShape s = ts_shape(c, plan);
  TsParams p;
  p.rows = c->d.rows;
  p.wscale = c->d.wscale;
  p.Xh = c->d.Xh;
  p.Xl = c->d.Xl;
  p.lmin = c->d.lmin;
  p.lmax = c->d.lmax;
  p.theta = c->d.theta;
  p.status = c->d.status;
  p.counters = c->d.counters;
  p.err = c->d.status + 1;
  p.step_ptr = r ? nullptr : c->d.step;
  p.step_out = r ? c->d.step : nullptr;
  p.step0 = r ? r->step : 0;
  p.iters = r ? r->iters : 1;
  p.out = r ? r->out : nullptr;
  p.emit = r ? r->emit : 0;
  p.thin = r ? r->thin : 1;
  p.phase = r ? r->phase : 0;
  p.n = c->n;
  p.seed = c->opts.seed;
  p.j = j;
  p.walker0 = c->opts.walker0;
  p.z = c->z;
  p.z_ld = plan->strips * kWalkers;
  p.kdim = c->kdim;
  p.k_chunks = c->k_pad / kTcKChunk;
  p.k_pad = c->k_pad;
  p.tiles_per_cta = s.tiles_per_cta;
  p.m_tiles = s.m_tiles;
  p.wt = make_walker_tail(c, 1, true);
  const int share = (kWalkers + s.C - 1) / s.C, items = (c->n + 7) / 8 * share;
  p.resident = r && items <= kEpiThreads ? 1 : 0;
  // The draw warps take what they get done beside the tiles: about 100 cycles an
  // MMA (six per K step) and 9000 of the rest of an iteration, against 3400 cycles
  // a round of 64 items (1700 a round of low-rank normals) and 2600 more with
  // U g.  The epilogue warps draw the others, a quad at a time, between their last
  // tile and theta, a gap of about 2000 cycles.
  const bool pc = c->pc_rank >= 0;
  int cycles = s.tiles_per_cta * (p.kdim / kTcK) * 600 + 9000;
  if (pc) cycles -= (share * (kMaxPcRank / 4) + kDrawThreads - 1) / kDrawThreads * 1700;
  p.draw_chunks = std::min(items, std::max(0, cycles / (pc ? 6000 : 3400)) * kDrawThreads) / share;

  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(s.C, plan->strips, 1);
  cfg.blockDim = dim3(r ? kThreadsTs : kThreadsOne, 1, 1);
  cfg.dynamicSmemBytes = kSmemTs;
  cfg.stream = c->stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = s.C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  // Programmatic dependent launch: the grid may be scheduled while the
  // previous kernel finishes; it waits (griddepcontrol.wait) before reading.
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  const TsKernel k = kTsKernels[r ? 1 : 0][4 * (p.k_chunks - 1) + last_chunk_steps(p.kdim, p.k_chunks) - 1];
  return cudaLaunchKernelEx(&cfg, k, plan->ah64, plan->al64, p);
}

}  // namespace

cudaError_t launch_recompute_ts(mhar_ctx* c, int j) { return launch_ts(c, j, nullptr); }

cudaError_t launch_recompute_ts_run(mhar_ctx* c, const SmallRun& r) { return launch_ts(c, 0, &r); }

}  // namespace mhar
