// kernels_screen.cu -- the chord of the FP64 and FP32 modes (Section 4.4),
// screened on the tensor cores.
//
// A chord end is one ratio, min over g_i > 0 of s_i / g_i (max over g_i < 0),
// so only the rows that can hold it need the mode's own arithmetic.  FP64 runs
// at 1/64 of the FP32 rate on this GPU and the CUDA cores' FP32 far below the
// tensor pipe, so an iteration
//  (1) splits every walker's point and direction into FP16 pairs
//      (screen_split_kernel), each scaled by its own power of two;
//  (2) forms P = X A^T and G = D A^T on the tensor cores from the pairs (three
//      products each, FP32 accumulation, the pipelines of kernels_sk.cu) and,
//      row by row, a lower bound of the ratio the mode's arithmetic would give:
//        (b_i - p_i - K_i |x|) / (g_i + K_i |d|),
//      K_i the bound of kernels_simt.cu (prepare_tc_kernel) on |computed -
//      exact| of a_i . x and a_i . d, which covers the FP16 split of both
//      operands; in the FP32 mode twice that mode's own margin is added to it.
//      Each epilogue thread keeps, per chord side, the least bound of its rows
//      with the row's index in the five low bits, and the second least
//      (screen_kernel);
//  (3) evaluates the row of the least bound in the mode's own arithmetic -- the
//      products added in index order by one thread, the bits of
//      chord_simt_kernel -- and every other row whose bound does not exceed
//      the ratio found (screen_finish_kernel; when a stream's second bound does
//      not, the bounds of its rows are formed again in FP32 by the block), then
//      draws theta and moves the walker as update_kernel does.
// On a 2000 x 100 body with 4096 walkers an iteration's chord and move take 48 us in
// FP64 (4131 us with chord_simt_kernel<double>, 63 % of the FP64 pipe) and 36 in FP32
// (234 us), after a draw of 24 and 2.5 us: split 7.8 and 5.5, screen 15.8 (the MMAs of
// 12 m n z flops and their epilogue, as in the recompute kernels), finish 24.3 and 14.8
// (latency of the serial sums).
// So the chord ends, theta and the points have the bits of the direct
// kernels.  Rows that tie within the bounds (duplicate rows, walkers on a
// facet) cost more evaluations, never a different result.  Values the bounds
// do not cover (outside 2^-50 .. 2^50) take the direct formulas: a body at
// creation, a walker by its flag (`force`).  An iteration that takes longer than the direct
// kernels take sends its context to them for a while (screen_slow_clocks here, screen_look
// in mhar_api.cu).
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "mhar_device.cuh"
#include "mhar_internal.h"
#include "screen_row.cuh"
#include "tc_common.cuh"

namespace mhar {
namespace {

using namespace tc;

constexpr int kPairs = 2;                            // slots of A: hi + lo of one K chunk
constexpr int kWSlots = 2;                           // slots of the walker operands' K chunks
constexpr int kWBytes = 4 * kOperandBytes;           // Dh, Dl, Xh, Xl
constexpr int kABytes = 2 * kOperandBytes;           // A hi, A lo
constexpr int kEpiWarps = 16;
constexpr int kPWarp = 2 + kEpiWarps;
static_assert(kRowsTile == 128 && kEpiWarps == 16, "screen_row's tiles and streams");
constexpr int kThreadsScr = (3 + kEpiWarps) * 32;
constexpr unsigned int kNone = 0x7f800000u;          // a bound at or above +Inf: no row

__device__ __forceinline__ double neg_inf() { return -__longlong_as_double(0x7ff0000000000000ll); }
__device__ __forceinline__ double pos_inf() { return __longlong_as_double(0x7ff0000000000000ll); }

// Per-walker results of the split: the factors of the row bounds (WalkerNorms)
// and the exponent of the direction's scale (ratios of the screen are the
// walk's times 2^ed).
struct ScreenWalker {
  float nxw2, nd2, ws, ndinf;
};

// ---- (1) FP16 pairs of the points and directions ---------------------------
// One warp per walker.  FP32 mode: also the norms of its own margins, added in
// the order of chord_simt_kernel (16 columns, then a butterfly).
template <typename T>
__global__ void __launch_bounds__(128)
screen_split_kernel(int z, int n, int n_ld, int k_pad, const T* __restrict__ X,
                    const T* __restrict__ D, const float* __restrict__ sigma,
                    const float* __restrict__ corrn, __half* Xh, __half* Xl, __half* Dh,
                    __half* Dl, ScreenWalker* sw, float4* nrm32, int2* flags) {
  const int lane = threadIdx.x & 31;
  const int k = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (k >= z) return;
  const T* x = X + static_cast<size_t>(k) * n_ld;
  const T* d = D + static_cast<size_t>(k) * n_ld;
  // In FP32 from here on, FP64 entries rounded once (2^-24 of the 2^-21 that K
  // grants the split): FP64 scaling took 33 us where this takes 8 (z = 4096,
  // n = 100).
  float mx = 0.0f, md = 0.0f;
  bool nan = false;
  for (int i = lane; i < n; i += 32) {
    const float is = pow2_recip(sigma[i]);
    const float xs = fabsf(static_cast<float>(x[i]) * is), ds = fabsf(static_cast<float>(d[i]) * is);
    nan |= !(xs <= 0x1p50f) || !(ds <= 0x1p50f);
    mx = fmaxf(mx, xs);
    md = fmaxf(md, ds);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    md = fmaxf(md, __shfl_xor_sync(0xffffffffu, md, off));
  }
  const bool force = __any_sync(0xffffffffu, nan) || (mx > 0.0f && mx < 0x1p-50f) ||
                     (md > 0.0f && md < 0x1p-50f);
  int ex = 0, ed = 0;
  if (!force && mx > 0.0f) frexpf(mx, &ex);
  if (!force && md > 0.0f) frexpf(md, &ed);
  const float ix = ldexpf(1.0f, -ex), id = ldexpf(1.0f, -ed);
  float ssx = 0.0f, ssd = 0.0f;
  const size_t row = static_cast<size_t>(k) * k_pad;
  for (int i = 2 * lane; i < n; i += 64) {
    __half2 xh2, xl2, dh2, dl2;
    float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int e = 0; e < 2; ++e)
      if (i + e < n && !force) {
        const float is = pow2_recip(sigma[i + e]);
        v[e] = static_cast<float>(x[i + e]) * is * ix;
        v[2 + e] = static_cast<float>(d[i + e]) * is * id;
      }
    ssx = fmaf(v[0], v[0], fmaf(v[1], v[1], ssx));
    ssd = fmaf(v[2], v[2], fmaf(v[3], v[3], ssd));
    xh2 = __floats2half2_rn(v[0], v[1]);
    dh2 = __floats2half2_rn(v[2], v[3]);
    xl2 = __floats2half2_rn(v[0] - __low2float(xh2), v[1] - __high2float(xh2));
    dl2 = __floats2half2_rn(v[2] - __low2float(dh2), v[3] - __high2float(dh2));
    *reinterpret_cast<__half2*>(Xh + row + i) = xh2;
    *reinterpret_cast<__half2*>(Xl + row + i) = xl2;
    *reinterpret_cast<__half2*>(Dh + row + i) = dh2;
    *reinterpret_cast<__half2*>(Dl + row + i) = dl2;
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    ssx += __shfl_xor_sync(0xffffffffu, ssx, off);
    ssd += __shfl_xor_sync(0xffffffffu, ssd, off);
  }
  if (lane == 0) {
    ScreenWalker w;
    w.ws = ldexpf(1.0f, ex);
    w.nxw2 = w.ws * norm_bound(ssx);
    w.nd2 = norm_bound(ssd);
    w.ndinf = 1.0f;                 // max |d_hat| < 1
    if (corrn != nullptr) {
      // The FP32 margin of a_i . d with equalities, ||a_i sigma||_2 corrn:
      // K_i >= 2^-22 |a_hat_i|_p.
      const float cc = 4194304.0f * corrn[k] * ldexpf(1.0f, -ed);
      w.nd2 += cc;
      w.ndinf += cc;
    }
    sw[k] = w;
    flags[k] = make_int2(force ? 1 : 0, ed);
  }
  if constexpr (sizeof(T) == 4) {
    T sx = T(0), sd = T(0), mxx = T(0), mxd = T(0);
    for (int i = lane & 15; i < n_ld; i += 16) {
      const T isig = T(1) / static_cast<T>(sigma[i]);
      const T xs = x[i] * isig, ds = d[i] * isig;
      sx += xs * xs;
      sd += ds * ds;
      mxx = fmax(mxx, fabs(xs));
      mxd = fmax(mxd, fabs(ds));
    }
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) {
      sx += __shfl_xor_sync(0xffffffffu, sx, off);
      sd += __shfl_xor_sync(0xffffffffu, sd, off);
      mxx = fmax(mxx, __shfl_xor_sync(0xffffffffu, mxx, off));
      mxd = fmax(mxd, __shfl_xor_sync(0xffffffffu, mxd, off));
    }
    if (lane == 0)
      nrm32[k] = make_float4(sqrt(sx) * 1.0009765625f, sqrt(sd) * 1.0009765625f, mxx, mxd);
  }
}

// The row blocks of the screen (tc_common.cuh, row_block): b / s_r lowered,
// then K for the slack and again for a_i . d, in the 2-norm or max-norm form
// that is the tighter for the block's rows.  kr (FP32 mode, 3 per row): the
// direct kernel's margin K_2, K_1 is added twice -- its computed slack and
// a_i . d lie within one margin of the exact values and are then moved by one
// more -- and b lowered by the roundings of its own lowered b.
// One warp per block, a lane per row.  outside: set when a row's scale or b lies
// beyond the screen's range.
__global__ void screen_rows_kernel(int groups, int m, const float* bS, const float* rowk,
                                   const float* row_scale, const double* b64, const float* kr,
                                   float d2, float dinf, float* rows, int* outside) {
  const int g = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), t = threadIdx.x & 31;
  if (g >= groups) return;
  const int r = 32 * g + t;
  float s2 = rowk[4 * r], s1 = rowk[4 * r + 2];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    s2 += __shfl_xor_sync(0xffffffffu, s2, off);
    s1 += __shfl_xor_sync(0xffffffffu, s1, off);
  }
  const int inf = s1 * dinf < s2 * d2 ? 1 : 0;
  float kk = rowk[4 * r + (inf ? 2 : 0)];
  float bl = bS[r];
  if (r < m) {
    // max |a_i sigma| = f row_scale, f in [0.5, 1); 1 for a zero row.
    const float sc = row_scale[r];
    if (!(sc <= 0x1p50f && sc >= 0x1p-49f && fabs(b64[r]) <= 0x1p50)) atomicOr(outside, 1);
    if (kr != nullptr) {
      kk += 2.0f * kr[3 * r + (inf ? 1 : 0)] / sc;
      kk *= 1.0f + 0x1p-20f;
      bl -= 0x1p-20f * fabsf(bl);
    }
  }
  float* blk = rows + static_cast<size_t>(g) * 128;
  blk[t] = bl;
  blk[32 + t] = kk;
  blk[64 + t] = kk;
  blk[96 + t] = inf ? 1.0f : 0.0f;
}

// ---- (2) the screen ----------------------------------------------------------
struct ScrParams {
  const float* rows;
  const ScreenWalker* sw;
  uint4* res;               // [stream][z_ld]: least and second bound, lambda_max then lambda_min
  unsigned int* tiles;      // [stream][z_ld]: row tile of the least bounds (lambda_max | lambda_min << 16)
  int* err;
  int z, z_ld, k_chunks, tiles_per_cta, m_tiles;
};

struct ScrTail {
  uint64_t w_full[kWSlots];
  uint64_t w_empty[kWSlots];
  uint64_t a_full[kPairs];
  uint64_t a_empty[kPairs];
  uint64_t t_full[2];
  uint64_t t_empty[2];
  uint32_t tmem_base;
  int timed_out;
};

constexpr size_t kSmemScr = 1024 + static_cast<size_t>(kWSlots) * kWBytes +
                            static_cast<size_t>(kPairs) * kABytes + sizeof(ScrTail);
static_assert(kSmemScr <= 232448, "screen_kernel exceeds the shared memory of a CTA");

__device__ __forceinline__ void mbar_arrive_scr(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ float rcp_approx(float v) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}

// The least two of the keys seen so far.
__device__ __forceinline__ void two_least(unsigned int r, unsigned int& m1, unsigned int& m2) {
  m2 = min(m2, max(m1, r));
  m1 = min(m1, r);
}

// Bounds of 32 rows on both sides.  s: the lowered slacks (>= +0).  A row
// counts on a side when its a_i . d may lie on it: the denominator, a_i . d
// moved by its bound towards that side, is then positive; otherwise the
// quotient's sign bit (or a NaN from 0 / 0, the padding rows) ranks it above
// +Inf as an unsigned key.
__device__ __forceinline__ void bound32(const float (&s)[32], const float (&g)[32],
                                        const float* rows, int row0, float nd, unsigned int& h1,
                                        unsigned int& h2, unsigned int& l1, unsigned int& l2) {
  const float4* k4 = reinterpret_cast<const float4*>(row_block(rows, row0)) + 16;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float4 kk = __ldg(k4 + i);
    const float kg[4] = {kk.x, kk.y, kk.z, kk.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int r = 4 * i + j;
      const unsigned int uh = __float_as_uint(s[r] * rcp_approx(fmaf(kg[j], nd, g[r])));
      const unsigned int ul = __float_as_uint(s[r] * rcp_approx(fmaf(kg[j], nd, -g[r])));
      two_least((uh & ~31u) | r, h1, h2);
      two_least((ul & ~31u) | r, l1, l2);
    }
  }
}

// Grid (splits of the row tiles, walker strips).  The operands of a body with
// at most two K chunks stay in shared memory for the CTA's whole row range;
// wider bodies stream them per tile.  Two threads issue the MMAs (G and P).
__global__ void __launch_bounds__(kThreadsScr, 1)
screen_kernel(const __grid_constant__ CUtensorMap tm_ah, const __grid_constant__ CUtensorMap tm_al,
              const __grid_constant__ CUtensorMap tm_dh, const __grid_constant__ CUtensorMap tm_dl,
              const __grid_constant__ CUtensorMap tm_xh, const __grid_constant__ CUtensorMap tm_xl,
              const ScrParams p, int last) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t* wslot = base;
  uint8_t* aslot = base + kWSlots * kWBytes;
  ScrTail* tail = reinterpret_cast<ScrTail*>(aslot + kPairs * kABytes);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int strip = blockIdx.y;
  const int t0 = blockIdx.x * p.tiles_per_cta;
  const int t1 = min(p.m_tiles, t0 + p.tiles_per_cta);
  const bool resident = p.k_chunks <= kWSlots;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kWSlots; ++s) { mbar_init(&tail->w_full[s], 1); mbar_init(&tail->w_empty[s], 2); }
    for (int s = 0; s < kPairs; ++s) { mbar_init(&tail->a_full[s], 1); mbar_init(&tail->a_empty[s], 2); }
    for (int b = 0; b < 2; ++b) { mbar_init(&tail->t_full[b], 2); mbar_init(&tail->t_empty[b], kEpiWarps); }
    tail->timed_out = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    prefetch_tmap(&tm_ah);
    prefetch_tmap(&tm_al);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tail->tmem_base)), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tail->tmem_base;
  volatile int* timed_out = &tail->timed_out;
  // A programmatic dependent of the split kernel: nothing it wrote is read
  // before this.
  asm volatile("griddepcontrol.wait;" ::: "memory");

  if (warp == 0) {
    if (lane == 0) {
      int it = 0;
      const int yw = strip * kWalkers;
      for (int nt = t0; nt < t1; ++nt) {
        for (int kc = 0; kc < p.k_chunks; ++kc, ++it) {
          const int x = kc * kTcKChunk;
          const int ws = resident ? kc : it % kWSlots;
          if (!resident || nt == t0) {
            if (!resident && it >= kWSlots)
              mbar_wait(&tail->w_empty[ws], ((it / kWSlots) - 1) & 1, timed_out, p.err);
            uint8_t* dst = wslot + ws * kWBytes;
            mbar_expect_tx(&tail->w_full[ws], kWBytes);
            tma_load_2d(dst, &tm_dh, &tail->w_full[ws], x, yw);
            tma_load_2d(dst + kOperandBytes, &tm_dl, &tail->w_full[ws], x, yw);
            tma_load_2d(dst + 2 * kOperandBytes, &tm_xh, &tail->w_full[ws], x, yw);
            tma_load_2d(dst + 3 * kOperandBytes, &tm_xl, &tail->w_full[ws], x, yw);
          }
          const int as = it % kPairs;
          if (it >= kPairs) mbar_wait(&tail->a_empty[as], ((it / kPairs) - 1) & 1, timed_out, p.err);
          mbar_expect_tx(&tail->a_full[as], kABytes);
          tma_load_2d(aslot + as * kABytes, &tm_ah, &tail->a_full[as], x, nt * kRowsTile);
          tma_load_2d(aslot + as * kABytes + kOperandBytes, &tm_al, &tail->a_full[as], x,
                      nt * kRowsTile);
        }
      }
    }
    __syncwarp();
  } else if (warp == 1 || warp == kPWarp) {
    if (lane == 0) {
      constexpr uint32_t idesc = make_idesc(kWalkers, kRowsTile);
      const bool g_side = warp == 1;
      const uint32_t op0 = g_side ? 0u : 2u * kOperandBytes;
      int it = 0;
      for (int nt = t0; nt < t1; ++nt) {
        const int gt = nt - t0, b = gt & 1;
        if (gt >= 2) mbar_wait(&tail->t_empty[b], ((gt >> 1) - 1) & 1, timed_out, p.err);
        tc_fence_after();
        const uint32_t d_tmem = tmem + static_cast<uint32_t>(b * 256) + (g_side ? 0u : 128u);
        for (int kc = 0; kc < p.k_chunks; ++kc, ++it) {
          const int ws = resident ? kc : it % kWSlots;
          const int as = it % kPairs;
          if (!resident) mbar_wait(&tail->w_full[ws], (it / kWSlots) & 1, timed_out, p.err);
          else if (gt == 0) mbar_wait(&tail->w_full[ws], 0, timed_out, p.err);
          mbar_wait(&tail->a_full[as], (it / kPairs) & 1, timed_out, p.err);
          tc_fence_after();
          const uint32_t w0 = smem_u32(wslot + ws * kWBytes) + op0;
          const uint64_t o_h = sw128_desc(w0), o_l = sw128_desc(w0 + kOperandBytes);
          const uint64_t a_h = sw128_desc(smem_u32(aslot + as * kABytes));
          const uint64_t a_l = sw128_desc(smem_u32(aslot + as * kABytes + kOperandBytes));
          const int ks = kc + 1 < p.k_chunks ? 4 : last;
          ss_run2_n(ks, d_tmem, o_h, o_l, a_h, idesc, kc > 0 ? 1u : 0u);
          ss_run1_n(ks, d_tmem, o_h, a_l, idesc);
          mma_commit(&tail->a_empty[as]);
          if (!resident) mma_commit(&tail->w_empty[ws]);
        }
        mma_commit(&tail->t_full[b]);
      }
    }
    __syncwarp();
  } else {
    const int q = warp & 3, cg = (warp - 2) >> 2;
    const int k = strip * kWalkers + q * 32 + lane;
    WalkerNorms wn;
    wn.nxw2 = wn.nd2 = wn.ndinf = 0.0f;
    wn.ws = 1.0f;
    if (k < p.z) {
      const float4 w = __ldg(reinterpret_cast<const float4*>(p.sw) + k);
      wn.nxw2 = w.x; wn.nd2 = w.y; wn.ws = w.z; wn.ndinf = w.w;
    }
    unsigned int h1 = ~0u, h2 = ~0u, l1 = ~0u, l2 = ~0u;
    unsigned int th = 0u, tl = 0u;
    const uint32_t lane_off = static_cast<uint32_t>(q * 32) << 16;
    for (int nt = t0; nt < t1; ++nt) {
      const int gt = nt - t0, b = gt & 1;
      const int row0 = nt * kRowsTile + cg * 32;
      if (lane < 4) prefetch_l1(row_block(p.rows, row0) + 32 * lane);
      mbar_wait(&tail->t_full[b], (gt >> 1) & 1, timed_out, p.err, true);
      tc_fence_after();
      const uint32_t gcol = tmem + lane_off + static_cast<uint32_t>(b * 256 + cg * 32);
      float sv[32], gv[32];
      tmem_ld32(gcol + 128u, sv);
      tmem_ld32(gcol, gv);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_scr(&tail->t_empty[b]);
      float fx, fd;
      wn.pick(p.rows, row0, fx, fd);
      slack32(sv, p.rows, row0, wn.ws, fx);
      const unsigned int ph = h1, pl = l1;
      // The tile's least two merge into the running pair as they come: the
      // row index stays in the key, the tile index beside it.
      bound32(sv, gv, p.rows, row0, fd, h1, h2, l1, l2);
      if (h1 != ph) th = static_cast<unsigned int>(nt);
      if (l1 != pl) tl = static_cast<unsigned int>(nt);
    }
    if (k < p.z) {
      const size_t o = static_cast<size_t>(blockIdx.x * 4 + cg) * p.z_ld + k;
      p.res[o] = make_uint4(h1, h2, l1, l2);
      p.tiles[o] = th | (tl << 16);
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u)
                 : "memory");
  }
}

// ---- (3) the rows that can hold a chord end, theta, the move -----------------
template <typename T>
struct FinParams {
  const T* A;
  const T* b;
  const T* kr;              // FP32: 3 per row; FP64: null
  const T* X;               // what the chord reads: X64, or Xhi
  const T* D;
  const float* corrn;
  const float4* nrm32;
  const uint4* res;
  const unsigned int* tiles;
  const int2* flags;
  const float* rows;        // the screen's row blocks, operands and walker factors
  const __half* Ah;
  const __half* Al;
  const __half* Xh;
  const __half* Xl;
  const __half* Dh;
  const __half* Dl;
  const ScreenWalker* sw;
  uint64_t seed;
  const uint64_t* step_ptr;
  int j;
  uint32_t walker0;
  int m, n, n_ld, k_pad, z, z_ld, streams, tiles_per_cta, m_tiles, mE;
  double* lmin;
  double* lmax;
  double* theta;
  int* status;
  unsigned long long* slow;  // screen_slow
  unsigned int slow_clocks;  // of a block: more, and the direct kernels take less time
  unsigned long long* counters;
  double* X64;
  float* Xhi;
  float* Xlo;
  const float* Q32;
  const float* corr;
};

// a . v in index order (the padding beyond n is zero), one thread's serial sum.
template <typename T>
__device__ __forceinline__ T dot_in_order(const T* __restrict__ a, const T* v, int n_ld) {
  constexpr int V = 16 / sizeof(T);
  T acc = T(0);
#pragma unroll 4
  for (int i = 0; i < n_ld; i += V) {
    alignas(16) T av[V];
    alignas(16) T xv[V];
    *reinterpret_cast<float4*>(av) = __ldg(reinterpret_cast<const float4*>(a + i));
    *reinterpret_cast<float4*>(xv) = *reinterpret_cast<const float4*>(v + i);
#pragma unroll
    for (int u = 0; u < V; ++u) acc += av[u] * xv[u];
  }
  return acc;
}

// The same for a warp's 32 sums at once (eight walkers x two sides' rows x (a . x,
// a . d)): the 16 rows, 8 points and 8 directions come into shared memory 128
// bytes of each at a time, whole lines, kFinStages steps ahead.  Read by the threads
// themselves each 16 bytes took a line of its own (136 clocks a term in FP64, 59 in
// FP32); with this and the move's loads in batches an iteration of a call on the 2000 x
// 100 body, draw and the call's own launches included, takes 41 us in FP32 (44.5 before)
// and 85.6 in FP64 (87.9, bound by the FP64 chain).
constexpr int kFinStages = 4;
constexpr int kFinRow = 144;                       // bytes between two staged pieces
constexpr int kFinDir = 24 * kFinRow + 64;         // the directions, off the points' banks
constexpr int kFinBuf = kFinDir + 8 * kFinRow;     // one step of a warp

template <typename T>
__device__ __forceinline__ T warp_dots(const T* __restrict__ A, const T* X, const T* D, int row,
                                       int k, int n_ld, uint8_t* buf) {
  constexpr int V = 16 / sizeof(T);
  const int lane = threadIdx.x & 31, piece = lane & 7;
  const int steps = n_ld * static_cast<int>(sizeof(T)) / 128;
  // Eight copies a step: lanes 8 q .. 8 q + 7 take vector 4 j + q.
  const uint8_t* src[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int v = 4 * j + (lane >> 3);
    const int who = j < 4 ? __shfl_sync(0xffffffffu, row, (2 * v) & 31)
                          : __shfl_sync(0xffffffffu, k, (4 * (v & 7)) & 31);
    const T* from = j < 4 ? A : j < 6 ? X : D;
    src[j] = reinterpret_cast<const uint8_t*>(from + static_cast<size_t>(who) * n_ld) + 16 * piece;
  }
  auto issue = [&](int st) {
    if (st < steps) {
      const uint32_t to = smem_u32(buf + (st % kFinStages) * kFinBuf) + 16 * piece;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int v = 4 * j + (lane >> 3);
        const uint32_t dst = to + static_cast<uint32_t>(v * kFinRow + (j >= 6 ? 64 : 0));
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src[j] + 128 * st)
                     : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  for (int st = 0; st < kFinStages - 1; ++st) issue(st);
  const int mine = (lane >> 1) * kFinRow;
  const int other = (lane & 1 ? kFinDir : 16 * kFinRow) + (lane >> 2) * kFinRow;
  T acc = T(0);
  for (int st = 0; st < steps; ++st) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kFinStages - 2) : "memory");
    __syncwarp();
    const uint8_t* at = buf + (st % kFinStages) * kFinBuf;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      alignas(16) T av[V];
      alignas(16) T xv[V];
      *reinterpret_cast<float4*>(av) = *reinterpret_cast<const float4*>(at + mine + 16 * u);
      *reinterpret_cast<float4*>(xv) = *reinterpret_cast<const float4*>(at + other + 16 * u);
#pragma unroll
      for (int e = 0; e < V; ++e) acc += av[e] * xv[e];
    }
    __syncwarp();
    issue(st + kFinStages - 1);      // over the step before, read by every lane
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncwarp();
  return acc;
}

// The slack and a_i . d of chord_simt_kernel from the two products.
template <typename T>
__device__ __forceinline__ bool row_terms(const FinParams<T>& p, int k, int row, T ax, T ad, T& s,
                                          T& g) {
  s = p.b[row] - ax;
  g = ad;
  if (p.kr != nullptr) {
    const float4 w = p.nrm32[k];
    const T k2 = p.kr[3 * row], k1 = p.kr[3 * row + 1];
    s -= fmin(k2 * static_cast<T>(w.x), k1 * static_cast<T>(w.z));
    T eg = fmin(k2 * static_cast<T>(w.y), k1 * static_cast<T>(w.w));
    if (p.corrn != nullptr) eg += p.kr[3 * row + 2] * static_cast<T>(p.corrn[k]);
    g = g > T(0) ? g + eg : (g < T(0) ? g - eg : g);
  }
  if (!isfinite(s) || !isfinite(g)) return false;
  if (s < T(0)) s = T(0);
  return true;
}

// Largest key of a bound that may still beat the ratio `lam` (>= 0; +Inf: none
// found yet) of a walker whose screen ratios are scaled by 2^ed.
__device__ __forceinline__ unsigned int key_limit(double lam, int ed) {
  if (lam == 0.0) return 0u;                      // nothing lies below 0
  const float f = static_cast<float>(scalbn(lam, ed)) * (1.0f + 0x1p-18f);
  return f < INFINITY ? (__float_as_uint(f) | 31u) : kNone - 1u;
}

constexpr int kFinThreads = 128;
constexpr int kFinWalkers = kFinThreads / 4;
constexpr size_t kFinSmem = static_cast<size_t>(kFinThreads / 32) * kFinStages * kFinBuf;
constexpr int kFinList = 256;     // streams that a block looks at again in one round

// Eight consecutive values hi + lo of an FP16 pair.
__device__ __forceinline__ void pair8(const __half* hi, const __half* lo, float (&v)[8]) {
  const uint4 h = __ldg(reinterpret_cast<const uint4*>(hi)), l = __ldg(reinterpret_cast<const uint4*>(lo));
  const uint32_t hw[4] = {h.x, h.y, h.z, h.w}, lw[4] = {l.x, l.y, l.z, l.w};
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&hw[e]));
    const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&lw[e]));
    v[2 * e] = a.x + b.x;
    v[2 * e + 1] = a.y + b.y;
  }
}

// Whether one row of walker k may hold a chord end on a side below the limit
// `lim` (key_limit): the screen's bound, formed again in FP32 from the same
// operands.  Four sums of a quarter of the products each stay inside the K's share for
// the accumulation, (T + 1) 2^-22 with T = 3 MMAs a step of 16 columns.
template <typename T>
__device__ __forceinline__ bool may_hold(const FinParams<T>& p, int k, int row, bool side,
                                         unsigned int lim) {
  const size_t ar = static_cast<size_t>(row) * p.k_pad, wr = static_cast<size_t>(k) * p.k_pad;
  float ps[4] = {}, gs[4] = {};
#pragma unroll 2
  for (int i = 0; i < p.n; i += 8) {
    float a[8], x[8], d[8];
    pair8(p.Ah + ar + i, p.Al + ar + i, a);
    pair8(p.Xh + wr + i, p.Xl + wr + i, x);
    pair8(p.Dh + wr + i, p.Dl + wr + i, d);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      ps[e & 3] = fmaf(a[e], x[e], ps[e & 3]);
      gs[e & 3] = fmaf(a[e], d[e], gs[e & 3]);
    }
  }
  const float P = (ps[0] + ps[1]) + (ps[2] + ps[3]), g = (gs[0] + gs[1]) + (gs[2] + gs[3]);
  const float* blk = row_block(p.rows, row & ~31);
  const int r = row & 31;
  const ScreenWalker w = p.sw[k];
  const bool inf = blk[96] != 0.0f;
  const float kk = blk[32 + r] * (1.0f + 0x1p-20f);
  const float sl = fmaf(-kk, inf ? w.ws : w.nxw2, fmaf(-P, w.ws, blk[r]));
  const float den = fmaf(kk, inf ? w.ndinf : w.nd2, side ? -g : g);
  if (!(den > 0.0f)) return false;
  const float q = fmaxf(sl, 0.0f) / den * (1.0f - 0x1p-18f);
  return __float_as_uint(q) <= lim;
}

// a . x and a . d of one row by one thread, each in index order.
template <typename T>
__device__ __forceinline__ void dots_in_order(const T* __restrict__ a, const T* x, const T* d,
                                              int n_ld, T& ax, T& ad) {
  constexpr int V = 16 / sizeof(T);
  ax = ad = T(0);
#pragma unroll 4
  for (int i = 0; i < n_ld; i += V) {
    alignas(16) T av[V];
    alignas(16) T xv[V];
    alignas(16) T dv[V];
    *reinterpret_cast<float4*>(av) = __ldg(reinterpret_cast<const float4*>(a + i));
    *reinterpret_cast<float4*>(xv) = *reinterpret_cast<const float4*>(x + i);
    *reinterpret_cast<float4*>(dv) = *reinterpret_cast<const float4*>(d + i);
#pragma unroll
    for (int u = 0; u < V; ++u) {
      ax += av[u] * xv[u];
      ad += av[u] * dv[u];
    }
  }
}

// Four threads per walker: (lambda_max, lambda_min) x (a . x, a . d).
template <typename T>
__global__ void __launch_bounds__(kFinThreads)
screen_finish_kernel(const FinParams<T> p) {
  __shared__ double theta_s[kFinWalkers];
  __shared__ unsigned long long again_s[2 * kFinWalkers];   // least ratio found in a list's rows
  __shared__ unsigned int limit_s[2 * kFinWalkers];
  __shared__ int list[kFinList];
  __shared__ int listed;
  extern __shared__ __align__(16) uint8_t fin_smem[];       // kFinStages steps a warp
  __shared__ unsigned int started;
  if (threadIdx.x == 0) started = static_cast<unsigned int>(clock());
  const int lane = threadIdx.x & 31;
  const int wl = threadIdx.x >> 2, t4 = threadIdx.x & 3;
  const int side = t4 >> 1, which = t4 & 1;
  const int k0 = blockIdx.x * kFinWalkers;
  const int k = k0 + wl;
  const bool live = k < p.z;
  const int kc = live ? k : p.z - 1;
  const int2 fl = p.flags[kc];
  const bool force = live && fl.x != 0;
  const bool go = live && !force;

  // Rows in the order of their bounds while they may lower the ratio found
  // (the two threads of a side share its streams and its two products): the
  // least bound of each stream and its row.
  double lam = pos_inf();          // |ratio| of this side
  bool bad = false;
  unsigned int last = 0u;          // the last (bound, stream) taken
  int last_st = -1;
  for (;;) {
    const unsigned int lim = key_limit(lam, fl.y);
    unsigned int b1 = ~0u;
    int bst = 0;
    if (go && lim != 0u)
      for (int st = which; st < p.streams; st += 2) {
        const uint4 v = p.res[static_cast<size_t>(st) * p.z_ld + kc];
        const unsigned int m1 = side ? v.z : v.x;
        if (m1 < b1 && (m1 > last || (m1 == last && st > last_st))) { b1 = m1; bst = st; }
      }
    const unsigned int o1 = __shfl_xor_sync(0xffffffffu, b1, 1);
    const int ost = __shfl_xor_sync(0xffffffffu, bst, 1);
    if (o1 < b1 || (o1 == b1 && ost < bst)) { b1 = o1; bst = ost; }
    const bool has = b1 <= lim && b1 < kNone;
    if (!__any_sync(0xffffffffu, has)) break;
    int row = 0;
    if (has) {
      row = screen_row(p.tiles[static_cast<size_t>(bst) * p.z_ld + kc], side != 0, bst, b1, p.m);
      last = b1;
      last_st = bst;
    }
    const T acc = warp_dots(p.A, p.X, p.D, row, kc, p.n_ld,
                            fin_smem + (threadIdx.x >> 5) * kFinStages * kFinBuf);
    const T oth = __shfl_xor_sync(0xffffffffu, acc, 1);
    if (has) {
      T s, g;
      if (!row_terms(p, kc, row, which ? oth : acc, which ? acc : oth, s, g))
        bad = true;
      else if (side ? g < T(0) : g > T(0))
        lam = fmin(lam, fabs(static_cast<double>(s / g)));
    }
  }
  // A stream whose second bound may lower it too: the bounds of all its rows
  // again, by the block, and the mode's arithmetic for those that may.  (All its
  // rows in that arithmetic by one warp held half of the FP64 iterations of a
  // 2000 x 100 body with 4096 walkers 60 us, every FP32 one 20.)
  int next = which;                          // this thread's next stream
  if (which == 0) {
    again_s[threadIdx.x >> 1] = 0x7ff0000000000000ull;
    limit_s[threadIdx.x >> 1] = key_limit(lam, fl.y);
  }
  for (;;) {
    if (threadIdx.x == 0) listed = 0;
    __syncthreads();
    const unsigned int lim = go ? limit_s[threadIdx.x >> 1] : 0u;
    if (lim == 0u) next = p.streams;
    for (; next < p.streams; next += 2) {
      const uint4 v = p.res[static_cast<size_t>(next) * p.z_ld + kc];
      if ((side ? v.w : v.y) > lim) continue;
      const int at = atomicAdd(&listed, 1);
      if (at >= kFinList) break;             // the next round's first
      list[at] = (next << 6) | (wl << 1) | side;
    }
    __syncthreads();
    const int count = min(listed, kFinList);
    for (int e = 0; e < count; ++e) {
      const int st = list[e] >> 6, ws = list[e] & 63;
      const int wk = k0 + (ws >> 1);
      const bool wside = ws & 1;
      const int ta = (st >> 2) * p.tiles_per_cta, tb = min(p.m_tiles, ta + p.tiles_per_cta);
      for (int nt = ta + (threadIdx.x >> 5); nt < tb; nt += kFinThreads / 32) {
        const int row = nt * kRowsTile + (st & 3) * 32 + lane;
        if (row >= p.m || !may_hold(p, wk, row, wside, limit_s[ws])) continue;
        T ax, ad, s, g;
        dots_in_order(p.A + static_cast<size_t>(row) * p.n_ld, p.X + static_cast<size_t>(wk) * p.n_ld,
                      p.D + static_cast<size_t>(wk) * p.n_ld, p.n_ld, ax, ad);
        if (!row_terms(p, wk, row, ax, ad, s, g))
          bad = true;
        else if (wside ? g < T(0) : g > T(0))
          atomicMin(&again_s[ws], static_cast<unsigned long long>(
                                      __double_as_longlong(fabs(static_cast<double>(s / g)))));
      }
    }
    if (!__syncthreads_or(next < p.streams)) break;
  }
  lam = fmin(lam, __longlong_as_double(static_cast<long long>(again_s[threadIdx.x >> 1])));
  // Walkers outside the screen's range: every row, one walker after the other.
  unsigned int forced = __ballot_sync(0xffffffffu, force && t4 == 0);
  while (forced) {
    const int src = __ffs(forced) - 1;
    forced &= forced - 1;
    const int wk = __shfl_sync(0xffffffffu, kc, src);
    const T* xk = p.X + static_cast<size_t>(wk) * p.n_ld;
    const T* dk = p.D + static_cast<size_t>(wk) * p.n_ld;
    double hi = pos_inf(), lo = pos_inf();
    for (int row = lane; row < p.m; row += 32) {
      const T* a = p.A + static_cast<size_t>(row) * p.n_ld;
      T s, g;
      if (!row_terms(p, wk, row, dot_in_order(a, xk, p.n_ld), dot_in_order(a, dk, p.n_ld), s, g)) {
        bad = true;
        continue;
      }
      if (g > T(0)) hi = fmin(hi, static_cast<double>(s / g));
      else if (g < T(0)) lo = fmin(lo, fabs(static_cast<double>(s / g)));
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      hi = fmin(hi, __shfl_xor_sync(0xffffffffu, hi, off));
      lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, off));
    }
    if ((lane & ~3) == src) lam = side ? lo : hi;
  }
  if (bad) atomicOr(p.status, MHAR_ST_NONFINITE);

  // Section 4.5 (the arithmetic of update_kernel).
  const double other = __shfl_xor_sync(0xffffffffu, lam, 2);
  if (t4 == 0) {
    double t = 0.0;
    if (live) {
      const double L = -other, H = lam;
      if (isinf(L) || isinf(H)) {
        atomicOr(p.status, MHAR_ST_UNBOUNDED);
        atomicAdd(&p.counters[1], 1ull);
      } else if (L > H) {
        atomicOr(p.status, MHAR_ST_STALL);
        atomicAdd(&p.counters[0], 1ull);
      } else {
        const uint64_t step = *p.step_ptr + static_cast<uint64_t>(p.j);
        const U4 w = philox_block(p.seed, step, p.walker0 + static_cast<uint32_t>(k), 0u,
                                  kStreamChord);
        const double u = open_unit_f64(w.x);
        t = L + u * (H - L);
        if (sizeof(T) != 8) t = static_cast<double>(static_cast<float>(t));
      }
      p.lmin[k] = L;
      p.lmax[k] = H;
      p.theta[k] = t;
    }
    theta_s[wl] = t;
  }
  __syncthreads();
  // A warp along the rows of every fourth walker of the block, the loads of four of
  // them before the first store (one after the other: 4 us of an FP64 iteration).
  // Padding: x and d are 0 there, and stay so.
  constexpr int V = 16 / sizeof(T), kWarps = kFinThreads / 32, kBatch = 4;
  for (int i = lane * V; i < p.n_ld; i += 32 * V) {
#pragma unroll 1
    for (int w0 = threadIdx.x >> 5; w0 < kFinWalkers; w0 += kBatch * kWarps) {
      float4 x4[kBatch], l4[kBatch], d4[kBatch];
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
        const int kk = min(k0 + w0 + q * kWarps, p.z - 1);
        const size_t o = static_cast<size_t>(kk) * p.n_ld + i;
        d4[q] = *reinterpret_cast<const float4*>(p.D + o);
        if constexpr (sizeof(T) == 8) {
          x4[q] = *reinterpret_cast<const float4*>(p.X64 + o);
        } else {
          x4[q] = *reinterpret_cast<const float4*>(p.Xhi + o);
          l4[q] = *reinterpret_cast<const float4*>(p.Xlo + o);
        }
      }
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
        const int w = w0 + q * kWarps, kk = k0 + w;
        if (kk >= p.z) break;
        const size_t o = static_cast<size_t>(kk) * p.n_ld + i;
        const double t = theta_s[w];
        if constexpr (sizeof(T) == 8) {
          double2 x = *reinterpret_cast<const double2*>(&x4[q]);
          const double2 d = *reinterpret_cast<const double2*>(&d4[q]);
          x.x += t * d.x;
          x.y += t * d.y;
          *reinterpret_cast<double2*>(p.X64 + o) = x;
        } else {
          const float tf = static_cast<float>(t);
          const float d[4] = {d4[q].x, d4[q].y, d4[q].z, d4[q].w};
          float h[4] = {x4[q].x, x4[q].y, x4[q].z, x4[q].w}, l[4] = {l4[q].x, l4[q].y, l4[q].z, l4[q].w};
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            df_axpy(h[u], l[u], tf, d[u]);
            if (p.corr != nullptr && tf != 0.0f) {
              const int c = i + u;
              float dlt = 0.0f;
              if (c < p.n)
                for (int e = 0; e < p.mE; ++e)
                  dlt = fmaf(p.Q32[static_cast<size_t>(e) * p.n_ld + c],
                             p.corr[static_cast<size_t>(kk) * p.mE + e], dlt);
              l[u] = fmaf(-tf, dlt, l[u]);
            }
          }
          *reinterpret_cast<float4*>(p.Xhi + o) = make_float4(h[0], h[1], h[2], h[3]);
          *reinterpret_cast<float4*>(p.Xlo + o) = make_float4(l[0], l[1], l[2], l[3]);
        }
      }
    }
  }
  if (threadIdx.x == 0 && static_cast<unsigned int>(clock()) - started > p.slow_clocks)
    atomicMax(p.slow, static_cast<unsigned long long>(*p.step_ptr + static_cast<uint64_t>(p.j) + 1ull));
}

// CTAs along the rows: up to what the SMs leave for each walker strip, the number with
// the least time estimated from a CTA's tiles (2700 clocks for the epilogue, no less than
// six MMAs of 85 a K step) and 850 clocks for each four streams more that the finish goes
// through.  As many as there are SMs, with few walkers, was slower than the direct FP32
// kernel: an iteration of 65 walkers of an 8000 x 64 body 72 us with 63 CTAs along the
// rows, 35 with 16 (21: 35, 8: 39; direct 26); of 300 of a 4000 x 64 body 39 and 31 (39).
int screen_tiles_per_cta(const mhar_ctx* c) {
  int sms = 148;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
  const int strips = (c->z + kWalkers - 1) / kWalkers, tiles = c->m_pad / kRowsTile;
  const int most = std::max(1, std::min(sms / strips, tiles));
  const long long tile = std::max(2700, 6 * 85 * (c->kdim / kTcK));
  int per = tiles;
  long long best = 0;
  for (int C = 1; C <= most; ++C) {
    const int t = (tiles + C - 1) / C;
    const long long est = t * tile + 850ll * C;
    if (best == 0 || est < best) { best = est; per = t; }
  }
  return per;
}

// The direct kernels' time, in clocks of a block of the finish: one that takes longer makes
// the iteration slower than they are.  Walkers outside the screen's range do, one after
// the other (an FP64 iteration of 4096 walkers of a 2000 x 100 body with 1, 2, 3, 4 of a
// warp's eight outside 1180, 2290, 3400, 4510 us, direct 4160; FP32 with one 535, 239), and
// bodies of very many rows that tie within the bounds: 4000 rows in one dimension, 3000
// walkers, FP32 4495 us (direct 129), 8800 rows about a circle, 300 walkers, 267 (40).
// Tiles of 64 rows x 64 walkers: in FP64 31 + 2.16 n_ld us a tile and SM, two tiles at
// least (203 us at 160 tiles, n_ld = 32, 2673 at 4032; 601 and 7984 at n_ld = 128), in
// FP32 2.6 + 0.116 n_ld and 6 (20, 173; 42, 446).  A warp a walker: 0.125 us for a column
// of 32 rows (570 us for 100 x 1500, 50 for 64 x 128).
unsigned int screen_slow_clocks(const mhar_ctx* c) {
  int sms = 148;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
  double us;
  if (simt_warp_path(c)) {
    us = 8.0 + 0.125 * c->n * ((c->m + 31) / 32) * std::max(1.0, c->z / 600.0);
  } else {
    const double tiles = static_cast<double>((c->m + 63) / 64) * ((c->z + 63) / 64) / sms;
    us = c->opts.precision == MHAR_FP64
             ? (31.0 + 2.16 * c->n_ld) * std::max(2.0, tiles)
             : (2.6 + 0.116 * c->n_ld) * std::max(2.0, tiles) + 6.0;
  }
  const int blocks = (c->z + kFinWalkers - 1) / kFinWalkers;
  const int waves = (blocks + 3 * sms - 1) / (3 * sms);      // three blocks on an SM
  return static_cast<unsigned int>(std::min(us * 1900.0 / waves, 4.0e9));
}

template <typename T>
cudaError_t launch_screen_t(mhar_ctx* c, int j, const T* A, const T* b, const T* kr, const T* X,
                            const T* D) {
  const TcPlan* plan = static_cast<const TcPlan*>(c->tc);
  mhar::DeviceBuffers& d = c->d;
  const int z_ld = plan->strips * kWalkers;
  auto* sw = reinterpret_cast<ScreenWalker*>(d.scr_walker);
  auto* nrm = reinterpret_cast<float4*>(d.scr_nrm);
  auto* flags = reinterpret_cast<int2*>(d.scr_flags);
  auto* res = reinterpret_cast<uint4*>(d.scr_res);
  screen_split_kernel<T><<<(c->z + 3) / 4, 128, 0, c->stream>>>(
      c->z, c->n, c->n_ld, c->k_pad, X, D, d.sigma, sizeof(T) == 4 ? d.corrn : nullptr, d.Xh, d.Xl,
      d.Dh, d.Dl, sw, nrm, flags);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;

  ScrParams p;
  p.rows = d.rows;
  p.sw = sw;
  p.res = res;
  p.tiles = d.scr_tiles;
  p.err = d.status + 1;
  p.z = c->z;
  p.z_ld = z_ld;
  p.k_chunks = c->k_pad / kTcKChunk;
  p.m_tiles = plan->m_tiles;
  p.tiles_per_cta = screen_tiles_per_cta(c);
  const int splits = (p.m_tiles + p.tiles_per_cta - 1) / p.tiles_per_cta;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(splits, plan->strips, 1);
  cfg.blockDim = dim3(kThreadsScr, 1, 1);
  cfg.dynamicSmemBytes = kSmemScr;
  cfg.stream = c->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, screen_kernel, plan->ah, plan->al, plan->dh, plan->dl, plan->xh,
                         plan->xl, p, last_chunk_steps(c->kdim, p.k_chunks));
  if (e != cudaSuccess) return e;

  FinParams<T> f;
  f.A = A; f.b = b; f.kr = kr; f.X = X; f.D = D;
  f.corrn = sizeof(T) == 4 ? d.corrn : nullptr;
  f.rows = d.rows; f.Ah = d.Ah; f.Al = d.Al; f.Xh = d.Xh; f.Xl = d.Xl; f.Dh = d.Dh; f.Dl = d.Dl;
  f.sw = sw; f.k_pad = c->k_pad;
  f.nrm32 = nrm; f.res = res; f.tiles = d.scr_tiles; f.flags = flags;
  f.seed = c->opts.seed; f.step_ptr = d.step; f.j = j; f.walker0 = c->opts.walker0;
  f.m = c->m; f.n = c->n; f.n_ld = c->n_ld; f.z = c->z; f.z_ld = z_ld;
  f.streams = 4 * splits; f.tiles_per_cta = p.tiles_per_cta; f.m_tiles = p.m_tiles; f.mE = c->mE;
  f.lmin = d.lmin; f.lmax = d.lmax; f.theta = d.theta; f.status = d.status; f.counters = d.counters;
  f.X64 = d.X64; f.Xhi = d.Xhi; f.Xlo = d.Xlo; f.Q32 = d.Q32;
  f.corr = sizeof(T) == 4 ? d.corr : nullptr;
  f.slow = screen_slow(d);
  f.slow_clocks = screen_slow_clocks(c);
  screen_finish_kernel<T>
      <<<(c->z + kFinWalkers - 1) / kFinWalkers, kFinThreads, kFinSmem, c->stream>>>(f);
  return cudaGetLastError();
}

}  // namespace

// Bodies past the warp-per-walker path; times of whole iterations, draw included.  FP64:
// 203 us and more with the direct kernel, 25 .. 88 with the screen (n = 4 .. 100, m = 700
// .. 4000, z = 300 .. 4096).  FP32, the screen against the direct kernel, by the products
// m n z from n = 64 on: 35 / 26 us at 33 10^6 (65 walkers, 8000 x 64), 27 / 27 at 38 10^6
// (300, 2000 x 64), 24 / 27 at 41 10^6 (640, 1000 x 64), 34 / 50 at 115 10^6 (300, 4000 x
// 96); a single strip of walkers 37 / 32 at 50 10^6 (65, 8000 x 96), 39 / 40 at 67 10^6.
// Fewer columns take the direct kernel longer than their products say: 25 / 21 at m z =
// 1.5 10^6, 26 / 45 at 3 10^6 (n = 16, 32).
// Of the bodies with fewer 64 x 64 tiles than SMs, in FP64 those that the small-body
// kernel does not take (equalities, A past its shared memory) where a warp's serial
// sums (n terms for every 32 rows) or all the products are many.  An iteration with
// one equality, a warp a walker against the screen: 19.5 us where the screen's
// launches take 23 (20 x 80 with 400 walkers, 60 terms), 32 (screen 24) at 160 terms,
// 49 (28.5) at 300, 157 (33) at 1170; 32 (25) for 1500 walkers of 60 terms; 575 (36)
// for 20 to 300 walkers of a 100 x 1500 body.
bool screen_eligible(const mhar_ctx* c) {
  if (c->k_pad > 2048 || c->m_pad / kRowsTile > 65535) return false;
  if (simt_warp_path(c))
    return c->opts.precision == MHAR_FP64 &&
           (static_cast<long long>(c->n) * ((c->m + 31) / 32) >= 128 ||
            static_cast<long long>(c->m) * c->n * c->z >= 1ll << 21);
  if (c->opts.precision == MHAR_FP64) return true;
  const long long mz = static_cast<long long>(c->m) * c->z;
  return c->n >= 64 ? mz * c->n >= (c->z <= kWalkers ? 1ll << 26 : 1ll << 25) : mz >= 1ll << 21;
}

size_t screen_arena(mhar_ctx* c, uint8_t* base) {
  DeviceBuffers& d = c->d;
  size_t off = 0;
  auto take = [&](auto** p, size_t count) {
    if (base) *p = reinterpret_cast<std::remove_reference_t<decltype(*p)>>(base + off);
    off += (count * sizeof(**p) + 255) / 256 * 256;
  };
  const size_t z = static_cast<size_t>(c->z), z_ld = (z + kWalkers - 1) / kWalkers * kWalkers;
  const size_t mp = static_cast<size_t>(c->m_pad);
  const int tiles = c->m_pad / kRowsTile, per = screen_tiles_per_cta(c);
  const size_t res = static_cast<size_t>(4) * ((tiles + per - 1) / per) * z_ld;
  take(&d.Ah, mp * c->k_pad);
  take(&d.Al, mp * c->k_pad);
  take(&d.row_scale, mp);
  take(&d.bS, mp);
  take(&d.rows, 4 * mp);
  take(&d.rowk, 4 * mp);
  for (__half** p : {&d.Dh, &d.Dl, &d.Xh, &d.Xl}) take(p, z_ld * c->k_pad);
  take(&d.scr_walker, 4 * z);
  take(&d.scr_nrm, 4 * z);
  take(&d.scr_flags, 2 * z);
  take(&d.scr_res, 4 * res);
  take(&d.scr_tiles, res);
  return off;
}

cudaError_t screen_prepare(mhar_ctx* c, int* outside) {
  cudaError_t e = launch_prepare_tc_operands(c, false);
  const int groups = c->m_pad / 32;
  if (e == cudaSuccess) {
    screen_rows_kernel<<<(groups + 3) / 4, 128, 0, c->stream>>>(
        groups, c->m, c->d.bS, c->d.rowk, c->d.row_scale, c->d.b64, c->d.kr32,
        static_cast<float>(c->dir_norm2), static_cast<float>(c->dir_norminf), c->d.rows, outside);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(screen_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(kSmemScr));
  if (e == cudaSuccess)
    e = c->opts.precision == MHAR_FP64
            ? cudaFuncSetAttribute(screen_finish_kernel<double>,
                                   cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   static_cast<int>(kFinSmem))
            : cudaFuncSetAttribute(screen_finish_kernel<float>,
                                   cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   static_cast<int>(kFinSmem));
  return e;
}

cudaError_t launch_screen(mhar_ctx* c, int j) {
  if (c->opts.precision == MHAR_FP64)
    return launch_screen_t<double>(c, j, c->d.A64, c->d.b64, nullptr, c->d.X64, c->d.D64);
  return launch_screen_t<float>(c, j, c->d.A32, c->d.b32, c->d.kr32, c->d.Xhi, c->d.D32);
}

}  // namespace mhar
