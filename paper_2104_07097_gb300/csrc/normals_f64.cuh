// normals_f64.cuh -- the FP64 Box-Muller pair from two 32-bit words.
//
// FP64 runs at 1/64 of the FP32 rate on this GPU (two operations a clock and SM),
// and log, sincospi and sqrt of the CUDA library spend about 260 of them on a
// pair: 4096 walkers of 100 dimensions took 62 us to draw.  The uniforms are
// (w + 1/2) 2^-32, odd multiples of 2^-33, so that the argument reductions are
// exact in integers or in one FMA, and short polynomials suffice: 50 FP64
// operations, 25 us.
//   ln u      table-driven (Tang, "Table-driven implementation of the logarithm
//             function in IEEE floating-point arithmetic", ACM TOMS 16, 1990):
//             u = 2^-k f, f in [1/sqrt 2, sqrt 2), r = f c - 1 exactly with c = 64 / i
//             to 13 bits, -ln u = k ln 2 + ln c - ln(1 + r), the first two in two
//             parts, the last by its Taylor series to r^9 (|r| < 0.0114).  c = 1
//             around f = 1, where the result is small, so it keeps its relative
//             accuracy.
//   sin, cos  of the nearest multiple of pi / 64 from a table in two parts, and of
//             the rest |delta| < 0.0246 by their Taylor series.
//   sqrt      Goldschmidt's iteration with Markstein's last step (Markstein, "IA-64
//             and Elementary Functions", 2000) from the FP32 reciprocal root.
// Largest errors over 2 10^7 words against extended precision: 0.86 ulp (radius),
// 0.79 (sin, cos); mean 0.27 and 0.25.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace mhar {

// i = 45 .. 91: 64 / i to 13 bits, and its logarithm as a multiple of 2^-42 and
// the rest.
static __device__ const double __align__(16) kLogTable[47][4] = {
    {0x1.6c10000000000p+0, 0x1.689983bca6000p-2, 0x1.25a53e0c9f034p-46, 0.0},
    {0x1.6430000000000p+0, 0x1.5234e0670a000p-2, 0x1.49483d21b40d9p-44, 0.0},
    {0x1.5ca0000000000p+0, 0x1.3c3b2736b4000p-2, -0x1.3e5d1e9d3ddf9p-47, 0.0},
    {0x1.5550000000000p+0, 0x1.268620f34d000p-2, 0x1.8f44b998bb50ep-44, 0.0},
    {0x1.4e60000000000p+0, 0x1.117ee81dfe000p-2, 0x1.30f778a2e8cbdp-44, 0.0},
    {0x1.47b0000000000p+0, 0x1.f99dc6c23c000p-3, -0x1.7ed06117b4369p-44, 0.0},
    {0x1.4140000000000p+0, 0x1.d0fb7f2256000p-3, -0x1.af52b20633b29p-47, 0.0},
    {0x1.3b10000000000p+0, 0x1.a926d3a4ae000p-3, -0x1.53935e85baac8p-44, 0.0},
    {0x1.3520000000000p+0, 0x1.8230164c1a000p-3, 0x1.98dd68a5d0b48p-46, 0.0},
    {0x1.2f70000000000p+0, 0x1.5c28060c46000p-3, 0x1.6ece374e0e858p-44, 0.0},
    {0x1.29e0000000000p+0, 0x1.3643cad058000p-3, 0x1.1e18f2132dfd5p-44, 0.0},
    {0x1.2490000000000p+0, 0x1.1168e8127e000p-3, 0x1.93436f195cb75p-46, 0.0},
    {0x1.1f70000000000p+0, 0x1.da6e7637c4000p-4, 0x1.a83eac951c1aap-46, 0.0},
    {0x1.1a80000000000p+0, 0x1.9375e55594000p-4, 0x1.eddc37380c364p-44, 0.0},
    {0x1.15b0000000000p+0, 0x1.4d1515b988000p-4, -0x1.8e7d02e3f5e95p-47, 0.0},
    {0x1.1110000000000p+0, 0x1.08498b51e4000p-4, -0x1.93b33c55fb24fp-46, 0.0},
    {0x1.0c90000000000p+0, 0x1.88729e70f0000p-5, -0x1.9c8d8f692991dp-45, 0.0},
    {0x1.0840000000000p+0, 0x1.03d5d85e70000p-5, 0x1.f778960ed29cfp-44, 0.0},
    {0x1.0410000000000p+0, 0x1.01f5658730000p-6, 0x1.6107d26f92eb5p-44, 0.0},
    {0x1.0000000000000p+0, 0x0.0p+0, 0x0.0p+0, 0.0},
    {0x1.f820000000000p-1, -0x1.fbea8b13c0000p-7, -0x1.ec927b17e4e13p-50, 0.0},
    {0x1.f080000000000p-1, -0x1.f7a9b16780000p-6, -0x1.42ad9271be7d7p-45, 0.0},
    {0x1.e920000000000p-1, -0x1.766d923c20000p-5, -0x1.ff0a82f1c24c1p-46, 0.0},
    {0x1.e1e0000000000p-1, -0x1.f0c30c1118000p-5, 0x1.caef3588b7d80p-45, 0.0},
    {0x1.dae0000000000p-1, -0x1.345179b63c000p-4, -0x1.d4203d36150d0p-44, 0.0},
    {0x1.d420000000000p-1, -0x1.6ef528c058000p-4, 0x1.5d462d767cadep-44, 0.0},
    {0x1.cd80000000000p-1, -0x1.a956d3ecac000p-4, -0x1.e63794c02c4afp-44, 0.0},
    {0x1.c720000000000p-1, -0x1.e2507702b0000p-4, 0x1.f897980522249p-45, 0.0},
    {0x1.c0e0000000000p-1, -0x1.0d79e7cd48000p-3, -0x1.cb422847849e4p-44, 0.0},
    {0x1.bac0000000000p-1, -0x1.299d30c606000p-3, -0x1.d4d0079dc08d9p-44, 0.0},
    {0x1.b4e0000000000p-1, -0x1.44f8b726f8000p-3, -0x1.df6a4432b9bb4p-44, 0.0},
    {0x1.af20000000000p-1, -0x1.601b076e7a000p-3, -0x1.152d7d4dfc8e5p-44, 0.0},
    {0x1.a980000000000p-1, -0x1.7b00916516000p-3, 0x1.ae75fcb067e57p-44, 0.0},
    {0x1.a420000000000p-1, -0x1.9509aa0044000p-3, -0x1.f1e675b4d35c6p-44, 0.0},
    {0x1.9ec0000000000p-1, -0x1.af6895610e000p-3, 0x1.148288bf7a937p-45, 0.0},
    {0x1.99a0000000000p-1, -0x1.c8df7cb9a8000p-3, -0x1.eee42f58e1e6ep-44, 0.0},
    {0x1.9480000000000p-1, -0x1.e2a877a6b2000p-3, -0x1.823817787081ap-44, 0.0},
    {0x1.8fa0000000000p-1, -0x1.fb7d86eee4000p-3, 0x1.1c061cdb8097bp-45, 0.0},
    {0x1.8ac0000000000p-1, -0x1.0a504e97bb000p-2, -0x1.03094e6690c44p-44, 0.0},
    {0x1.8620000000000p-1, -0x1.1661caecba000p-2, 0x1.171fff9fc4abbp-44, 0.0},
    {0x1.8180000000000p-1, -0x1.22981fbef8000p-2, 0x1.a1421609580dap-44, 0.0},
    {0x1.7d00000000000p-1, -0x1.2e9e2bce12000p-2, -0x1.4300c128d1dc2p-45, 0.0},
    {0x1.78a0000000000p-1, -0x1.3a71c56bb5000p-2, 0x1.ce772094aef70p-44, 0.0},
    {0x1.7460000000000p-1, -0x1.4610bc29c6000p-2, 0x1.e82c9f310c8e6p-46, 0.0},
    {0x1.7020000000000p-1, -0x1.51d1d93104000p-2, -0x1.5b0faa20d9c8ep-44, 0.0},
    {0x1.6c20000000000p-1, -0x1.5d01dc49ff000p-2, -0x1.740ab8cfa5ed3p-45, 0.0},
    {0x1.6820000000000p-1, -0x1.68518244d0000p-2, 0x1.3c6e803ba0773p-44, 0.0},
};
// sin(i pi / 64) and what its rounding leaves.
static __device__ const double __align__(16) kSinTable[33][2] = {
    {0x0.0p+0, 0x0.0p+0},
    {0x1.91f65f10dd814p-5, -0x1.912bd0d569a90p-61},
    {0x1.917a6bc29b42cp-4, -0x1.e2718d26ed688p-60},
    {0x1.2c8106e8e613ap-3, 0x1.13000a89a11e0p-58},
    {0x1.8f8b83c69a60bp-3, -0x1.26d19b9ff8d82p-57},
    {0x1.f19f97b215f1bp-3, -0x1.42deef11da2c4p-57},
    {0x1.294062ed59f06p-2, -0x1.5d28da2c4612dp-56},
    {0x1.58f9a75ab1fddp-2, -0x1.efdc0d58cf620p-62},
    {0x1.87de2a6aea963p-2, -0x1.72cedd3d5a610p-57},
    {0x1.b5d1009e15cc0p-2, 0x1.5b362cb974183p-57},
    {0x1.e2b5d3806f63bp-2, 0x1.e0d891d3c6841p-58},
    {0x1.073879922ffeep-1, -0x1.a5a014347406cp-55},
    {0x1.1c73b39ae68c8p-1, 0x1.b25dd267f6600p-55},
    {0x1.30ff7fce17035p-1, -0x1.efcc626f74a6fp-57},
    {0x1.44cf325091dd6p-1, 0x1.8076a2cfdc6b3p-57},
    {0x1.57d69348ceca0p-1, -0x1.75720992bfbb2p-55},
    {0x1.6a09e667f3bcdp-1, -0x1.bdd3413b26456p-55},
    {0x1.7b5df226aafafp-1, -0x1.0f537acdf0ad7p-56},
    {0x1.8bc806b151741p-1, -0x1.2c5e12ed1336dp-55},
    {0x1.9b3e047f38741p-1, -0x1.30ee286712474p-55},
    {0x1.a9b66290ea1a3p-1, 0x1.9f630e8b6dac8p-60},
    {0x1.b728345196e3ep-1, -0x1.bc69f324e6d61p-55},
    {0x1.c38b2f180bdb1p-1, -0x1.6e0b1757c8d07p-56},
    {0x1.ced7af43cc773p-1, -0x1.e7b6bb5ab58aep-58},
    {0x1.d906bcf328d46p-1, 0x1.457e610231ac2p-56},
    {0x1.e212104f686e5p-1, -0x1.014c76c126527p-55},
    {0x1.e9f4156c62ddap-1, 0x1.760b1e2e3f81ep-55},
    {0x1.f0a7efb9230d7p-1, 0x1.52c7adc6b4989p-56},
    {0x1.f6297cff75cb0p-1, 0x1.562172a361fd3p-56},
    {0x1.fa7557f08a517p-1, -0x1.7a0a8ca13571fp-55},
    {0x1.fd88da3d12526p-1, -0x1.87df6378811c7p-55},
    {0x1.ff621e3796d7ep-1, -0x1.c57bc2e24aa15p-57},
    {0x1.0000000000000p+0, 0x0.0p+0},
};

// A signed 32-bit integer as a double, with one FP64 subtraction: 2^52 + 2^31 + v.
__device__ __forceinline__ double int_f64(int32_t v) {
  return __hiloint2double(0x43300000, static_cast<int>(static_cast<uint32_t>(v) ^ 0x80000000u)) -
         4503601774854144.0;
}

// sqrt(-2 ln u), u = (w + 1/2) 2^-32.
__device__ __forceinline__ double radius_f64(uint32_t w) {
  // v = 2 w + 1 = 2^(32 - k) f, f in [1/sqrt 2, sqrt 2).
  const uint64_t v = 2ull * w + 1ull;
  const int lz = __clzll(static_cast<long long>(v));        // 31 .. 63
  const uint64_t m = v << (lz - 11);                         // bit 52 set
  const bool half = m >= 0x0016a09e667f3bcdull;              // above sqrt 2
  const uint64_t bits = (m & 0x000fffffffffffffull) | (half ? 0x3fe0000000000000ull : 0x3ff0000000000000ull);
  const double f = __longlong_as_double(static_cast<long long>(bits));
  const int k = lz - 30 - (half ? 1 : 0);
  // The nearest multiple of 1/64 (f is m 2^-52, or half of it).
  const int i = static_cast<int>(((m >> (half ? 46 : 45)) + 1) >> 1) - 45;
  const double2 t0 = *reinterpret_cast<const double2*>(&kLogTable[i][0]);
  const double lo_c = kLogTable[i][2];
  const double r = fma(f, t0.x, -1.0);                       // exact
  const double r2 = r * r;
  double q = fma(r, 1.0 / 9.0, -1.0 / 8.0);
  q = fma(r, q, 1.0 / 7.0);
  q = fma(r, q, -1.0 / 6.0);
  q = fma(r, q, 1.0 / 5.0);
  q = fma(r, q, -1.0 / 4.0);
  q = fma(r, q, 1.0 / 3.0);
  const double p = fma(-r, q, 0.5);                          // r - ln(1 + r) = r^2 p
  const double kd = int_f64(k);
  const double hi = fma(kd, 0x1.62e42fefa3800p-1, t0.y);     // exact
  const double lo = fma(kd, 0x1.ef35793c76730p-45, lo_c);
  const double s = hi - r;
  const double e = (hi - s) - r;                             // |hi| >= |r|, or hi = 0
  const double x = 2.0 * (s + fma(r2, p, e + lo));
  // sqrt(x), 2^-33 < x < 47.
  const double y = static_cast<double>(rsqrtf(static_cast<float>(x)));
  double g = x * y, h = 0.5 * y;
  const double d = fma(-h, g, 0.5);
  g = fma(g, d, g);
  h = fma(h, d, h);
  return fma(fma(-g, g, x), h, g);
}

// sin and cos of 2 pi u, u = (w + 1/2) 2^-32.
__device__ __forceinline__ void unit_circle_f64(uint32_t w, double& sn, double& cs) {
  // The phase 2 w + 1 of 2^33: multiples of 2^26 (pi / 64) and the rest.
  const uint32_t i = (w + (1u << 24)) >> 25;                // (2 w + 1 + 2^25) >> 26, up to 128
  const int32_t rest = static_cast<int32_t>(2u * w + 1u - (i << 26));   // |rest| < 2^25
  const uint32_t j = i & 31u, quarter = (i >> 5) & 3u;
  const double2 a = *reinterpret_cast<const double2*>(&kSinTable[j][0]);
  const double2 b = *reinterpret_cast<const double2*>(&kSinTable[32 - j][0]);
  const double rd = int_f64(rest);
  const double d = rd * 0x1.921fb54442d18p-31;
  const double dl = fma(rd, 0x1.1a62633145c07p-85, fma(rd, 0x1.921fb54442d18p-31, -d));
  const double d2 = d * d;
  double p = fma(d2, -1.0 / 5040.0, 1.0 / 120.0);
  p = fma(d2, p, -1.0 / 6.0);
  p = fma(d * d2, p, dl);                                    // sin d - d
  double c = fma(d2, -1.0 / 720.0, 1.0 / 24.0);
  c = d2 * fma(d2, c, -0.5);                                 // cos d - 1
  // The largest terms last.
  const double s0 = a.x + fma(b.x, d, fma(b.x, p, fma(a.x, c, a.y)));
  const double c0 = b.x + fma(-a.x, d, fma(-a.x, p, fma(b.x, c, b.y)));
  sn = quarter & 1u ? c0 : s0;
  cs = quarter & 1u ? s0 : c0;
  if (quarter & 2u) sn = -sn;
  if (quarter == 1u || quarter == 2u) cs = -cs;
}

// The tables into L1 ahead of the first draw (threads tid = 0 .. 16 or more).
__device__ __forceinline__ void prefetch_normals_f64(int tid) {
  const char* t = tid < 12 ? reinterpret_cast<const char*>(kLogTable) + 128 * tid
                           : reinterpret_cast<const char*>(kSinTable) + 128 * (tid - 12);
  if (tid < 17) asm volatile("prefetch.global.L1 [%0];" ::"l"(t));
}

// Box-Muller pair from two words.
__device__ __forceinline__ void box_muller_f64(uint32_t wa, uint32_t wb, double& z0, double& z1) {
  const double r = radius_f64(wa);
  double s, c;
  unit_circle_f64(wb, s, c);
  z0 = r * c;
  z1 = r * s;
}

}  // namespace mhar
