// jacobi_angle.cuh -- the rotation that zeroes one off-diagonal entry of a symmetric
// matrix (Golub & Van Loan, Matrix Computations, Section 8.5), its angle from FP32.
//
// The matrix is scaled to a trace near 1.  __fdividef is accurate for divisors between
// 2^-126 and 2^126 and undefined past them (0 over a subnormal is 0 * Inf), so an entry
// below 2^-126, 1e-38 of the trace, is left alone, and |tau| is cut at 2^62, where the
// entry is below 2^-62 of the diagonal's difference: both far below the 1e-15 at which
// the sweeps stop.
#pragma once
#include <cmath>
#include <cuda_runtime.h>

namespace mhar {

__device__ __forceinline__ float sqrt_approx(float v) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}

// (cos, sin) for the entry apq and diff = a_qq - a_pp.
__device__ __forceinline__ double2 jacobi_rotation(float apq, float diff) {
  double2 r = make_double2(1.0, 0.0);
  if (fabsf(apq) >= 0x1p-126f) {
    const float tau = __fdividef(diff, 2.0f * apq), a = fminf(fabsf(tau), 0x1p62f);
    const float root = a + sqrt_approx(fmaf(a, a, 1.0f));
    const double tn = static_cast<double>(__fdividef(tau >= 0.0f ? 1.0f : -1.0f, root));
    // 1 / sqrt(1 + tn^2), 1 <= 1 + tn^2 <= 2: one step of third order from
    // the FP32 value (error below 1e-20 of it before rounding).
    const double w = fma(tn, tn, 1.0);
    const double y = static_cast<double>(rsqrtf(static_cast<float>(w)));
    const double d = fma(-w * y, y, 1.0);
    r.x = fma(y * d, fma(0.375, d, 0.5), y);
    r.y = tn * r.x;
  }
  return r;
}

}  // namespace mhar
