"""The fit's Jacobi rotation (csrc/jacobi_angle.cuh), compiled for the host with
__fdividef as its documentation has it: a quotient for divisors in 2^-126 .. 2^126, and
here NaN for any other.

cos^2 + sin^2 = 1 to 4 roundings of FP64, and the tangent t of a rotation solves
t^2 + 2 tau t = 1 to the 1e-5 that FP32's quotient and root leave, for every entry that is
a normal number and |tau| up to 2^60; a smaller entry, a larger tau: any rotation."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2104_07097_gb300", "csrc")

MAIN = r"""
#include <cmath>
#include <cstdio>
#include <random>
#define __device__
#define __forceinline__ inline
struct double2 { double x, y; };
static double2 make_double2(double x, double y) { return {x, y}; }
static float rsqrtf(float x) { return 1.0f / sqrtf(x); }
static float sqrt_approx(float x) { return sqrtf(x); }
static float __fdividef(float x, float y) {
  return fabsf(y) >= 0x1p-126f && fabsf(y) <= 0x1p126f ? x / y : NAN;
}
#include "angle.h"
int main() {
  std::mt19937_64 g(1);
  long bad = 0;
  double worst = 0;
  auto value = [&](int lo) {
    const int k = int(g() % 12);
    if (k == 0) return 0.0f;
    const float v = ldexpf(0.5f + 0.5f * float(g() >> 40) * 0x1p-24f, lo + int(g() % (1 - lo)));
    return g() & 1 ? v : -v;
  };
  for (long t = 0; t < 4000000; ++t) {
    float apq = value(-148);
    float diff = t % 4 ? value(-148) : 0.0f;
    if (t % 5 == 0) diff = 2.0f * apq * value(-20);
    const double2 r = mhar::jacobi_rotation(apq, diff);
    if (!(fabs(r.x * r.x + r.y * r.y - 1.0) <= 4.5e-16) || !(r.x > 0.7)) { ++bad; continue; }
    if (fabsf(apq) < 0x1p-126f) continue;
    const double tau = double(diff) / (2.0 * double(apq));
    if (fabs(tau) > 0x1p60) continue;
    const double tn = r.y / r.x;
    const double want = (tau >= 0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
    worst = fmax(worst, fabs(tn / want - 1.0));
  }
  printf("%ld %.3e\n", bad, worst);
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_rotation_is_one(tmp_path):
    text = open(os.path.join(CSRC, "jacobi_angle.cuh")).read()
    text = text.replace("#include <cuda_runtime.h>", "")
    at = text.index("__device__ __forceinline__ float sqrt_approx")   # PTX
    text = text[:at] + text[text.index("// (cos, sin) for the entry"):]
    (tmp_path / "angle.h").write_text(text)
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = str(tmp_path / "angle")
    subprocess.run(["g++", "-O2", "-w", "-ffp-contract=off", str(tmp_path / "main.cpp"), "-o", exe],
                   check=True)
    bad, worst = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert int(bad) == 0 and float(worst) <= 1e-5
