"""The FP64 Box-Muller pair (csrc/normals_f64.cuh), compiled for the host, against extended
precision: the ends of the 32-bit range, every table bin's edges, words at random.

Bounds: sqrt(-2 ln u) one unit in the last place (half from a logarithm with an error of
at most one, half from the root's rounding), sin and cos one (half from the last sum, the
rest from the table's and the terms' roundings)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2104_07097_gb300", "csrc")

MAIN = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
#define __device__
#define __forceinline__ inline
#define __align__(x)
struct double2 { double x, y; };
static double __hiloint2double(int h, int l) {
  uint64_t b = (uint64_t(uint32_t(h)) << 32) | uint32_t(l);
  double d; memcpy(&d, &b, 8); return d;
}
static double __longlong_as_double(long long b) { double d; memcpy(&d, &b, 8); return d; }
static int __clzll(long long v) { return __builtin_clzll(v); }
static float rsqrtf(float x) { return 1.0f / sqrtf(x); }
#include "normals.h"
static double ulps(long double got, long double ref) {
  int e; frexpl(ref, &e); return double(fabsl(got - ref) / ldexpl(1.0L, e - 53));
}
int main() {
  std::mt19937_64 g(1);
  const long double pi = acosl(-1.0L), q = sqrtl(0.5L);
  const long double cv[8] = {1, q, 0, -q, -1, -q, 0, q}, sv[8] = {0, q, 1, q, 0, -q, -1, -q};
  double mr = 0, mt = 0;
  for (long t = 0; t < 3000000; ++t) {
    uint32_t w = uint32_t(g());
    if (t < 400000) w = uint32_t(t);
    else if (t < 800000) w = ~uint32_t(t - 400000);
    else if (t < 1200000) w = (uint32_t(t % 129) << 25) + uint32_t(g() % 4001) - 2000u;
    else if (t < 1600000) {   // the logarithm's bins at every binary exponent
      const int k = t % 32;
      w = uint32_t(((64ull + (t / 32) % 64) * 2 + 1) << 25 >> k) + uint32_t(g() % 65) - 32u;
    }
    const long double u = ((long double)w + 0.5L) * ldexpl(1.0L, -32);
    const long double r = sqrtl(u > 0.5L ? -2 * log1pl(u - 1) : -2 * logl(u));
    mr = fmax(mr, ulps(mhar::radius_f64(w), r));
    const uint64_t p = 2ull * w + 1;
    const int o = int((p + (1ull << 29)) >> 30) & 7;
    const long double d = (long double)(int64_t(p) - int64_t((p + (1ull << 29)) >> 30 << 30)) * pi * ldexpl(1.0L, -32);
    const long double C = cv[o] * cosl(d) - sv[o] * sinl(d), S = sv[o] * cosl(d) + cv[o] * sinl(d);
    double s, c;
    mhar::unit_circle_f64(w, s, c);
    mt = fmax(mt, fmax(ulps(s, S), ulps(c, C)));
  }
  printf("%.4f %.4f\n", mr, mt);
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_normals_within_one_ulp(tmp_path):
    text = open(os.path.join(CSRC, "normals_f64.cuh")).read()
    text = text.replace("#include <cuda_runtime.h>", "")
    at = text.index("// The tables into L1")            # the one function that is PTX
    text = text[:at] + text[text.index("// Box-Muller pair"):]
    (tmp_path / "normals.h").write_text(text)
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = str(tmp_path / "normals")
    subprocess.run(["g++", "-O2", "-w", "-ffp-contract=off", str(tmp_path / "main.cpp"), "-o", exe],
                   check=True)
    radius, circle = map(float, subprocess.run([exe], check=True, capture_output=True,
                                               text=True).stdout.split())
    assert radius <= 1.0 and circle <= 1.0
