"""The row of a screen's bound (csrc/screen_row.cuh), compiled for the host: every row of a
body comes back, and no key or tile word of a padded tile leads past the body."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2104_07097_gb300", "csrc")

MAIN = r"""
#include <cstdint>
#include <cstdio>
#include <initializer_list>
#define __host__
#define __device__
#include "row.h"
int main() {
  long bad = 0;
  for (int m : {1, 31, 32, 33, 127, 128, 129, 700, 1024, 2000, 5000, 8388480}) {
    const int tiles = (m + 127) / 128;
    for (int t = tiles > 50 ? tiles - 50 : 0; t < tiles; ++t)
      for (int st = 0; st < 12; ++st)
        for (uint32_t low5 = 0; low5 < 32; ++low5)
          for (int low = 0; low < 2; ++low) {
            const uint32_t other = 0x1234u;
            const uint32_t word = low ? (uint32_t(t) << 16) | other : (other << 16) | uint32_t(t);
            const int row = 128 * t + 32 * (st & 3) + int(low5);
            const int got = mhar::screen_row(word, low, st, 0x3f800000u | low5, m);
            bad += got < 0 || got >= m || (row < m && got != row);
          }
  }
  printf("%ld\n", bad);
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_rows_stay_inside(tmp_path):
    text = open(os.path.join(CSRC, "screen_row.cuh")).read()
    (tmp_path / "row.h").write_text(text.replace("#include <cuda_runtime.h>", ""))
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = str(tmp_path / "row")
    subprocess.run(["g++", "-O2", "-w", str(tmp_path / "main.cpp"), "-o", exe], check=True)
    assert subprocess.run([exe], check=True, capture_output=True, text=True).stdout == "0\n"
