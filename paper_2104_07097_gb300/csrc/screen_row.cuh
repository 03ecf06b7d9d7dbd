// screen_row.cuh -- the row that a bound kept by the screen belongs to (kernels_screen.cu).
//
// tiles: the row tiles of a stream's least bounds, lambda_max's in the low half,
// lambda_min's in the high; a stream covers 32 rows of each 128-row tile; key: the bound,
// the row within those 32 in its low five bits.  Padding rows bound nothing, but after an
// expired wait the sums are unfinished ones and theirs may look finite: never past m.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace mhar {

__host__ __device__ inline int screen_row(uint32_t tiles, bool low, int stream, uint32_t key,
                                          int m) {
  const int row = static_cast<int>(low ? tiles >> 16 : tiles & 0xffffu) * 128 + (stream & 3) * 32 +
                  static_cast<int>(key & 31u);
  return row < m ? row : m - 1;
}

}  // namespace mhar
