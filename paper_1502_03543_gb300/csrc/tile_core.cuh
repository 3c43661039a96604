// tile_core.cuh -- tile sizes and the lower-triangle tile order shared by the
// SIMT normal-matrix builder (M = A D A', Section V) and the Cholesky factors.
#pragma once

#include "pdas_internal.cuh"

namespace pdas {

constexpr int kKc = 16;  // K chunk of the SIMT normal matrices

constexpr int kBig = 128;
static_assert(kBig == kCholTile, "the tile Cholesky works on 128 x 128 tiles");

// Lower-triangle tile index t -> (ti, tj) with ti >= tj.
__device__ __forceinline__ void lower_tile(int64_t t, int64_t& ti, int64_t& tj) {
  int64_t i = (int64_t)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);  // FP32 estimate, corrected below
  while (i * (i + 1) / 2 > t) --i;
  while ((i + 1) * (i + 2) / 2 <= t) ++i;
  ti = i;
  tj = t - i * (i + 1) / 2;
}

}  // namespace pdas
