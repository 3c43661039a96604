// syrk_simt.cuh -- the SIMT normal matrices (syrk_simt.cu): how M is cut into
// tiles and K slices, and the launches.
#pragma once

#include "pdas_internal.cuh"

namespace pdas {

struct SimtPlan {
  int tile = 0;         // tile edge
  int64_t tiles = 0;    // lower-triangle tiles (one ticket each, zero between launches)
  int64_t ldk = 0;      // FP32: columns of the operand planes (2 x m x ldk floats)
  int64_t kslice = 0;   // columns per slice (a multiple of 16)
  int slices = 1;       // K slices per tile
  size_t part_bytes = 0;  // FP32: workspace of the partial tiles (0 with one slice)
};
SimtPlan simt_plan_fp64(int64_t m, int64_t n);
SimtPlan simt_plan_fp32(int64_t m, int64_t n);
size_t simt_fp64_part_bytes(int64_t m);    // FP64: workspace of the partial tiles, for any n
int64_t simt_ticket_count(int64_t m);      // tickets of either, for any n

// Lower triangle of M = A D A' in FP64.  part: simt_fp64_part_bytes(m).
template <typename T>
cudaError_t launch_syrk_fp64(cudaStream_t st, int64_t m, int64_t n, const T* A, const double* D, double* M,
                             int64_t ldm, void* part, unsigned* tickets, const Scalars* sc);
// Lower triangle of M = A D A' in FP32; adds its launches to
// *launches.
template <typename T>
cudaError_t launch_syrk_fp32(cudaStream_t st, int64_t m, int64_t n, const T* A, const double* D, float* planes,
                             float* M, int64_t ldm, void* part, unsigned* tickets, const Scalars* sc, int* launches);

}  // namespace pdas
