// passes.cuh -- the passes over A of a handle (passes.cu).
#pragma once

#include "pdas_internal.cuh"

namespace pdas {

// How A'u is cut: column blocks of 32 V columns (V by dtype and alignment) and
// `chunks` row chunks of `rows` rows each.
struct PassTPlan {
  int64_t cblocks = 0;
  int chunks = 1;
  int64_t rows = 0;
};
PassTPlan pass_t_plan(int64_t m, int64_t n, int elem_bytes, bool vec);
// Workspace of any plan of (m, n): doubles of partial column sums, tickets
// (zero between launches).
int64_t pass_t_part_doubles(int64_t m, int64_t n, int elem_bytes);
int64_t pass_t_tickets(int64_t n);

// FP32 pairs of an n-vector as two planes: v = vh + vl, vh at p, vl at p + pairs_pitch(n).
inline int64_t pairs_pitch(int64_t n) { return (n + 7) / 8 * 8; }

// The vector of an A'u pass: u itself, or (p != null) the next direction of
// the conjugate gradients, p_new = u + b p with b = rz / sc->rz[1 - par], or p_new
// = u if first; rz, the sum of the nrz numbers at rz_part, goes to sc->rz[par] and
// p_new (another buffer than p) receives the direction.
struct PassTSrc {
  const double* u = nullptr;
  const double* p = nullptr;
  double* p_new = nullptr;
  const double* rz_part = nullptr;
  int nrz = 0;
  int par = 0;
  int first = 0;
  int absmax = 0;  // max |u| into sc->dynorm
};

// w = A'u, then per mode:
//   0: out0 = w
//   1: direction: out0 = dx = D w - x, out1 = ds = -w, out2 = w (may be null)
//   2: scaled:    out0 = D w (may be null), out2 = w (may be null), and with pairs != null the
//                 FP32 pairs of D w for a double-float pass
// With rd (mode 1, the infeasible-start variant) ds = rd - w instead of -w.
// df: double-float on the FP32 pipes (A FP32 or BF16), else FP64.
template <typename T>
cudaError_t launch_pass_t(cudaStream_t st, int64_t m, int64_t n, const T* A, bool df, const PassTSrc& src,
                          double* part, double* maxpart, unsigned* ctickets, int mode, const double* x, const double* D,
                          double* out0, double* out1, double* out2, float* pairs, Scalars* sc,
                          const double* rd = nullptr);

// out_p = A_p. v (base == null) or base_p - A_p. v, in FP64 (v) or, with pairs
// != null, in double-float (the pairs of v).  norm_slot 0, 1: max |out_p| into
// sc->rnorm or sc->rho_norm.  dot != null: sum_p dot_p out_p into sc->dot_b.
template <typename T>
cudaError_t launch_pass(cudaStream_t st, int64_t m, int64_t n, const T* A, const double* v, const float* pairs,
                        const double* base, double* out, double* part, unsigned* tickets, Scalars* sc, int norm_slot,
                        const double* dot = nullptr);

// The pairs of v (n doubles).
cudaError_t launch_split_pairs(cudaStream_t st, int64_t n, const double* v, float* pairs);

}  // namespace pdas
