// pdas_internal.cuh -- shared declarations of the libpdas CUDA sources.
//
// Layout in HBM (all row-major, all resident for the life of a handle):
//   A       m x n, caller-owned, in its storage dtype (f64 / f32 / bf16);
//   M, L    m x m with leading dimension ldm = round_up(m, 16), lower
//           triangle only; L overwrites M in place;
//   vectors D, r, dy, w, ... in FP64.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "pdas.h"
#include "pdas_components.h"

namespace pdas {

constexpr int kThreads = 256;   // threads of every elementwise / reduction kernel
constexpr int kTile = 64;       // SIMT SYRK / Cholesky tile edge
constexpr int kPartMax = 65536;  // capacity of the reduction-partials buffer (blocks)

// Scalars written by the device reductions; the host reads the whole struct
// once per iteration.
struct Scalars {
  double dmax, dmin;   // max, min of D = x/s
  double psi, theta;   // ratio test and step length
  double cx, by, xs;   // c'x, b'y, x's after the step
  double rel_gap;      // (c'x - b'y)/(1+|c'x|)
  double rnorm;        // ||A x||_inf
  double rho_norm;     // ||A x - M dy||_inf of the latest residual
  double rz[2];        // conjugate gradients: rho'z of this step and the one before, in turn
  double dot_b;        // ... p'q
  double mnorm;        // max_p M_pp of the formed normal matrix (a lower bound on ||M||)
  double dynorm;       // ||dy||_inf
  double pres, dres;   // infeasible-start variant: relative primal and dual residuals
  int status;          // 0, or a pdas_status error detected on the device
  int fail_index;      // failing pivot for PDAS_ERR_NOT_SPD
  int bad_iterate;     // nonzero if some x_j <= 0 or s_j <= 0 (or not finite)
  int wait_us;         // limit of the bounded inter-block waits in microseconds (0: 2 s)
};

// Counters for the "last block finishes the reduction" pattern and the
// triangular-solve tickets.
enum Ticket { T_SCALING = 0, T_PSI, T_STEP, T_NORM, T_NORM2, T_DOT, T_TRSVB, T_RES, T_COUNT };

// ---- exact widening of the stored A ---------------------------------------
__device__ __forceinline__ double widen(double v) { return v; }
__device__ __forceinline__ double widen(float v) { return (double)v; }
__device__ __forceinline__ double widen(__nv_bfloat16 v) { return (double)__bfloat162float(v); }
// FP32 -> FP64 widening by bit manipulation on the integer pipes: on GB300
// the FP64 pipe is the bound of every pass over A, and a conversion
// instruction would occupy it as long as the multiply-add does.  Exact for
// every FP32 value: normal numbers move their exponent from bias 127 to
// 1023, zeros keep their sign, Inf/NaN map to exponent 2047; subnormals take
// the conversion instruction (they do not occur in practice).
__device__ __forceinline__ double widen_bits(uint32_t u) {
  const uint32_t e = (u >> 23) & 0xffu;
  const uint32_t mant = u & 0x7fffffu;
  const unsigned long long sign = (unsigned long long)(u & 0x80000000u) << 32;
  if (e == 0u) {
    if (mant == 0u) return __longlong_as_double((long long)sign);
    return (double)__uint_as_float(u);
  }
  const unsigned long long e64 = (e == 0xffu) ? 2047ull : (unsigned long long)(e + 896u);
  return __longlong_as_double((long long)(sign | (e64 << 52) | ((unsigned long long)mant << 29)));
}

// widen() without the conversion instruction.
__device__ __forceinline__ double widen_int(double v) { return v; }
__device__ __forceinline__ double widen_int(float v) { return widen_bits(__float_as_uint(v)); }
__device__ __forceinline__ double widen_int(__nv_bfloat16 v) {
  return widen_bits((uint32_t)__bfloat16_as_ushort(v) << 16);
}

__device__ __forceinline__ float widen32(double v) { return (float)v; }
__device__ __forceinline__ float widen32(float v) { return v; }
__device__ __forceinline__ float widen32(__nv_bfloat16 v) { return __bfloat162float(v); }

// ---- launch helpers (host) ------------------------------------------------
// Lets a kernel whose dynamic shared memory depends on the handle be launched
// with `bytes` of it.  The limit belongs to the function, not to a handle: it is
// set to all that the device gives, so that a handle made later does not lower it
// under an earlier one.
template <typename K>
cudaError_t allow_smem(K* kernel, size_t bytes) {
  cudaFuncAttributes fa;
  int dev = 0, most = 0;
  cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  most -= (int)fa.sharedSizeBytes;
  if (bytes > (size_t)most) return cudaErrorInvalidValue;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
}

// Each returns cudaGetLastError() of its launch.
// Partial column sums of A'u by row chunks (no handle; passes.cuh has a handle's passes).
template <typename T>
cudaError_t launch_gemv_t(cudaStream_t st, int64_t m, int64_t n, const T* A, const double* u, double* part,
                          int chunks, int64_t rows_per_chunk);

// out = the sum of those partials.
cudaError_t launch_gemv_t_sum(cudaStream_t st, int64_t n, int chunks, const double* part, double* out,
                              const Scalars* sc);
// The direction from w = A'dy: ds = -w, dx = D w - x; with rd (the
// infeasible-start variant) ds = rd - w, dx = D (w - rd) - x.
cudaError_t launch_direction(cudaStream_t st, int64_t n, const double* w, const double* x, const double* D, double* dx,
                             double* ds, const Scalars* sc, const double* rd = nullptr);
// Infeasible-start variant: rd = (c - w) - s (w = A'y) and nu = -(D rd), so
// that b - A nu = b + A D rd is the right-hand side of the normal equations.
cudaError_t launch_dual_residual(cudaStream_t st, int64_t n, const double* c, const double* s, const double* w,
                                 const double* D, double* rd, double* nu, const Scalars* sc);
// sc->pres = max|rp| / (1 + max|b|) with rp = b - A x (m), sc->dres =
// max|(c - w) - s| / (1 + max|c|) with w = A'y (n).
cudaError_t launch_residual_norms(cudaStream_t st, int64_t m, int64_t n, const double* b, const double* rp,
                                  const double* c, const double* w, const double* s, double* part,
                                  unsigned* tickets, Scalars* sc);
cudaError_t launch_scaling(cudaStream_t st, int64_t n, const double* x, const double* s, double* D, double* part,
                           unsigned* tickets, Scalars* sc);
// capped: theta = min(1, alpha/psi) (infeasible-start variant) instead of 1 when psi <= 1.
cudaError_t launch_psi(cudaStream_t st, int64_t n, const double* x, const double* s, const double* dx,
                       const double* ds, double alpha, double* part, unsigned* tickets, Scalars* sc,
                       bool capped = false);
cudaError_t launch_step(cudaStream_t st, int64_t m, int64_t n, const double* b, const double* c, double* x,
                        double* y, double* s, const double* dx, const double* dy, const double* ds, double* part,
                        unsigned* tickets, Scalars* sc);
// *out = *sc and then *seq = want, both in pinned host memory.
cudaError_t launch_snapshot(cudaStream_t st, const Scalars* sc, Scalars* out, unsigned* seq, unsigned want);
cudaError_t launch_axpy(cudaStream_t st, int64_t n, double a, const double* xv, double* yv, const Scalars* sc);
// The step length rz / pq of the conjugate gradients (rz = rho'z, pq = p'M p).
// False if there is no step to take: a quotient of two positive numbers that is
// finite is the only one that descends.  (pq is zero, negative or NaN where M
// is singular to working precision or where the numbers leave the exponent
// range; the device and the host decide by this same rule.)
__host__ __device__ inline bool cg_step_length(double rz, double pq, double* a) {
  *a = rz / pq;
  return rz > 0.0 && pq > 0.0 && *a <= 1.7976931348623157e308;
}
// One step of the conjugate gradients: with a = *rz / sc->dot_b, dy += a p,
// rho -= a q (nothing unless cg_step_length), and the largest magnitudes of dy
// and rho to sc->dynorm and sc->rho_norm.
struct CgStep {
  const double* p;
  const double* q;
  double* dy;
  const double* rz;
};
// The step and rho'z (to dpart[0]) where the triangular solves do not carry them.
cudaError_t launch_cg_update(cudaStream_t st, int64_t m, const CgStep& upd, double* rho, double* part,
                             unsigned* tickets, Scalars* sc);
cudaError_t launch_cg_dot(cudaStream_t st, int64_t m, const double* a, const double* b, double* part, double* dpart,
                          unsigned* tickets, Scalars* sc);

// Blocked Cholesky in place; dinv (m) receives the reciprocals of the pivots.
template <typename T>
cudaError_t cholesky(cudaStream_t st, int64_t m, int64_t ldm, T* M, T* dinv, Scalars* sc);

// The single-launch tile Cholesky (chol_tiles.cu): 128 x 128 tiles; the task
// list comes from chol_tile_tasks (built once per m); state holds nb^2 + nb + 1
// ints (nb = chol_tile_count(m)), cleared here.
// Beyond 256 tile rows (m > 32768) the task list (~nb^3/6 tasks, built on
// the host at handle creation) grows past ~3M entries; such handles keep the
// multi-launch blocked factor.
constexpr int kTileCholMaxTiles = 256;
constexpr int kCholTile = 128;  // tile edge of the tile Cholesky and its triangular solves
int64_t chol_tile_count(int64_t m);
int chol_tiles_resident();  // resident CTAs on the current device, 0 on error
void chol_tile_tasks(int64_t m, int nproc, std::vector<int4>* out);
// Uinv receives U_l = L_ll^{-T} for every diagonal tile (nb x 128 x 128,
// row-major per tile), for trsv_blk_solve.
template <typename T>
cudaError_t cholesky_tiles(cudaStream_t st, int64_t m, int64_t ldm, T* M, T* dinv, T* Uinv, const int4* tasks,
                           int ntasks, int* state, Scalars* sc, unsigned char* planes);
// Bytes of the BF16 operand planes of the FP32 tile factor (every tile below
// the diagonal, 96 KB each).
int64_t chol_plane_bytes(int64_t m);
// The double-float tile factor of the FP64 matrix M (FP64 tier of the mixed
// forms): M's lower triangle is turned into double-float pairs in place,
// factored by the tile Cholesky on the FP32 pipes (task list as the FP32
// factor's), and turned back into the FP64 factor L and FP64 pivot
// reciprocals dinv.  A pivot that is not positive sets PDAS_ERR_NOT_SPD.
cudaError_t cholesky_tiles_df(cudaStream_t st, int64_t m, int64_t ldm, double* M, double* dinv, const int4* tasks,
                              int ntasks, int* state, Scalars* sc);
// The triangular solves with the FP32 tile factor (trsv_blk.cu): out =
// (L L')^{-1} rhs through z.  z holds the unset pattern (every bit set) in all
// entries before and after, as does *ticket zero, unless a wait gave up: then
// both have to be set again.  out must not alias rhs or z.  upd != null: rhs and
// dy first take that step (npart: 2 nb doubles).  dpart != null: the nb =
// chol_tile_count(m) parts of rhs'out.  Two launches.
cudaError_t trsv_blk_solve(cudaStream_t st, int64_t m, int64_t ldm, const float* L, const float* Uinv, double* rhs,
                           double* z, double* out, const CgStep* upd, double* dpart, double* npart, unsigned* ticket,
                           Scalars* sc);
// inv != null (launch_invert_diag64's; the FP64 tier of the mixed forms, a
// preconditioner): the diagonal blocks are applied as inverses, a shorter chain.
// Else by substitution: FP32 on pivot-scaled rows, FP64 plain (the plain FP64
// form's direct solve).  L's rows are 16-byte aligned.
template <typename T>
cudaError_t trsv_lower(cudaStream_t st, int64_t m, int64_t ldm, const T* L, const T* dinv, const T* inv,
                       const double* v, double* z, int* flags, Scalars* sc);
template <typename T>
cudaError_t trsv_upper_t(cudaStream_t st, int64_t m, int64_t ldm, const T* L, const T* dinv, const T* inv,
                         const double* z, double* y, int* flags, Scalars* sc);
// inv (round_up(m, 64) x 64) = the inverses of L's 64 x 64 diagonal blocks.
cudaError_t launch_invert_diag64(cudaStream_t st, int64_t m, int64_t ldm, const double* L, const double* dinv,
                                 double* inv, const Scalars* sc);

// sc->mnorm = max_p M[p][p] (before the factorization overwrites it).
template <typename T>
cudaError_t launch_diag_max(cudaStream_t st, int64_t m, int64_t ldm, const T* M, double* part, unsigned* tickets,
                            Scalars* sc);
// Lower triangle of M64 = A D A' in double-float on the FP32 pipes (A exact
// in FP32: float or BF16 storage); D2 (n float2) receives D as hi + lo.
template <typename T>
cudaError_t launch_syrk_df(cudaStream_t st, int64_t m, int64_t n, const T* A, const double* D, float2* D2,
                           double* M64, int64_t ldm, const Scalars* sc);

// Akept (m x k, row-major) = the columns idx[0..k) of A; Dkept = D[idx].
template <typename T>
cudaError_t launch_gather_columns(cudaStream_t st, int64_t m, int64_t n, const T* A, const double* D, int64_t k,
                                  const int* idx, T* Akept, double* Dkept);

// Adjoint helpers: u = D .* g;  lb = D .* (w - g);  dA = -(la x' + y lb').
// out_p = (A D A')_pp without forming the matrix (m outputs).
template <typename T>
cudaError_t launch_normal_diag(cudaStream_t st, int64_t m, int64_t n, const T* A, const double* D, double* out,
                               const Scalars* sc);
cudaError_t launch_scale_vec(cudaStream_t st, int64_t n, const double* D, const double* g, double* u,
                             const Scalars* sc);
cudaError_t launch_adjoint_lb(cudaStream_t st, int64_t n, const double* D, const double* w, const double* g,
                              double* lb, const Scalars* sc);
// Refinement of the full adjoint system (see pdas_backward):
//   init:   lb = D (w - g), lc = -lb / x, wt = w
//   resid:  r1 = g - wt - s.*lc, r3 = -lb - x.*lc, t = D r1 - r3 - lb
//   update: db = D (w - r1) + r3, dc = (r3 - db) / x; lb += db, lc += dc, wt += w
cudaError_t launch_adjoint_init(cudaStream_t st, int64_t n, const double* D, const double* w, const double* g,
                                const double* x, double* lb, double* lc, double* wt, const Scalars* sc);
cudaError_t launch_adjoint_resid(cudaStream_t st, int64_t n, const double* D, const double* g, const double* x,
                                 const double* s, const double* wt, const double* lb, const double* lc, double* r1,
                                 double* r3, double* t, const Scalars* sc);
cudaError_t launch_adjoint_update(cudaStream_t st, int64_t n, const double* D, const double* w, const double* x,
                                  const double* r1, const double* r3, double* lb, double* lc, double* wt,
                                  const Scalars* sc);
cudaError_t launch_adjoint_dA(cudaStream_t st, int64_t m, int64_t n, const double* la, const double* x,
                              const double* y, const double* lb, double* dA, const Scalars* sc);

// The lower triangle of M kept in its upper one (the diagonal in diag, m
// doubles), or put back from there.
cudaError_t launch_mirror_lower(cudaStream_t st, int64_t m, int64_t ldm, double* M, double* diag, bool put_back);

cudaError_t launch_convert_matrix(cudaStream_t st, int64_t m, int64_t ld_src, const void* src, int src_f64,
                                  int64_t ld_dst, void* dst, int dst_f64);

}  // namespace pdas
