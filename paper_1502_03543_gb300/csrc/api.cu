// api.cu -- the C ABI of libpdas (include/pdas.h, include/pdas_components.h):
// handle life cycle, the per-iteration orchestration of the Newton-direction
// solve (Eq. 3 via Eq. 4, Section V), the psi ratio test and the step of the
// algorithm in Section III, and pdas_solve's outer loop.
//
// One iteration on the handle's stream (FP64 form):
//   scaling D = x/s -> r = A x -> M = A D A' (lower) -> Cholesky -> L z = r ->
//   L' dy = z -> w = A' dy, ds = -w, dx = D w - x -> psi, theta -> step, gap.
// Mixed forms replace the SYRK and Cholesky by their low-precision versions
// and refine dy in FP64 (refine()): the residual A x - A(D(A' dy)) is formed
// matrix-free in FP64 and corrected with the low-precision factor, as plain
// iterative refinement and, when that stalls, as conjugate gradients
// preconditioned by the same factor.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <type_traits>
#include <vector>

#include "pdas_internal.cuh"
#include "chol_dig.cuh"
#include "passes.cuh"
#include "syrk_dig.cuh"
#include "syrk_simt.cuh"
#include "syrk_tc.cuh"

using namespace pdas;

struct pdas_ctx {
  std::vector<void*> allocs;  // every device allocation of the handle itself
  int64_t m = 0, n = 0, ldm = 0;
  pdas_options opt{};
  cudaStream_t st = nullptr;
  // FP64 vectors
  double *D = nullptr, *r = nullptr, *dy = nullptr, *dx = nullptr, *ds = nullptr, *w = nullptr, *u = nullptr;
  double *z = nullptr, *rho = nullptr, *delta = nullptr, *kp = nullptr, *kq = nullptr, *kz = nullptr;
  double* kp2 = nullptr;      // the search direction of every other step
  double* zb = nullptr;       // hand-off of the blocked FP32 solves (all unset between them)
  bool solve_dirty = false;   // a call failed: zb and the tickets have to be set again
  double* rd = nullptr;       // infeasible-start variant: dual residual c - A'y - s (n)
  double* part = nullptr;     // reduction partials (kPartMax)
  double* gt_part = nullptr;  // partial column sums of A'u
  unsigned* ctickets = nullptr;  // ... and its column blocks' tickets, zero between launches
  unsigned* tickets = nullptr;
  int* flags = nullptr;
  Scalars* sc = nullptr;
  Scalars* sc_host = nullptr;  // pinned; written by the device (read_scalars)
  unsigned* sc_seq = nullptr;  // ... and the number of the snapshot in it
  unsigned seq = 0;            // number of the last snapshot asked for
  int wait_us = 0;             // limit of the bounded inter-block waits (0: the 2 s default)
  int* wait_pinned = nullptr;  // pinned copy of wait_us, the source of its copy into sc
  double* M64 = nullptr;      // FP64 form; mixed forms: the FP64 tier's matrix (allocated at create)
  float* M32 = nullptr;
  double* dinv64 = nullptr;  // reciprocals of the pivots of the FP64 / FP32 factor
  double* inv64 = nullptr;   // inverses of the FP64 factor's 64 x 64 diagonal blocks (mixed forms)
  float* dinv32 = nullptr;
  void* simt_part = nullptr;        // SIMT normal matrices: partial tiles of their K slices
  unsigned* simt_tickets = nullptr;  // one per tile, zero between launches
  float* simt_planes = nullptr;      // FP32_IR: operand planes of the normal matrix
  TcWorkspace tc{};
  DigWorkspace dig{};  // FP64 tier on the tensor cores (BF16 A): digit planes
  CholDigWorkspace cdig{};  // FP64 tier: the factor's trailing updates on the tensor cores
  int cur_f64 = 1;     // the workspace matrix in use is M64
  int refactored = 0;  // a mixed form switched to FP64 for good
  // column dropping for the FP64 factor of the mixed forms
  void* akept = nullptr;        // m x n elements of A's dtype (mixed forms with drop_tol > 0)
  double* dkept = nullptr;      // n
  int* kidx = nullptr;          // n
  std::vector<double> dhost;
  std::vector<int> idx_host;
  int64_t last_kept = 0;        // columns in the last FP64 factor of a mixed form
  bool no_drop_once = false;    // the dropped factor failed: use every column this time
  bool no_df_once = false;      // the double-float factor failed: form in FP64 this time
  float2* d2 = nullptr;         // D as FP32 pairs (double-float formation)
  int last_normal_form = 3;     // pdas_iter_info.normal_form of the last formation
  int last_factor_form = 3;     // pdas_iter_info.factor_form of the last factor
  bool have_factor = false;     // a factor from a previous step is in the workspace
  double* adj = nullptr;        // adjoint vectors (5 n + m)
  int4* chol_tasks = nullptr;   // task list of the tile Cholesky (FP32 factor)
  int chol_ntasks = 0;
  int* chol_state = nullptr;    // counters of the tile Cholesky: per tile, then panels per diagonal tile
  float* uinv32 = nullptr;      // L_ll^{-T} of every diagonal tile of the FP32 tile factor
  unsigned char* chol_planes = nullptr;  // BF16 operand planes of the tile factor's off-diagonal tiles
  float* pairs = nullptr;       // the vector of a double-float pass as FP32 pairs (n, two planes)
  int switch_reason = 0;  // pdas_iter_info.fp64_reason of that switch
  bool last_factor_df = false;    // the last factor was a fast FP64-tier factor (tensor-core or double-float)
  double last_rel_gap = HUGE_VAL;  // relative gap of the iterate after the last step
  bool plain_simt = false;        // plain FP64 form: this call is a retry with the SIMT factor
  bool no_dffactor_once = false;  // this iteration: that factor failed, use the FP64 factor
  int64_t err_index = -1;
  char errmsg[256] = {0};
  // diagnostics of the last direction
  int last_sweeps = 0;
  double last_resid = 0.0;
  int last_fp64 = 0;
  // profiling: event pairs around stages, and the kernel-launch count
  bool prof = false;
  std::vector<cudaEvent_t> evs;
  std::vector<int> ev_stage;  // per recorded pair: stage index
  size_t ev_used = 0;
  int open_stage = -1;
  double prof_ms[PDAS_STAGE_COUNT] = {0};
  int64_t prof_calls[PDAS_STAGE_COUNT] = {0};
  int64_t launches = 0;
};

namespace {

bool is_mixed(const pdas_ctx* h) { return h->opt.form != PDAS_FP64; }

pdas_status cuda_fail(pdas_ctx* h, cudaError_t e, const char* where) {
  snprintf(h->errmsg, sizeof(h->errmsg), "%s: %s", where, cudaGetErrorString(e));
  return PDAS_ERR_CUDA;
}

#define CK(call)                                              \
  do {                                                        \
    cudaError_t e_ = (call);                                  \
    if (e_ != cudaSuccess) return cuda_fail(h, e_, #call);    \
  } while (0)

// A launch helper that starts `k` kernels: checked and counted.
#define KL(call, k)        \
  do {                     \
    CK(call);              \
    h->launches += (k);    \
  } while (0)

int64_t chol_launches(int64_t m) {
  int64_t k = 0;
  for (int64_t k0 = 0; k0 < m; k0 += kTile) k += (m - k0 - kTile > 0) ? 2 : 1;
  return k;
}

pdas_status prof_fold(pdas_ctx* h);

cudaError_t prof_record(pdas_ctx* h) {
  if (h->ev_used == h->evs.size()) {
    cudaEvent_t e;
    cudaError_t r = cudaEventCreate(&e);
    if (r != cudaSuccess) return r;
    h->evs.push_back(e);
  }
  return cudaEventRecord(h->evs[h->ev_used++], h->st);
}

pdas_status stage_begin(pdas_ctx* h, int stage) {
  if (!h->prof) return PDAS_OK;
  if (h->ev_used + 2 > 8192) {
    pdas_status s = prof_fold(h);
    if (s != PDAS_OK) return s;
  }
  CK(prof_record(h));
  h->open_stage = stage;
  return PDAS_OK;
}

pdas_status stage_end(pdas_ctx* h) {
  if (!h->prof || h->open_stage < 0) return PDAS_OK;
  CK(prof_record(h));
  h->ev_stage.push_back(h->open_stage);
  h->open_stage = -1;
  return PDAS_OK;
}

// Synchronise and add the recorded pairs to the accumulators.
pdas_status prof_fold(pdas_ctx* h) {
  CK(cudaStreamSynchronize(h->st));
  for (size_t i = 0; i < h->ev_stage.size(); ++i) {
    float ms = 0.f;
    CK(cudaEventElapsedTime(&ms, h->evs[2 * i], h->evs[2 * i + 1]));
    h->prof_ms[h->ev_stage[i]] += ms;
    h->prof_calls[h->ev_stage[i]] += 1;
  }
  h->ev_stage.clear();
  h->ev_used = 0;
  h->open_stage = -1;
  return PDAS_OK;
}

#define STAGE(h, k)                               \
  do {                                            \
    pdas_status s_ = stage_begin((h), (k));       \
    if (s_ != PDAS_OK) return s_;                 \
  } while (0)
#define STAGE_END(h)                              \
  do {                                            \
    pdas_status s_ = stage_end(h);                \
    if (s_ != PDAS_OK) return s_;                 \
  } while (0)

template <typename F>
pdas_status with_dtype(int dt, F&& f) {
  switch (dt) {
    case PDAS_A_F64: return f((const double*)nullptr);
    case PDAS_A_F32: return f((const float*)nullptr);
    case PDAS_A_BF16: return f((const __nv_bfloat16*)nullptr);
  }
  return PDAS_ERR_ARG;
}

// Reads the device scalars: a one-warp launch writes them to pinned host memory,
// then the snapshot's number, for which the host polls.  A copy and a stream
// synchronisation take 12-15 us from the last kernel's end to the next launch
// (two to five times per direction), this about 7 (512 x 2048: 499 -> 475 us
// a direction).  Nothing is left running: the snapshot is the stream's last launch.
pdas_status read_scalars(pdas_ctx* h) {
  const unsigned want = ++h->seq;
  KL(launch_snapshot(h->st, h->sc, h->sc_host, h->sc_seq, want), 1);
  for (unsigned spin = 1;; ++spin) {
    if (__atomic_load_n(h->sc_seq, __ATOMIC_ACQUIRE) == want) return PDAS_OK;
    if ((spin & 0xfff) == 0) {  // an error on the stream (or a capture) never writes it
      const cudaError_t e = cudaStreamQuery(h->st);
      if (e == cudaErrorNotReady) continue;
      CK(e);
      if (__atomic_load_n(h->sc_seq, __ATOMIC_ACQUIRE) == want) return PDAS_OK;
      CK(cudaStreamSynchronize(h->st));
      if (__atomic_load_n(h->sc_seq, __ATOMIC_ACQUIRE) == want) return PDAS_OK;
      return cuda_fail(h, cudaErrorUnknown, "scalars not written");
    }
  }
}

pdas_status device_status(pdas_ctx* h) {
  const Scalars& s = *h->sc_host;
  if (s.status != 0) h->solve_dirty = true;  // launches may have stopped between a ticket and its reset
  if (s.status == PDAS_ERR_NOT_SPD) h->err_index = s.fail_index;
  return (pdas_status)s.status;
}

pdas_status reset_status(pdas_ctx* h) {
  CK(cudaMemsetAsync(h->sc, 0, sizeof(Scalars), h->st));
  if (h->solve_dirty) {
    CK(cudaMemsetAsync(h->tickets, 0, sizeof(unsigned) * T_COUNT, h->st));
    if (h->zb) CK(cudaMemsetAsync(h->zb, 0xff, sizeof(double) * h->m, h->st));
    h->solve_dirty = false;
  }
  if (h->wait_us > 0)  // a limit of the handle's own (pdas_set_wait_limit)
    CK(cudaMemcpyAsync(&h->sc->wait_us, h->wait_pinned, sizeof(int), cudaMemcpyHostToDevice, h->st));
  return PDAS_OK;
}

// A v -> out (base == null) or base - A v -> out; norm_slot as in launch_pass.
// Double-float passes over A (passes.cu) are available to the mixed forms
// when A is exact in FP32 (stored as FP32 or BF16) and exact_passes is off.
// The solve uses them only for the conjugate-gradient operator M p of the
// refinement while it factors in FP32: every quantity the acceptance test or
// the direction depends on
// (r = A x, the true residual r - A(D(A' dy)), w = A' dy) stays FP64, since
// the double-float rounding of a residual is close to the 1e-14 acceptance
// level, while in M p it scales with the search direction and only slows
// the iteration by rounding.  The component entry points pdas_gemv /
// pdas_gemv_t of a mixed handle expose the double-float pass itself.
bool df_passes(const pdas_ctx* h) { return is_mixed(h) && h->opt.a_dtype != PDAS_A_F64 && !h->opt.exact_passes; }

// df: h->pairs holds the FP32 pairs of v, or (v given) receives them first.
// dot: also sum_p dot_p out_p into sc->dot_b.
pdas_status gemv(pdas_ctx* h, const void* A, const double* v, const double* base, double* out, int norm_slot,
                 bool df = false, const double* dot = nullptr) {
  if (df && v) KL(launch_split_pairs(h->st, h->n, v, h->pairs), 1);
  return with_dtype(h->opt.a_dtype, [&](auto tag) -> pdas_status {
    using T = std::remove_const_t<std::remove_pointer_t<decltype(tag)>>;
    KL(launch_pass<T>(h->st, h->m, h->n, (const T*)A, v, df ? h->pairs : nullptr, base, out, h->part, h->tickets,
                      h->sc, norm_slot, dot), 1);
    return PDAS_OK;
  });
}

// w = A'(src), then the mode of launch_pass_t; pairs: the FP32 pairs of D w to
// h->pairs (mode 2).
pdas_status gemv_t(pdas_ctx* h, const void* A, const PassTSrc& src, int mode, const double* x, double* o0, double* o1,
                   double* o2, bool df = false, const double* rd = nullptr, bool pairs = false) {
  return with_dtype(h->opt.a_dtype, [&](auto tag) -> pdas_status {
    using T = std::remove_const_t<std::remove_pointer_t<decltype(tag)>>;
    KL(launch_pass_t<T>(h->st, h->m, h->n, (const T*)A, df, src, h->gt_part, h->part + 3 * kPartMax, h->ctickets, mode,
                        x, h->D, o0, o1, o2, pairs ? h->pairs : nullptr, h->sc, rd), 1);
    return PDAS_OK;
  });
}
pdas_status gemv_t(pdas_ctx* h, const void* A, const double* u, int mode, const double* x, double* o0, double* o1,
                   double* o2, bool df = false, const double* rd = nullptr) {
  PassTSrc src;
  src.u = u;
  return gemv_t(h, A, src, mode, x, o0, o1, o2, df, rd);
}

bool want_fp64(const pdas_ctx* h) { return !is_mixed(h) || h->refactored; }

size_t dtype_size(int dt) { return dt == PDAS_A_F64 ? 8 : dt == PDAS_A_F32 ? 4 : 2; }

// Columns for the FP64 factor of a mixed form: those with D_j >= drop_tol
// max D, at least drop_keep m of them (the largest D_j).  Returns the count
// (n = keep all; then idx is not built).
pdas_status select_columns(pdas_ctx* h, int64_t* kept) {
  const int64_t n = h->n;
  *kept = n;
  if (!(h->opt.drop_tol > 0) || h->no_drop_once) return PDAS_OK;
  h->dhost.resize(n);
  CK(cudaMemcpyAsync(h->dhost.data(), h->D, sizeof(double) * n, cudaMemcpyDeviceToHost, h->st));
  CK(cudaStreamSynchronize(h->st));
  double dmax = 0.0;
  for (double d : h->dhost) dmax = std::max(dmax, d);
  double t = h->opt.drop_tol * dmax;
  int64_t count = 0;
  for (double d : h->dhost) count += d >= t;
  int64_t kmin = (int64_t)std::ceil(h->opt.drop_keep * (double)h->m);
  kmin = std::min(std::max<int64_t>(kmin, h->m), n);
  if (count < kmin) {  // lower the threshold to the kmin-th largest D
    std::vector<double> tmp(h->dhost);
    std::nth_element(tmp.begin(), tmp.begin() + (kmin - 1), tmp.end(), std::greater<double>());
    t = tmp[kmin - 1];
  }
  h->idx_host.clear();
  for (int64_t j = 0; j < n; ++j)
    if (h->dhost[j] >= t) h->idx_host.push_back((int)j);
  const int64_t k = (int64_t)h->idx_host.size();
  if (k >= n) return PDAS_OK;
  CK(cudaMemcpyAsync(h->kidx, h->idx_host.data(), sizeof(int) * k, cudaMemcpyHostToDevice, h->st));
  *kept = k;
  return PDAS_OK;
}

// a3: the normal matrix in the current precision.
pdas_status form_normal(pdas_ctx* h, const void* A) {
  if (want_fp64(h)) {
    pdas_status s;
    h->cur_f64 = 1;
    int64_t kept = h->n;
    if (is_mixed(h) && (s = select_columns(h, &kept)) != PDAS_OK) return s;
    h->last_kept = kept;
    // A mixed form whose A is exact in FP32 forms this matrix in double-float
    // on the FP32 pipes (FP64 remains the fallback when that factor fails).
    const bool df = is_mixed(h) && h->opt.a_dtype != PDAS_A_F64 && !h->no_df_once;
    // ... and, for BF16 A, on the tensor cores from exact fixed-point digit
    // planes (FP64-grade), when the kept columns fit the digit workspace
    const bool dig = df && h->opt.a_dtype == PDAS_A_BF16 && h->dig.planes && kept <= h->dig.kstride;
    h->last_normal_form = dig ? 4 : df ? 2 : 3;
    if (dig) {
      int kl = 0;
      CK(dig_syrk(h->st, &h->dig, (const __nv_bfloat16*)A, h->n, h->D, kept, kept < h->n ? h->kidx : nullptr,
                  h->M64, h->ldm, h->sc, &kl));
      h->launches += kl;
      return PDAS_OK;
    }
    return with_dtype(h->opt.a_dtype, [&](auto tag) -> pdas_status {
      using T = std::remove_const_t<std::remove_pointer_t<decltype(tag)>>;
      const T* Aop = (const T*)A;
      const double* Dop = h->D;
      int64_t cols = h->n;
      if (kept < h->n) {
        KL(launch_gather_columns<T>(h->st, h->m, h->n, (const T*)A, h->D, kept, h->kidx, (T*)h->akept, h->dkept), 1);
        Aop = (const T*)h->akept;
        Dop = h->dkept;
        cols = kept;
      }
      if constexpr (std::is_same<T, double>::value) {
        KL(launch_syrk_fp64<T>(h->st, h->m, cols, Aop, Dop, h->M64, h->ldm, h->simt_part, h->simt_tickets, h->sc), 1);
      } else {
        if (df) KL(launch_syrk_df<T>(h->st, h->m, cols, Aop, Dop, h->d2, h->M64, h->ldm, h->sc), 2);
        else KL(launch_syrk_fp64<T>(h->st, h->m, cols, Aop, Dop, h->M64, h->ldm, h->simt_part, h->simt_tickets, h->sc), 1);
      }
      return PDAS_OK;
    });
  }
  h->cur_f64 = 0;
  h->last_normal_form = h->opt.form == PDAS_FP32_IR ? 1 : 0;
  if (h->opt.form == PDAS_FP32_IR) {
    return with_dtype(h->opt.a_dtype, [&](auto tag) -> pdas_status {
      using T = std::remove_const_t<std::remove_pointer_t<decltype(tag)>>;
      int kl = 0;
      CK(launch_syrk_fp32<T>(h->st, h->m, h->n, (const T*)A, h->D, h->simt_planes, h->M32, h->ldm, h->simt_part,
                             h->simt_tickets, h->sc, &kl));
      h->launches += kl;
      return PDAS_OK;
    });
  }
  int k = 0;
  if (h->prof && h->open_stage >= 0) h->open_stage = PDAS_STAGE_FOLD;  // the open interval starts the fold
  CK(tc_prepare(h->st, &h->tc, A, h->D, &k));
  h->launches += k;
  STAGE_END(h);
  STAGE(h, PDAS_STAGE_NORMAL);
  CK(tc_syrk(h->st, &h->tc, A, h->M32, h->ldm, h->sc, &k));
  h->launches += k;
  return PDAS_OK;
}

// The FP64 tier of a mixed form factors with the double-float tile factor
// (~3.5x faster than the FP64 factor on GB300's FP64 pipes) while the
// relative gap of the iterate exceeds opt.df_factor_floor, and with the FP64
// factor below it.  In the last iterations the forward error of the refined
// direction sets the gap that can be reached (the refinement accepts on a
// backward-error test), and a slightly different preconditioner there moved
// the gap-1e-8 run of the 8192 x 32768 problem from 54 iterations to 80.
pdas_status factor(pdas_ctx* h) {
  h->last_factor_df = false;
  if (h->cur_f64 && h->cdig.m > 0 && !h->no_dffactor_once) {
    // The plain FP64 form and the FP64 tier with fp64_tier_tc: the FP64 factor whose trailing updates run
    // on the tensor cores from exact digit planes (FP64-grade at every gap);
    // on a failed pivot the next attempt uses the FP64 SIMT factor
    h->last_factor_df = true;
    h->last_factor_form = 4;
    int k = 0;
    CK(cholesky_dig(h->st, &h->cdig, h->ldm, h->M64, h->dinv64, h->sc, &k));
    h->launches += k;
  } else if (h->cur_f64 && is_mixed(h) && h->chol_ntasks > 0 && !h->no_dffactor_once &&
      h->last_rel_gap > h->opt.df_factor_floor) {
    // FP64 tier of a mixed form: the double-float tile factor (FP32 pipes),
    // while the iterate is not yet close to the optimum
    h->last_factor_df = true;
    h->last_factor_form = 2;
    KL(cholesky_tiles_df(h->st, h->m, h->ldm, h->M64, h->dinv64, h->chol_tasks, h->chol_ntasks, h->chol_state, h->sc),
       4);
  } else if (h->cur_f64) {
    h->last_factor_form = 3;
    KL(cholesky<double>(h->st, h->m, h->ldm, h->M64, h->dinv64, h->sc), chol_launches(h->m));
  } else if (h->chol_ntasks == 0) {
    h->last_factor_form = 1;
    KL(cholesky<float>(h->st, h->m, h->ldm, h->M32, h->dinv32, h->sc), chol_launches(h->m));
  } else {
    h->last_factor_form = 0;
    KL(cholesky_tiles<float>(h->st, h->m, h->ldm, h->M32, h->dinv32, h->uinv32, h->chol_tasks, h->chol_ntasks,
                             h->chol_state, h->sc, h->chol_planes),
       1);
  }
  if (h->cur_f64 && h->inv64)
    KL(launch_invert_diag64(h->st, h->m, h->ldm, h->M64, h->dinv64, h->inv64, h->sc), 1);
  return PDAS_OK;
}

// out = (L L')^{-1} rhs with the current factor.  upd: first that step of the
// conjugate gradients on rhs = h->rho; *nrz: then rhs'out as *nrz parts at
// rz_part(h).
double* rz_part(pdas_ctx* h) { return h->part + 2 * kPartMax; }

pdas_status factor_solve(pdas_ctx* h, double* rhs, double* out, const CgStep* upd = nullptr, int* nrz = nullptr) {
  if (!h->cur_f64 && h->chol_ntasks > 0) {  // the tile factor, with the inverses of its diagonal tiles
    KL(trsv_blk_solve(h->st, h->m, h->ldm, h->M32, h->uinv32, rhs, h->zb, out, upd, nrz ? rz_part(h) : nullptr,
                      h->part, h->tickets + T_TRSVB, h->sc),
       2);
    if (nrz) *nrz = (int)chol_tile_count(h->m);
    return PDAS_OK;
  }
  if (upd) KL(launch_cg_update(h->st, h->m, *upd, rhs, h->part, h->tickets, h->sc), 1);
  if (h->cur_f64) {
    KL(trsv_lower<double>(h->st, h->m, h->ldm, h->M64, h->dinv64, h->inv64, rhs, h->z, h->flags, h->sc), 1);
    KL(trsv_upper_t<double>(h->st, h->m, h->ldm, h->M64, h->dinv64, h->inv64, h->z, out, h->flags, h->sc), 1);
  } else {
    KL(trsv_lower<float>(h->st, h->m, h->ldm, h->M32, h->dinv32, nullptr, rhs, h->z, h->flags, h->sc), 1);
    KL(trsv_upper_t<float>(h->st, h->m, h->ldm, h->M32, h->dinv32, nullptr, h->z, out, h->flags, h->sc), 1);
  }
  if (nrz) {
    KL(launch_cg_dot(h->st, h->m, rhs, out, h->part, rz_part(h), h->tickets, h->sc), 1);
    *nrz = 1;
  }
  return PDAS_OK;
}

// FP64 refinement of dy for the mixed forms (a6): conjugate gradients on
// M dy = r with the factor as preconditioner, started from dy = (L L')^{-1} r.
// M is applied matrix-free in FP64 (A(D(A' v))), so the result is as
// accurate as FP64 arithmetic allows whatever the precision of the factor.
// The recurrence residual is confirmed against the true residual r - M dy
// before acceptance and every 10 steps (and replaces it when they differ).
// Accepted when ||r - M dy||_inf <= refine_tol ||r||_inf, or when the
// normwise backward error ||r - M dy||_inf / (max_p M_pp ||dy||_inf +
// ||r||_inf) <= refine_be.  On return h->w = A' dy of the final dy;
// *ok = 0 if neither test passed within refine_max steps.  A step that
// cg_step_length refuses is not taken and ends the refinement.  A step is four
// launches (p and u = D A'p; q = A u and p'q; the two triangular solves, which
// carry the updates and rho'z) and one read of the scalars.  The first read
// also brings the factor's status (PDAS_ERR_NOT_SPD).
pdas_status refine(pdas_ctx* h, const void* A, int* ok) {
  *ok = 0;
  const double tol = h->opt.refine_tol, be_tol = h->opt.refine_be;
  const int cap = h->opt.refine_max;
  pdas_status s;
  // With an FP32 factor the first residual is ~1e-7 of r and starts the
  // conjugate gradients: the double-float passes form it (two FP64 passes
  // saved per direction); a first residual that would be accepted is formed
  // again by the FP64 passes.
  const bool cheap_first = df_passes(h) && !h->cur_f64;
  // The operator: not in double-float once the solve has switched to an FP64
  // factor (there the FP64 factor dominates the iteration, and near the end
  // the operator's rounding decides whether the refinement still reaches its
  // tolerance).
  const bool df_op = df_passes(h) && !h->refactored;
  // rho = r - A(D(A' dy)), ||rho||, ||dy||, w = A'dy; df: by the double-float
  // passes, for a residual that only starts the conjugate gradients
  auto true_residual = [&](bool df = false) -> pdas_status {
    PassTSrc src;
    src.u = h->dy;
    src.absmax = 1;
    pdas_status t = gemv_t(h, A, src, 2, nullptr, df ? nullptr : h->u, nullptr, h->w, df, nullptr, df);
    if (t == PDAS_OK) t = gemv(h, A, df ? nullptr : h->u, h->r, h->rho, 1, df);
    if (t != PDAS_OK) return t;
    if ((t = read_scalars(h)) != PDAS_OK) return t;
    return device_status(h);
  };
  if ((s = true_residual(cheap_first)) != PDAS_OK) return s;
  const double rn = h->sc_host->rnorm > 0 ? h->sc_host->rnorm : 1.0;
  const double mn = h->sc_host->mnorm;
  auto accepted = [&](double res, double dyn) { return res <= tol * rn || res <= be_tol * (mn * dyn + rn); };
  double res = h->sc_host->rho_norm, dyn = h->sc_host->dynorm;
  if (cheap_first && accepted(res, dyn)) {  // acceptance is decided on the FP64 passes
    if ((s = true_residual()) != PDAS_OK) return s;
    res = h->sc_host->rho_norm;
    dyn = h->sc_host->dynorm;
  }
  int its = 0;
  if (accepted(res, dyn)) {
    *ok = 1;
  } else {
    double *p = h->kp, *pn = h->kp2;
    bool first = true;  // p = z = P^{-1} rho, no direction before it
    bool stale = false;  // dy has moved since the last true residual
    int nrz = 0;
    if (cap > 0 && (s = factor_solve(h, h->rho, h->kz, nullptr, &nrz)) != PDAS_OK) return s;
    while (its < cap) {
      PassTSrc src;
      src.u = h->kz;
      src.p = p;
      src.p_new = pn;
      src.rz_part = rz_part(h);
      src.nrz = nrz;
      src.par = its & 1;
      src.first = first;
      if ((s = gemv_t(h, A, src, 2, nullptr, df_op ? nullptr : h->u, nullptr, nullptr, df_op, nullptr, df_op)) != PDAS_OK)
        return s;
      if ((s = gemv(h, A, df_op ? nullptr : h->u, nullptr, h->kq, -1, df_op, pn)) != PDAS_OK) return s;  // q = M p
      const CgStep upd{pn, h->kq, h->dy, &h->sc->rz[src.par]};
      if ((s = factor_solve(h, h->rho, h->kz, &upd, &nrz)) != PDAS_OK) return s;
      std::swap(p, pn);
      first = false;
      if ((s = read_scalars(h)) != PDAS_OK) return s;
      if ((s = device_status(h)) != PDAS_OK) return s;
      double a;
      if (!cg_step_length(h->sc_host->rz[src.par], h->sc_host->dot_b, &a)) break;  // (nothing was updated)
      ++its;
      stale = true;
      res = h->sc_host->rho_norm;
      dyn = h->sc_host->dynorm;
      if (accepted(res, dyn) || its % 10 == 0 || its == cap) {
        if ((s = true_residual()) != PDAS_OK) return s;
        stale = false;
        res = h->sc_host->rho_norm;
        dyn = h->sc_host->dynorm;
        if (accepted(res, dyn)) {
          *ok = 1;
          break;
        }
        if (its < cap && (s = factor_solve(h, h->rho, h->kz, nullptr, &nrz)) != PDAS_OK) return s;
        first = true;
      }
    }
    if (stale) {  // the steps ended in between: w and the residual of this dy
      if ((s = true_residual()) != PDAS_OK) return s;
      res = h->sc_host->rho_norm;
      dyn = h->sc_host->dynorm;
      *ok = accepted(res, dyn);
    }
  }
  h->last_sweeps = its;
  h->last_resid = res / rn;
  return PDAS_OK;
}

// The right-hand side of the normal equations at (x, s): D = x/s, then
// r = A x (a2; the paper's system, which assumes A x = b and A'y + s = c),
// or, for the infeasible-start variant (iv != null: y, b, c), the dual
// residual rd = c - A'y - s and r = b + A D rd.
struct Infeasible {
  const double *y, *b, *c;
};
pdas_status normal_rhs(pdas_ctx* h, const void* A, const double* x, const double* s, const Infeasible* iv) {
  pdas_status st;
  KL(launch_scaling(h->st, h->n, x, s, h->D, h->part, h->tickets, h->sc), 1);
  if (!iv) return gemv(h, A, x, nullptr, h->r, 0);  // r = A x
  if ((st = gemv_t(h, A, iv->y, 0, nullptr, h->w, nullptr, nullptr)) != PDAS_OK) return st;  // w = A'y
  KL(launch_dual_residual(h->st, h->n, iv->c, s, h->w, h->D, h->rd, h->u, h->sc), 1);     // rd, u = -D rd
  return gemv(h, A, h->u, iv->b, h->r, 0);                                                // r = b - A u
}

// One Newton direction at (x, s): fills h->D, h->r, h->dy, h->dx, h->ds (and
// h->rd for the infeasible-start variant, iv != null).
pdas_status direction(pdas_ctx* h, const void* A, const double* x, const double* s, const Infeasible* iv = nullptr) {
  pdas_status st;
  if ((st = reset_status(h)) != PDAS_OK) return st;
  const double* rd = iv ? h->rd : nullptr;
  STAGE(h, PDAS_STAGE_RHS);
  if ((st = normal_rhs(h, A, x, s, iv)) != PDAS_OK) return st;
  STAGE_END(h);
  if (is_mixed(h) && !h->refactored && h->opt.dspread_refactor > 0) {
    if ((st = read_scalars(h)) != PDAS_OK) return st;
    if ((st = device_status(h)) != PDAS_OK) return st;
    if (h->sc_host->dmax / h->sc_host->dmin > h->opt.dspread_refactor) {
      h->refactored = 1;
      h->switch_reason = 1;
    }
  }
  h->no_drop_once = false;
  h->no_df_once = false;
  h->no_dffactor_once = h->plain_simt;
  for (int attempt = 0; attempt < 5; ++attempt) {
    STAGE(h, PDAS_STAGE_NORMAL);
    if ((st = form_normal(h, A)) != PDAS_OK) return st;
    STAGE_END(h);
    if (is_mixed(h)) {  // max_p M_pp for the backward-error test of the refinement
      if (h->cur_f64) KL(launch_diag_max<double>(h->st, h->m, h->ldm, h->M64, h->part, h->tickets, h->sc), 1);
      else KL(launch_diag_max<float>(h->st, h->m, h->ldm, h->M32, h->part, h->tickets, h->sc), 1);
    }
    STAGE(h, PDAS_STAGE_FACTOR);
    if ((st = factor(h)) != PDAS_OK) return st;
    STAGE_END(h);
    h->have_factor = true;  // (a failed factor is reported below and retried)
    STAGE(h, PDAS_STAGE_SOLVE);
    if ((st = factor_solve(h, h->r, h->dy)) != PDAS_OK) return st;
    h->last_fp64 = h->cur_f64;
    if (!is_mixed(h)) {  // the plain FP64 form: the direct solve of Section V-A, unrefined
      STAGE_END(h);
      h->last_sweeps = 0;
      h->last_resid = 0.0;
      STAGE(h, PDAS_STAGE_DIR);
      if ((st = gemv_t(h, A, h->dy, 1, x, h->dx, h->ds, nullptr, false, rd)) != PDAS_OK) return st;  // a7
      STAGE_END(h);
      return PDAS_OK;
    }
    int ok = 0;
    st = refine(h, A, &ok);  // (its first read brings the factor's status)
    if (st == PDAS_ERR_NOT_SPD) {  // low-precision factor broke down: FP64 from now on
      STAGE_END(h);
      if (h->cur_f64) {
        if (h->last_factor_df) h->no_dffactor_once = true;        // the FP64 factor next
        else if (h->last_normal_form == 2 || h->last_normal_form == 4) h->no_df_once = true;  // form it in FP64 next
        else if (h->last_kept < h->n) h->no_drop_once = true;      // then from every column
        else return st;                                            // the whole FP64 matrix is not SPD
      }
      if (!h->refactored) h->switch_reason = 2;
      h->refactored = 1;
      if ((st = reset_status(h)) != PDAS_OK) return st;
      if ((st = normal_rhs(h, A, x, s, iv)) != PDAS_OK) return st;
      continue;
    }
    if (st != PDAS_OK) return st;
    STAGE_END(h);
    if (ok || h->cur_f64) {
      // w = A' dy of the accepted dy is in h->w: dx = D w - x, ds = -w.  (An
      // FP64 factor is the last tier: its refined direction is used as is.)
      STAGE(h, PDAS_STAGE_DIR);
      KL(launch_direction(h->st, h->n, h->w, x, h->D, h->dx, h->ds, h->sc, rd), 1);
      STAGE_END(h);
      return PDAS_OK;
    }
    h->refactored = 1;  // refinement failed: re-form and re-factor in FP64
    h->switch_reason = 3;
  }
  return PDAS_ERR_NOT_SPD;
}

pdas_status check_vec_args(const void* A, const double* x, const double* s) {
  if (!A || !x || !s) return PDAS_ERR_ARG;
  return PDAS_OK;
}

void fill_info(pdas_ctx* h, pdas_iter_info* info, bool stepped) {
  if (!info) return;
  const Scalars& s = *h->sc_host;
  memset(info, 0, sizeof(*info));
  info->dmax = s.dmax;
  info->dmin = s.dmin;
  info->refine_sweeps = h->last_sweeps;
  info->refine_resid = h->last_resid;
  info->used_fp64 = h->last_fp64;
  info->fp64_reason = (h->last_fp64 && is_mixed(h)) ? h->switch_reason : 0;
  info->factor_columns = (h->last_fp64 && is_mixed(h)) ? h->last_kept : h->n;
  info->normal_form = h->last_normal_form;
  info->factor_form = h->last_factor_form;
  if (stepped) {
    info->psi = s.psi;
    info->theta = s.theta;
    info->rel_gap = s.rel_gap;
    info->cx = s.cx;
    info->by = s.by;
    info->xs = s.xs;
    if (h->opt.infeasible) {
      info->pres = s.pres;
      info->dres = s.dres;
    }
  }
}

// The plain FP64 form reads the device's status only at the end of a call:
// where the factor with tensor-core updates met a pivot that is not positive,
// the call is done over with the SIMT factor (nothing of the caller's has been
// touched), so that a matrix at the edge is judged as by that factor.
bool retry_simt(pdas_ctx* h, pdas_status st) {
  if (st != PDAS_ERR_NOT_SPD || is_mixed(h) || h->last_factor_form != 4) return false;
  h->plain_simt = true;
  return true;
}
// The end of a call that may have been done over: the next one starts with the
// tensor-core factor again.
void end_retry(pdas_ctx* h) {
  if (h->plain_simt) h->no_dffactor_once = false;
  h->plain_simt = false;
}

// One step in place, up to the device's status; *read: it was read.
pdas_status step_once(pdas_ctx* h, const void* A, const double* b, const double* c, double* x, double* y, double* s,
                      double alpha, const Infeasible* iv, bool* read) {
  *read = false;
  pdas_status st = direction(h, A, x, s, iv);
  if (st != PDAS_OK) return st;
  STAGE(h, PDAS_STAGE_STEP);
  KL(launch_psi(h->st, h->n, x, s, h->dx, h->ds, alpha, h->part, h->tickets, h->sc, iv != nullptr), 1);
  KL(launch_step(h->st, h->m, h->n, b, c, x, y, s, h->dx, h->dy, h->ds, h->part, h->tickets, h->sc), 1);
  if (iv) {  // residuals of the new iterate: b - A x and c - A'y - s
    if ((st = gemv(h, A, x, b, h->rho, -1)) != PDAS_OK) return st;
    if ((st = gemv_t(h, A, y, 0, nullptr, h->w, nullptr, nullptr)) != PDAS_OK) return st;
    KL(launch_residual_norms(h->st, h->m, h->n, b, h->rho, c, h->w, s, h->part, h->tickets, h->sc), 1);
  }
  STAGE_END(h);
  if ((st = read_scalars(h)) != PDAS_OK) return st;
  *read = true;
  return device_status(h);
}

// Newton direction to the caller's arrays, synchronous.
pdas_status direction_out(pdas_ctx* h, const void* A, const double* x, const double* s, const Infeasible* iv, double* dx,
                          double* dy, double* ds, pdas_iter_info* info) {
  pdas_status st;
  do {
    h->err_index = -1;
    if ((st = direction(h, A, x, s, iv)) != PDAS_OK) break;
    CK(cudaMemcpyAsync(dx, h->dx, sizeof(double) * h->n, cudaMemcpyDeviceToDevice, h->st));
    CK(cudaMemcpyAsync(ds, h->ds, sizeof(double) * h->n, cudaMemcpyDeviceToDevice, h->st));
    CK(cudaMemcpyAsync(dy, h->dy, sizeof(double) * h->m, cudaMemcpyDeviceToDevice, h->st));
    if ((st = read_scalars(h)) != PDAS_OK) break;
    st = device_status(h);
    fill_info(h, info, false);
  } while (retry_simt(h, st));
  end_retry(h);
  return st;
}

}  // namespace

// ===========================================================================
extern "C" {

void pdas_default_options(pdas_options* opt) {
  if (!opt) return;
  memset(opt, 0, sizeof(*opt));
  opt->form = PDAS_FP64;
  opt->a_dtype = PDAS_A_F64;
  opt->max_iter = 500;
  opt->refine_tol = 1e-14;
  opt->refine_max = 40;
  opt->refine_be = 1e-14;
  opt->drop_tol = 1e-10;
  opt->drop_keep = 1.25;
  opt->exact_passes = 0;
  opt->dspread_refactor = 0.0;
  opt->stream = nullptr;
  opt->splits = 0;
  opt->stall_theta = 1e-12;
  opt->stall_count = 5;
  opt->infeasible = 0;
  opt->fp64_tier_tc = 1;
  opt->df_factor_floor = 1e-6;
}

const char* pdas_status_str(pdas_status st) {
  switch (st) {
    case PDAS_OK: return "ok";
    case PDAS_OPTIMAL: return "optimal (relative gap below tol)";
    case PDAS_OPTIMAL_EXACT: return "optimal (psi <= 1, full step)";
    case PDAS_MAX_ITER: return "iteration cap reached";
    case PDAS_STALLED: return "stalled (step lengths below stall_theta)";
    case PDAS_ZERO_DIRECTION: return "zero direction";
    case PDAS_ERR_ARG: return "invalid argument";
    case PDAS_ERR_NOT_INTERIOR: return "iterate not interior (x > 0 and s > 0 required)";
    case PDAS_ERR_NOT_SPD: return "normal matrix not positive definite";
    case PDAS_ERR_NONFINITE: return "non-finite value in direction or ratio test";
    case PDAS_ERR_TIMEOUT: return "device-side wait timed out";
    case PDAS_ERR_CUDA: return "CUDA error";
    case PDAS_ERR_UNSUPPORTED: return "unsupported";
  }
  return "unknown status";
}

pdas_status pdas_create(int64_t m, int64_t n, const pdas_options* opt_in, pdas_handle* out) {
  if (!out) return PDAS_ERR_ARG;
  *out = nullptr;
  pdas_options opt;
  if (opt_in) opt = *opt_in;
  else pdas_default_options(&opt);
  if (m < 1 || n <= m || m > (int64_t)1 << 20 || n > (int64_t)1 << 31) return PDAS_ERR_ARG;
  if (opt.form < PDAS_FP64 || opt.form > PDAS_FP32_IR) return PDAS_ERR_ARG;
  if (opt.a_dtype < PDAS_A_F64 || opt.a_dtype > PDAS_A_BF16) return PDAS_ERR_ARG;
  if (opt.max_iter < 1 || opt.refine_max < 0 || !(opt.refine_tol > 0) || !(opt.refine_be >= 0) ||
      !(opt.drop_tol >= 0) || !(opt.drop_keep >= 1.0) || opt.splits < 0 || (opt.exact_passes & ~1) ||
      opt.splits > 3 || (opt.infeasible & ~1) ||
      opt.stall_count < 1 || !(opt.stall_theta >= 0) || (opt.fp64_tier_tc & ~1) ||
      !(opt.df_factor_floor >= 0))
    return PDAS_ERR_ARG;
  if (opt.form == PDAS_BF16_IR && opt.a_dtype != PDAS_A_BF16) return PDAS_ERR_UNSUPPORTED;
  // TF32 form: TF32 x 3 (splits 0 or 3) or one TF32 product (splits 1); FP64 or FP32 storage
  if (opt.form == PDAS_TF32_IR && (opt.a_dtype == PDAS_A_BF16 || opt.splits == 2)) return PDAS_ERR_UNSUPPORTED;
  pdas_ctx* h = new (std::nothrow) pdas_ctx();
  if (!h) return PDAS_ERR_CUDA;
  h->m = m;
  h->n = n;
  h->ldm = (m + 15) / 16 * 16;
  h->opt = opt;
  h->st = (cudaStream_t)opt.stream;
  const int64_t nblk = (m + kTile - 1) / kTile;
  cudaError_t e = cudaSuccess;
  // Buffers of up to 1 MB share 4 MB allocations (a cudaMalloc takes 20-60 us).
  unsigned char* chunk = nullptr;
  size_t left = 0;
  auto al = [&](void** p, size_t bytes) {
    if (e != cudaSuccess) return;
    const size_t need = (bytes + 255) / 256 * 256;
    if (need > ((size_t)1 << 20)) {
      e = cudaMalloc(p, bytes);
      if (e == cudaSuccess) h->allocs.push_back(*p);
      return;
    }
    if (need > left) {
      void* c = nullptr;
      if ((e = cudaMalloc(&c, (size_t)4 << 20)) != cudaSuccess) return;
      h->allocs.push_back(c);
      chunk = (unsigned char*)c;
      left = (size_t)4 << 20;
    }
    *p = chunk;
    chunk += need;
    left -= need;
  };
  al((void**)&h->D, sizeof(double) * n);
  al((void**)&h->dx, sizeof(double) * n);
  al((void**)&h->ds, sizeof(double) * n);
  al((void**)&h->w, sizeof(double) * n);
  al((void**)&h->u, sizeof(double) * n);
  al((void**)&h->r, sizeof(double) * m);
  al((void**)&h->dy, sizeof(double) * m);
  al((void**)&h->z, sizeof(double) * m);
  al((void**)&h->rho, sizeof(double) * m);
  al((void**)&h->delta, sizeof(double) * m);
  al((void**)&h->kp, sizeof(double) * m);
  al((void**)&h->kq, sizeof(double) * m);
  al((void**)&h->kz, sizeof(double) * m);
  al((void**)&h->kp2, sizeof(double) * m);
  if (opt.infeasible) al((void**)&h->rd, sizeof(double) * n);
  al((void**)&h->part, sizeof(double) * kPartMax * 4);
  al((void**)&h->gt_part, sizeof(double) * pass_t_part_doubles(m, n, (int)dtype_size(opt.a_dtype)));
  al((void**)&h->ctickets, sizeof(unsigned) * pass_t_tickets(n));
  al((void**)&h->tickets, sizeof(unsigned) * T_COUNT);
  al((void**)&h->flags, sizeof(int) * (nblk + 1));
  if (opt.form != PDAS_FP64 && opt.a_dtype != PDAS_A_F64) al((void**)&h->pairs, sizeof(float) * 2 * pairs_pitch(n));
  al((void**)&h->sc, sizeof(Scalars));
  if (e == cudaSuccess) e = cudaMallocHost((void**)&h->sc_host, sizeof(Scalars) + sizeof(unsigned));
  if (e == cudaSuccess) {
    h->sc_seq = (unsigned*)(h->sc_host + 1);
    *h->sc_seq = 0;
  }
  if (e == cudaSuccess) e = cudaMallocHost((void**)&h->wait_pinned, sizeof(int));
  if (e == cudaSuccess) *h->wait_pinned = 0;
  al((void**)&h->adj, sizeof(double) * (5 * n + m));  // pdas_backward
  if (e == cudaSuccess) {
    // Every buffer of the FP64 tier of a mixed form is allocated here too, so
    // that a solve allocates nothing once it runs (an out-of-memory error
    // comes back from pdas_create, not from an iteration in mid-solve): the
    // FP64 matrix and its pivots, D as FP32 pairs for the double-float
    // formation, and the compact copy of the kept columns.
    al((void**)&h->M64, sizeof(double) * h->ldm * m);
    al((void**)&h->dinv64, sizeof(double) * m);
    if (opt.form != PDAS_FP64) {
      al((void**)&h->M32, sizeof(float) * h->ldm * m);
      al((void**)&h->dinv32, sizeof(float) * m);
      al((void**)&h->inv64, sizeof(double) * nblk * kTile * kTile);
      if (opt.a_dtype != PDAS_A_F64) al((void**)&h->d2, sizeof(float2) * n);
      if (opt.drop_tol > 0) {
        al((void**)&h->akept, dtype_size(opt.a_dtype) * m * n);
        al((void**)&h->dkept, sizeof(double) * n);
        al((void**)&h->kidx, sizeof(int) * n);
      }
    }
  }
  {  // the SIMT normal matrices
    size_t part = simt_fp64_part_bytes(m);
    if (opt.form == PDAS_FP32_IR) {
      const SimtPlan p = simt_plan_fp32(m, n);
      part = std::max(part, p.part_bytes);
      al((void**)&h->simt_planes, sizeof(float) * 2 * m * p.ldk);
    }
    if (part) al(&h->simt_part, part);
    al((void**)&h->simt_tickets, sizeof(unsigned) * simt_ticket_count(m));
    if (e == cudaSuccess) e = cudaMemsetAsync(h->simt_tickets, 0, sizeof(unsigned) * simt_ticket_count(m), h->st);
  }
  if (e == cudaSuccess && opt.form != PDAS_FP64 && chol_tile_count(m) <= kTileCholMaxTiles) {
    // the single-launch tile Cholesky of the FP32 factor
    std::vector<int4> tasks;
    const int workers = chol_tiles_resident();
    if (workers < 1) e = cudaErrorUnknown;
    chol_tile_tasks(m, workers, &tasks);
    const int64_t nb = chol_tile_count(m);
    h->chol_ntasks = (int)tasks.size();
    al((void**)&h->chol_tasks, sizeof(int4) * tasks.size());
    al((void**)&h->zb, sizeof(double) * m);
    if (e == cudaSuccess) e = cudaMemsetAsync(h->zb, 0xff, sizeof(double) * m, h->st);
    al((void**)&h->chol_state, sizeof(int) * (nb * nb + nb + 1));
    al((void**)&h->uinv32, sizeof(float) * nb * kCholTile * kCholTile);
    if (nb > 1) al((void**)&h->chol_planes, (size_t)chol_plane_bytes(m));
    if (e == cudaSuccess)
      e = cudaMemcpy(h->chol_tasks, tasks.data(), sizeof(int4) * tasks.size(), cudaMemcpyHostToDevice);
  }
  if (e == cudaSuccess && opt.form != PDAS_FP64 && opt.a_dtype == PDAS_A_BF16 && opt.fp64_tier_tc)
    e = dig_workspace_create(&h->dig, m, n);
  // (The plain form takes this factor up to kFp64FormDigMaxM rows.  Nothing refines its end game, and there the
  // last digits of a run belong to the rounding: 20 LPs of m = 256 to 6144 solved to 1e-8, each in two orders of its
  // rows, end with the same residuals with this factor and the SIMT one, and their iteration counts differ as those
  // of the two orders do, by one or two, in either direction.  At 8192 x 32768 one order of four runs stood out: 55
  // iterations to a relative gap of -2.6e-8 with this factor, where the other order takes 53 to 5.9e-9 and the SIMT
  // factor 53 in both, to 9.4e-10 and 7.7e-9.  Beyond 4096 the factor is less than 10 % of the time (98 against 107
  // s at 8192, 11.1 against 12.6 at 4096, 0.2 against 0.4 at 1024), so the line lies on the side where what a solve
  // returned stays as it was.)
  if (e == cudaSuccess && opt.fp64_tier_tc && (opt.form == PDAS_FP64 ? m <= kFp64FormDigMaxM : m > kCholDigMinM))
    e = chol_dig_create(&h->cdig, m);
  if (e == cudaSuccess && (opt.form == PDAS_BF16_IR || opt.form == PDAS_TF32_IR)) {
    e = tc_workspace_create(&h->tc, opt.form, opt.a_dtype, opt.splits, m, n);
    if (e == cudaErrorNotSupported) {
      cudaGetLastError();
      pdas_destroy(h);
      return PDAS_ERR_UNSUPPORTED;
    }
  }
  if (e == cudaSuccess) e = cudaMemsetAsync(h->tickets, 0, sizeof(unsigned) * T_COUNT, h->st);
  if (e == cudaSuccess) e = cudaMemsetAsync(h->ctickets, 0, sizeof(unsigned) * pass_t_tickets(n), h->st);
  if (e == cudaSuccess) e = cudaMemsetAsync(h->sc, 0, sizeof(Scalars), h->st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->st);
  if (e != cudaSuccess) {
    pdas_destroy(h);
    return PDAS_ERR_CUDA;
  }
  h->cur_f64 = opt.form == PDAS_FP64;
  *out = h;
  return PDAS_OK;
}

void pdas_destroy(pdas_handle h) {
  if (!h) return;
  if (h->st) cudaStreamSynchronize(h->st);
  else cudaDeviceSynchronize();
  for (void* p : h->allocs) cudaFree(p);
  if (h->sc_host) cudaFreeHost(h->sc_host);
  if (h->wait_pinned) cudaFreeHost(h->wait_pinned);
  tc_workspace_destroy(&h->tc);
  dig_workspace_destroy(&h->dig);
  chol_dig_destroy(&h->cdig);
  for (cudaEvent_t e : h->evs) cudaEventDestroy(e);
  delete h;
}

int64_t pdas_last_error_index(pdas_handle h) { return h ? h->err_index : -1; }

pdas_status pdas_set_wait_limit(pdas_handle h, int64_t microseconds) {
  if (!h || microseconds < 0 || microseconds > 2147483647) return PDAS_ERR_ARG;
  CK(cudaStreamSynchronize(h->st));  // no copy of the old value is still pending
  h->wait_us = (int)microseconds;
  *h->wait_pinned = (int)microseconds;
  return PDAS_OK;
}

const char* pdas_last_error_message(pdas_handle h) { return h ? h->errmsg : ""; }

pdas_status pdas_profile_enable(pdas_handle h, int enable) {
  if (!h) return PDAS_ERR_ARG;
  if (enable) {
    CK(cudaStreamSynchronize(h->st));
    h->ev_stage.clear();
    h->ev_used = 0;
    h->open_stage = -1;
    for (int i = 0; i < PDAS_STAGE_COUNT; ++i) {
      h->prof_ms[i] = 0.0;
      h->prof_calls[i] = 0;
    }
    h->launches = 0;
  }
  h->prof = enable != 0;
  return PDAS_OK;
}

pdas_status pdas_profile_read(pdas_handle h, pdas_profile* out) {
  if (!h || !out) return PDAS_ERR_ARG;
  pdas_status s = prof_fold(h);
  if (s != PDAS_OK) return s;
  for (int i = 0; i < PDAS_STAGE_COUNT; ++i) {
    out->ms[i] = h->prof_ms[i];
    out->calls[i] = h->prof_calls[i];
  }
  out->launches = h->launches;
  return PDAS_OK;
}

pdas_status pdas_direction(pdas_handle h, const void* A, const double* x, const double* s, double* dx, double* dy,
                           double* ds, pdas_iter_info* info) {
  if (!h || check_vec_args(A, x, s) != PDAS_OK || !dx || !dy || !ds) return PDAS_ERR_ARG;
  return direction_out(h, A, x, s, nullptr, dx, dy, ds, info);
}

pdas_status pdas_direction_infeasible(pdas_handle h, const void* A, const double* b, const double* c,
                                      const double* x, const double* y, const double* s, double* dx, double* dy,
                                      double* ds, pdas_iter_info* info) {
  if (!h || check_vec_args(A, x, s) != PDAS_OK || !b || !c || !y || !dx || !dy || !ds) return PDAS_ERR_ARG;
  if (!h->opt.infeasible) return PDAS_ERR_ARG;
  const Infeasible iv{y, b, c};
  return direction_out(h, A, x, s, &iv, dx, dy, ds, info);
}

pdas_status pdas_step(pdas_handle h, const void* A, const double* b, const double* c, double* x, double* y,
                      double* s, double alpha, pdas_iter_info* info) {
  if (!h || check_vec_args(A, x, s) != PDAS_OK || !b || !c || !y) return PDAS_ERR_ARG;
  if (!(alpha > 0.0 && alpha < 1.0)) return PDAS_ERR_ARG;
  const bool variant = h->opt.infeasible != 0;
  const Infeasible iv{y, b, c};
  pdas_status st;
  bool read = false;
  do {
    h->err_index = -1;
    st = step_once(h, A, b, c, x, y, s, alpha, variant ? &iv : nullptr, &read);
  } while (retry_simt(h, st));
  end_retry(h);
  if (read) fill_info(h, info, st == PDAS_OK);
  if (st != PDAS_OK) return st;
  h->last_rel_gap = variant ? fmax(fabs(h->sc_host->rel_gap), fmax(h->sc_host->pres, h->sc_host->dres))
                            : h->sc_host->rel_gap;
  // a full step ends the paper's method at an optimum; the variant's never does
  return !variant && h->sc_host->psi <= 1.0 ? PDAS_OPTIMAL_EXACT : PDAS_OK;
}

pdas_status pdas_solve(pdas_handle h, const void* A, const double* b, const double* c, double* x, double* y,
                       double* s, double alpha, double tol, int* iters_out, double* rel_gap_out) {
  if (iters_out) *iters_out = 0;
  if (!h || check_vec_args(A, x, s) != PDAS_OK || !b || !c || !y) return PDAS_ERR_ARG;
  if (!(alpha > 0.0 && alpha < 1.0) || !(tol > 0.0)) return PDAS_ERR_ARG;
  h->err_index = -1;
  h->refactored = 0;
  h->switch_reason = 0;
  // interior check before anything is modified
  pdas_status st = reset_status(h);
  if (st != PDAS_OK) return st;
  KL(launch_scaling(h->st, h->n, x, s, h->D, h->part, h->tickets, h->sc), 1);
  if ((st = read_scalars(h)) != PDAS_OK) return st;
  if ((st = device_status(h)) != PDAS_OK) return st;
  int small = 0, k = 0;
  pdas_status result = PDAS_MAX_ITER;
  double gap = INFINITY;
  for (k = 0; k < h->opt.max_iter; ++k) {
    pdas_iter_info info;
    st = pdas_step(h, A, b, c, x, y, s, alpha, &info);
    if (st < 0) {
      result = st;
      break;
    }
    gap = info.rel_gap;
    if (st == PDAS_OPTIMAL_EXACT) {
      result = st;
      ++k;
      break;
    }
    const bool converged = h->opt.infeasible ? fabs(gap) < tol && info.pres < tol && info.dres < tol : gap < tol;
    if (converged) {
      result = PDAS_OPTIMAL;
      ++k;
      break;
    }
    small = info.theta < h->opt.stall_theta ? small + 1 : 0;
    if (small >= h->opt.stall_count) {
      result = PDAS_STALLED;
      ++k;
      break;
    }
  }
  if (iters_out) *iters_out = k;
  if (rel_gap_out) *rel_gap_out = gap;
  return result;
}

pdas_status pdas_backward(pdas_handle h, const void* A, const double* x, const double* y, const double* s,
                          const double* dL_dx, double* dL_dA, double* dL_db, double* dL_dc) {
  if (!h || check_vec_args(A, x, s) != PDAS_OK || !y || !dL_dx || !dL_db || !dL_dc) return PDAS_ERR_ARG;
  if (!h->have_factor) return PDAS_ERR_ARG;  // the preconditioner comes from a previous step
  h->err_index = -1;
  const int64_t m = h->m, n = h->n;
  pdas_status st = reset_status(h);
  if (st != PDAS_OK) return st;
  double* lb = h->adj;      // dL/dc
  double* lc = lb + n;      // multiplier of X s = sigma
  double* wt = lc + n;      // A' la
  double* r1 = wt + n;      // residual of A' la + S lc = g
  double* r3 = r1 + n;      // residual of lb + X lc = 0
  double* la = r3 + n;      // dL/db (m)
  // The preconditioner is the factor of the previous iterate's D: allow the
  // conjugate gradients four times the usual number of steps.
  const int cap = h->opt.refine_max;
  auto solve_normal = [&](int* ok) -> pdas_status {  // (A D A') dy = h->r, w = A' dy
    pdas_status t = factor_solve(h, h->r, h->dy);
    if (t != PDAS_OK) return t;
    h->opt.refine_max = 4 * cap;
    t = refine(h, A, ok);
    h->opt.refine_max = cap;
    return t;
  };
  KL(launch_scaling(h->st, n, x, s, h->D, h->part, h->tickets, h->sc), 1);
  // max_p M_pp at this D for the backward-error test of the refinement (the
  // matrix itself is not formed: the preconditioner is the last factor);
  // ldm = 0 makes the diagonal reduction read the m-vector M_pp.
  st = with_dtype(h->opt.a_dtype, [&](auto tag) -> pdas_status {
    using T = std::remove_const_t<std::remove_pointer_t<decltype(tag)>>;
    KL(launch_normal_diag<T>(h->st, m, n, (const T*)A, h->D, h->kq, h->sc), 1);
    return PDAS_OK;
  });
  if (st != PDAS_OK) return st;
  KL(launch_diag_max<double>(h->st, m, 0, h->kq, h->part, h->tickets, h->sc), 1);
  // reduced solve: (A D A') la = A (D g); lb = D (A' la - g); lc = -lb / x
  KL(launch_scale_vec(h->st, n, h->D, dL_dx, h->u, h->sc), 1);
  if ((st = gemv(h, A, h->u, nullptr, h->r, 0)) != PDAS_OK) return st;
  int ok = 0;
  if ((st = solve_normal(&ok)) != PDAS_OK) return st;
  if (!ok) return PDAS_ERR_NOT_SPD;
  CK(cudaMemcpyAsync(la, h->dy, sizeof(double) * m, cudaMemcpyDeviceToDevice, h->st));
  KL(launch_adjoint_init(h->st, n, h->D, h->w, dL_dx, x, lb, lc, wt, h->sc), 1);
  // lb = D (A' la - g) cancels where D is large; two steps of refinement on
  // the full adjoint system [A' 0 S; 0 A 0; 0 I X] (la, lb, lc) = (g, 0, 0)
  // with FP64 residuals recover it.  Each correction solves the same
  // normal equations: (A D A') da = A (D r1 - r3 - lb).
  for (int it = 0; it < 2; ++it) {
    KL(launch_adjoint_resid(h->st, n, h->D, dL_dx, x, s, wt, lb, lc, r1, r3, h->u, h->sc), 1);
    if ((st = gemv(h, A, h->u, nullptr, h->r, 0)) != PDAS_OK) return st;
    if ((st = solve_normal(&ok)) != PDAS_OK) return st;
    if (!ok) break;  // the correction is at the rounding level: keep what we have
    KL(launch_axpy(h->st, m, 1.0, h->dy, la, h->sc), 1);
    KL(launch_adjoint_update(h->st, n, h->D, h->w, x, r1, r3, lb, lc, wt, h->sc), 1);
  }
  CK(cudaMemcpyAsync(dL_db, la, sizeof(double) * m, cudaMemcpyDeviceToDevice, h->st));
  CK(cudaMemcpyAsync(dL_dc, lb, sizeof(double) * n, cudaMemcpyDeviceToDevice, h->st));
  if (dL_dA) KL(launch_adjoint_dA(h->st, m, n, la, x, y, lb, dL_dA, h->sc), 1);
  if ((st = read_scalars(h)) != PDAS_OK) return st;
  return device_status(h);
}

// ---- components ------------------------------------------------------------
pdas_status pdas_form_normal(pdas_handle h, const void* A, const double* x, const double* s) {
  if (!h || check_vec_args(A, x, s) != PDAS_OK) return PDAS_ERR_ARG;
  pdas_status st = reset_status(h);
  if (st != PDAS_OK) return st;
  KL(launch_scaling(h->st, h->n, x, s, h->D, h->part, h->tickets, h->sc), 1);
  STAGE(h, PDAS_STAGE_NORMAL);
  if ((st = form_normal(h, A)) != PDAS_OK) return st;
  STAGE_END(h);
  if ((st = read_scalars(h)) != PDAS_OK) return st;
  return device_status(h);
}

pdas_status pdas_copy_matrix(pdas_handle h, void* dst, int* dtype_out) {
  if (!h || !dst) return PDAS_ERR_ARG;
  const size_t es = h->cur_f64 ? sizeof(double) : sizeof(float);
  const void* src = h->cur_f64 ? (const void*)h->M64 : (const void*)h->M32;
  if (!src) return PDAS_ERR_ARG;
  CK(cudaMemcpy2DAsync(dst, es * h->m, src, es * h->ldm, es * h->m, h->m, cudaMemcpyDeviceToDevice, h->st));
  CK(cudaStreamSynchronize(h->st));
  if (dtype_out) *dtype_out = h->cur_f64 ? PDAS_A_F64 : PDAS_A_F32;
  return PDAS_OK;
}

pdas_status pdas_load_matrix(pdas_handle h, const void* src, int dtype) {
  if (!h || !src || (dtype != PDAS_A_F64 && dtype != PDAS_A_F32)) return PDAS_ERR_ARG;
  if (!h->cur_f64 && !h->M32) return PDAS_ERR_ARG;
  void* dst = h->cur_f64 ? (void*)h->M64 : (void*)h->M32;
  if (!dst) return PDAS_ERR_ARG;
  KL(launch_convert_matrix(h->st, h->m, h->m, src, dtype == PDAS_A_F64, h->ldm, dst, h->cur_f64), 1);
  CK(cudaStreamSynchronize(h->st));
  return PDAS_OK;
}

pdas_status pdas_factor(pdas_handle h) {
  if (!h) return PDAS_ERR_ARG;
  h->err_index = -1;
  pdas_status st = reset_status(h);
  if (st != PDAS_OK) return st;
  // The plain form's tensor-core factor overwrites M: M is kept in its upper
  // triangle meanwhile, for the SIMT factor's own verdict on a failed pivot.
  const bool keep = !is_mixed(h) && h->cdig.m > 0;
  if (keep) KL(launch_mirror_lower(h->st, h->m, h->ldm, h->M64, h->kq, false), 1);
  if ((st = factor(h)) != PDAS_OK) return st;
  if ((st = read_scalars(h)) != PDAS_OK) return st;
  st = device_status(h);
  if (keep && st == PDAS_ERR_NOT_SPD) {
    h->err_index = -1;
    if ((st = reset_status(h)) != PDAS_OK) return st;
    KL(launch_mirror_lower(h->st, h->m, h->ldm, h->M64, h->kq, true), 1);
    h->no_dffactor_once = true;
    st = factor(h);
    h->no_dffactor_once = false;
    if (st != PDAS_OK) return st;
    if ((st = read_scalars(h)) != PDAS_OK) return st;
    st = device_status(h);
  }
  h->have_factor = st == PDAS_OK;
  return st;
}

pdas_status pdas_factor_solve(pdas_handle h, const double* rhs, double* out) {
  if (!h || !rhs || !out) return PDAS_ERR_ARG;
  pdas_status st = reset_status(h);
  if (st != PDAS_OK) return st;
  CK(cudaMemcpyAsync(h->rho, rhs, sizeof(double) * h->m, cudaMemcpyDeviceToDevice, h->st));
  if ((st = factor_solve(h, h->rho, h->delta)) != PDAS_OK) return st;
  CK(cudaMemcpyAsync(out, h->delta, sizeof(double) * h->m, cudaMemcpyDeviceToDevice, h->st));
  if ((st = read_scalars(h)) != PDAS_OK) return st;
  return device_status(h);
}

pdas_status pdas_gemv(pdas_handle h, const void* A, const double* v, double* out) {
  if (!h || !A || !v || !out) return PDAS_ERR_ARG;
  pdas_status st = reset_status(h);
  if (st != PDAS_OK) return st;
  if ((st = gemv(h, A, v, nullptr, out, -1, df_passes(h))) != PDAS_OK) return st;
  if ((st = read_scalars(h)) != PDAS_OK) return st;
  return device_status(h);
}

pdas_status pdas_gemv_t(pdas_handle h, const void* A, const double* u, double* out) {
  if (!h || !A || !u || !out) return PDAS_ERR_ARG;
  pdas_status st = reset_status(h);
  if (st != PDAS_OK) return st;
  if ((st = gemv_t(h, A, u, 0, nullptr, out, nullptr, nullptr, df_passes(h))) != PDAS_OK) return st;
  if ((st = read_scalars(h)) != PDAS_OK) return st;
  return device_status(h);
}

}  // extern "C"
