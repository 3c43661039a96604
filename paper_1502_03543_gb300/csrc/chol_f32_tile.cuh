// chol_f32_tile.cuh -- the 128 x 128 tile operations of the FP32 tile Cholesky
// (chol_tiles.cu) that lie on its dependency chain: the factor of a diagonal
// tile and the triangular solve of a tile against it, by one CTA of 256
// threads, on tiles held column by column in shared memory (element (r, c) at
// T[c][r], pitch 132 floats).
//
// What bounds them is latency, not arithmetic: 128 pivots, each a reciprocal
// square root and a few dependent operations, and the reads of shared memory in
// between.  Column-major tiles make a thread per row conflict-free and let
// every coefficient be read as a 16-byte broadcast.  Both operations run in
// 32-column blocks, and inside a block in groups of 8 columns:
//   * the 8 x 8 diagonal block of a group is factored redundantly by every
//     thread in registers, so its chain has no shuffle and no barrier
//     (reciprocal square root, multiply, multiply-add per pivot);
//   * a thread per row then solves its row against it and applies the 8 new
//     columns to the rest of its 32;
//   * the trailing columns take a whole 32-column block at a time from
//     shared memory, in register tiles.
// Loops over groups and blocks stay rolled (the thread's row moves down by 8
// registers per group): fully unrolled, the instruction fetch costs more than
// it saves.  Measured on one tile: the factorisation 11 us (26 us with a warp
// per 32 x 32 block and two shared-memory reads per multiply-add), the solve 10 us
// (16 us column by column), 15 us with its panels streamed from L2.
#pragma once

#include "pdas_internal.cuh"
#include "tile_core.cuh"

namespace pdas {
namespace ft {

constexpr int kPt = kBig + 4;  // pitch of a column: 16-byte aligned, columns 4 banks apart
using Tile = float (*)[kPt];
constexpr size_t kTileBytes = sizeof(float) * kBig * kPt;

// Thread unit v (0..15): row r and first column c of its 4 consecutive
// columns.  A warp covers 16 rows x 8 columns: whole 32-byte sectors in global
// memory, 32 distinct banks in the transposed tile.
__device__ __forceinline__ void unit_rc(int v, int& r, int& c) {
  const int lane = threadIdx.x & 31, u = (threadIdx.x >> 5) + 8 * v;
  r = 16 * (u & 7) + (lane & 15);
  c = 8 * (u >> 3) + 4 * (lane >> 4);
}

// Rows p0.. and columns q0.. of M (through L2) into registers.  Rows are
// padded to 16 columns (ldm), so a 16-byte load that starts inside the matrix
// stays inside its row.
__device__ __forceinline__ void fetch_tile(float4 (&x)[16], int64_t m, int64_t ldm, const float* M, int64_t p0,
                                           int64_t q0) {
#pragma unroll
  for (int v = 0; v < 16; ++v) {
    int r, c;
    unit_rc(v, r, c);
    x[v] = (p0 + r < m && q0 + c < m) ? __ldcg(reinterpret_cast<const float4*>(M + (p0 + r) * ldm + q0 + c))
                                     : make_float4(0.f, 0.f, 0.f, 0.f);
  }
}
// ... and from there into the tile.  diag: only the lower triangle counts
// (zeros above it), and rows and columns past m are the identity's; else rows
// past m are zero.
__device__ __forceinline__ void put_tile(const float4 (&x)[16], int64_t m, int64_t p0, bool diag, Tile T) {
  const int kb = (int)(m - p0 < kBig ? m - p0 : kBig);
#pragma unroll
  for (int v = 0; v < 16; ++v) {
    int r, c;
    unit_rc(v, r, c);
    const float e[4] = {x[v].x, x[v].y, x[v].z, x[v].w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const bool in = r < kb && (!diag || c + k <= r);
      T[c + k][r] = in ? e[k] : (diag && r == c + k) ? 1.f : 0.f;
    }
  }
}

// Hardware estimates of 1 / d and 1 / sqrt(d) for normal d (within 2 ulp; the
// FP32 factor is a preconditioner, and every entry of a column is scaled by
// the same value).
__device__ __forceinline__ float fast_rcp(float d) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
  return r;
}
__device__ __forceinline__ float fast_rsqrt(float d) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
  return r;
}

__device__ __forceinline__ void bar_warps(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// a[8 + q] -= sum_{c < 8} a[c] L_{q0 + q, c0 + c} for the next 8 nch columns of
// the thread's row (L column-major: L[c0 + c][q0 + q], 16-byte broadcasts).
__device__ __forceinline__ void apply_group(float (&a)[32], const float (*L)[kPt], int c0, int q0, int nch) {
#pragma unroll
  for (int h = 0; h < 3; ++h) {
    if (h < nch) {
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const float4 lo = *reinterpret_cast<const float4*>(&L[c0 + c][q0 + 8 * h]);
        const float4 hi = *reinterpret_cast<const float4*>(&L[c0 + c][q0 + 8 * h + 4]);
        float* t = a + 8 + 8 * h;
        t[0] = fmaf(-a[c], lo.x, t[0]), t[1] = fmaf(-a[c], lo.y, t[1]);
        t[2] = fmaf(-a[c], lo.z, t[2]), t[3] = fmaf(-a[c], lo.w, t[3]);
        t[4] = fmaf(-a[c], hi.x, t[4]), t[5] = fmaf(-a[c], hi.y, t[5]);
        t[6] = fmaf(-a[c], hi.z, t[6]), t[7] = fmaf(-a[c], hi.w, t[7]);
      }
    }
  }
}

// The lower triangle of the 8 x 8 block at column c0 (column-major in T).
__device__ __forceinline__ void load_block8(float (&t)[8][8], const float (*T)[kPt], int c0) {
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const float4 lo = *reinterpret_cast<const float4*>(&T[c0 + j][c0]);
    const float4 hi = *reinterpret_cast<const float4*>(&T[c0 + j][c0 + 4]);
    t[0][j] = lo.x, t[1][j] = lo.y, t[2][j] = lo.z, t[3][j] = lo.w;
    t[4][j] = hi.x, t[5][j] = hi.y, t[6][j] = hi.z, t[7][j] = hi.w;
  }
}

// t = chol(t) (lower triangle) in registers, rs = 1 / L_cc.  The sweep runs in
// the L D L' form (a pivot's chain is a reciprocal, a multiply and a
// multiply-add); the columns are scaled at the end.  Returns false if a pivot or its reciprocal leaves the normal range (then
// t is spoilt).
__device__ __forceinline__ bool chol8(float (&t)[8][8], float (&rs)[8]) {
  bool ok = true;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const float d = t[c][c];
    ok = ok && d >= 1.17549435e-38f && d <= 8.5e37f;
    const float ri = fast_rcp(d);
    rs[c] = fast_rsqrt(d);
#pragma unroll
    for (int j = c + 1; j < 8; ++j) {
      const float u = t[j][c] * ri;
#pragma unroll
      for (int i = j; i < 8; ++i) t[i][j] = fmaf(-u, t[i][c], t[i][j]);
    }
  }
#pragma unroll
  for (int c = 0; c < 8; ++c)
#pragma unroll
    for (int i = c + 1; i < 8; ++i) t[i][c] *= rs[c];
  return ok;
}

// The same by plain sweeps with full range; returns the first pivot that is
// not positive and finite, or -1.
__device__ __noinline__ int chol8_careful(const float (*T)[kPt], int c0, float* tout, float* rs) {
  float t[8][8];
  int bad = -1;
#pragma unroll 1
  for (int j = 0; j < 8; ++j)
#pragma unroll 1
    for (int i = 0; i < 8; ++i) t[i][j] = T[c0 + j][c0 + i];
#pragma unroll 1
  for (int c = 0; c < 8; ++c) {
    const float d = t[c][c];
    if (bad < 0 && (!(d > 0.f) || !isfinite(d))) bad = c;
    rs[c] = rsqrtf(d);
#pragma unroll 1
    for (int i = c + 1; i < 8; ++i) t[i][c] *= rs[c];
#pragma unroll 1
    for (int j = c + 1; j < 8; ++j)
#pragma unroll 1
      for (int i = j; i < 8; ++i) t[i][j] = fmaf(-t[i][c], t[j][c], t[i][j]);
  }
#pragma unroll 1
  for (int e = 0; e < 64; ++e) tout[e] = t[e >> 3][e & 7];
  return bad;
}

// C_rq -= sum_{k < 32} S_r,k0+k S_q,k0+k in 4 x 4 units of the lower triangle,
// rows r >= rlo, columns qlo <= q < qhi, spread over threads p of P.
__device__ __forceinline__ void potrf_update(Tile S, int k0, int rlo, int qlo, int qhi, int p, int P) {
  const int nr4 = (kBig - rlo) >> 2, n = nr4 * ((qhi - qlo) >> 2);
#pragma unroll 1
  for (int u = p; u < n; u += P) {
    const int r = rlo + 4 * (u % nr4), q = qlo + 4 * (u / nr4);
    if (q > r) continue;  // (units: q and r are multiples of 4)
    float4 t[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) t[j] = *reinterpret_cast<const float4*>(&S[q + j][r]);
#pragma unroll 8
    for (int k = 0; k < 32; ++k) {
      const float4 a = *reinterpret_cast<const float4*>(&S[k0 + k][r]);
      const float4 b = *reinterpret_cast<const float4*>(&S[k0 + k][q]);
      const float bb[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        t[j].x = fmaf(-a.x, bb[j], t[j].x), t[j].y = fmaf(-a.y, bb[j], t[j].y);
        t[j].z = fmaf(-a.z, bb[j], t[j].z), t[j].w = fmaf(-a.w, bb[j], t[j].w);
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) *reinterpret_cast<float4*>(&S[q + j][r]) = t[j];
  }
}

// L = chol(S) in place (lower triangle; entries above it are left undefined),
// reciprocals of the pivots to rcp.  All 256 threads, after a barrier that
// made S visible; ends with one.  Returns -1 or the index of the first pivot
// that is not positive and finite (the same in all threads; the sweep then
// stops after that 32-column block).  Block b: warps 0 .. 3 - b factor its 32
// columns, a thread per row, while the others apply block b - 1 to the
// columns past block b; then every thread applies block b to the next 32
// columns.  store(b) is called by every thread once block b is final, and
// publish(b) behind the next barrier.
template <class Store, class Publish>
__device__ __forceinline__ int potrf(Tile S, float* rcp, int* s_fail, Store&& store, Publish&& publish) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) *s_fail = -1;
#pragma unroll 1
  for (int b = 0; b < 4; ++b) {
    const int c0 = 32 * b, nw = 4 - b;
    if (warp < nw) {
      const int row = c0 + 32 * warp + lane;
      float a[32];
#pragma unroll
      for (int q = 0; q < 32; ++q) a[q] = S[c0 + q][row];
#pragma unroll 1
      for (int g = 0; g < 4; ++g) {
        const int g0 = c0 + 8 * g;
        float t[8][8], rs[8];
        load_block8(t, S, g0);
        if (!chol8(t, rs)) {  // (the same outcome in every thread)
          float tt[64], rr[8];
          const int bad = chol8_careful(S, g0, tt, rr);
#pragma unroll
          for (int e = 0; e < 64; ++e) t[e >> 3][e & 7] = tt[e];
#pragma unroll
          for (int c = 0; c < 8; ++c) rs[c] = rr[c];
          if (tid == 0 && bad >= 0 && *s_fail < 0) *s_fail = g0 + bad;
        }
        if (tid == 0) {
#pragma unroll
          for (int c = 0; c < 8; ++c) rcp[g0 + c] = rs[c];
        }
        // the row against the group (a row of the group itself gets its own
        // entries of L up to its diagonal)
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          float x = a[c];
#pragma unroll
          for (int k = 0; k < c; ++k) x = fmaf(-a[k], t[c][k], x);
          a[c] = x * rs[c];
        }
        bar_warps(1, 32 * nw);  // every thread has read the group's block
        if (row >= g0) {
#pragma unroll
          for (int c = 0; c < 8; ++c)
            if (row >= g0 + c) S[g0 + c][row] = a[c];
        }
        if (g == 3) break;
        bar_warps(2, 32 * nw);  // the group's columns are in place
        apply_group(a, S, g0, g0 + 8, 3 - g);
        if (warp == 0 && lane >= 8 * g + 8 && lane < 8 * g + 16) {  // the next group's block
#pragma unroll
          for (int c = 0; c < 8; ++c) S[g0 + 8 + c][row] = a[8 + c];
        }
#pragma unroll
        for (int q = 0; q < 24; ++q) a[q] = a[q + 8];
        bar_warps(1, 32 * nw);  // the next group's block is in place
      }
    } else if (b > 0) {
      potrf_update(S, c0 - 32, c0 + 32, c0 + 32, kBig, tid - 32 * nw, kThreads - 32 * nw);
    }
    __syncthreads();
    if (*s_fail >= 0) break;
    store(b);
    if (b < 3) potrf_update(S, c0, c0 + 32, c0 + 32, c0 + 64, tid, kThreads);
    __syncthreads();
    publish(b);
  }
  return *s_fail;
}

// The 32 entries c0 .. c0 + 31 of row r of X L' = C, in place; P: the panel of L
// (column c0 + c at P[c]).
__device__ __forceinline__ void solve_row(Tile C, const float (*P)[kPt], const float* rcp, int c0, int r) {
  const float(*L)[kPt] = P - c0;
  float a[32];
#pragma unroll
  for (int q = 0; q < 32; ++q) a[q] = C[c0 + q][r];
#pragma unroll 1
  for (int g = 0; g < 4; ++g) {
    const int g0 = c0 + 8 * g;
    float t[8][8];
    load_block8(t, L, g0);
    const float4 r0 = *reinterpret_cast<const float4*>(rcp + g0), r1 = *reinterpret_cast<const float4*>(rcp + g0 + 4);
    const float rs[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      float x = a[c];
#pragma unroll
      for (int k = 0; k < c; ++k) x = fmaf(-a[k], t[c][k], x);
      a[c] = x * rs[c];
      C[g0 + c][r] = a[c];
    }
    if (g == 3) break;
    apply_group(a, L, g0, g0 + 8, 3 - g);
#pragma unroll
    for (int q = 0; q < 24; ++q) a[q] = a[q + 8];
  }
}

// C columns q0 .. q0 + 31 -= X L' for the 32 columns k0 .. of X = C, by the
// 32 W threads p = 0 .. of the caller: thread (tx, ty) = (p % 16, p / 16) owns
// rows 4 tx.. and 64 + 4 tx.. and 16 / W columns.
template <int W>
__device__ __forceinline__ void trsm_update(Tile C, const float (*P)[kPt], int k0, int q0, int p) {
  constexpr int NC = 16 / W;  // columns per thread
  const float(*L)[kPt] = P - k0;  // the panel's column k0 + k at P[k]
  static_assert(NC == 2 || NC == 4, "8 or 4 warps");
  const int tx = p & 15, q = q0 + NC * (p >> 4);
  float4 t[NC][2];
#pragma unroll
  for (int e = 0; e < NC; ++e)
#pragma unroll
    for (int h = 0; h < 2; ++h) t[e][h] = *reinterpret_cast<const float4*>(&C[q + e][64 * h + 4 * tx]);
#pragma unroll 8
  for (int k = 0; k < 32; ++k) {
    const float4 a[2] = {*reinterpret_cast<const float4*>(&C[k0 + k][4 * tx]),
                         *reinterpret_cast<const float4*>(&C[k0 + k][64 + 4 * tx])};
    float b[NC];
    if constexpr (NC == 4) *reinterpret_cast<float4*>(b) = *reinterpret_cast<const float4*>(&L[k0 + k][q]);
    else *reinterpret_cast<float2*>(b) = *reinterpret_cast<const float2*>(&L[k0 + k][q]);
#pragma unroll
    for (int e = 0; e < NC; ++e)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        t[e][h].x = fmaf(-a[h].x, b[e], t[e][h].x), t[e][h].y = fmaf(-a[h].y, b[e], t[e][h].y);
        t[e][h].z = fmaf(-a[h].z, b[e], t[e][h].z), t[e][h].w = fmaf(-a[h].w, b[e], t[e][h].w);
      }
  }
#pragma unroll
  for (int e = 0; e < NC; ++e)
#pragma unroll
    for (int h = 0; h < 2; ++h) *reinterpret_cast<float4*>(&C[q + e][64 * h + 4 * tx]) = t[e][h];
}

// One 32-column panel b of the factor L of the diagonal tile at row q0 of M:
// rows from 32 b on, 16-byte loads through L2 (thread unit v of 4: row r,
// columns 32 b + c .. + 3), then into a column-major panel buffer (entries above
// the diagonal are never used; rows past m are the identity's).
__host__ __device__ __forceinline__ void panel_rc(int tid, int v, int& r, int& c) {
  const int lane = tid & 31, u = (tid >> 5) + 8 * v;
  r = 16 * (u & 7) + (lane & 15);
  c = 8 * (u >> 3) + 4 * (lane >> 4);
}
// Whether the vector at row r, column c of that tile is read: only where it
// starts on or below the diagonal, so at a column <= its row < m, from where a
// row padded to a multiple of 16 columns holds all of it.  (A panel's 32
// columns can reach past the padding: m = 33 has rows of 48 and a panel from 32
// to 63.)
__host__ __device__ __forceinline__ bool panel_reads(int64_t m, int64_t q0, int r, int c) {
  return c <= r && q0 + r < m;
}
__device__ __forceinline__ void fetch_panel(float4 (&x)[4], int64_t m, int64_t ldm, const float* M, int64_t q0, int b) {
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    int r, c;
    panel_rc(threadIdx.x, v, r, c);
    x[v] = panel_reads(m, q0, r, 32 * b + c)
               ? __ldcg(reinterpret_cast<const float4*>(M + (q0 + r) * ldm + q0 + 32 * b + c))
               : make_float4(0.f, 0.f, 0.f, 0.f);
  }
}
__device__ __forceinline__ void put_panel(const float4 (&x)[4], Tile P) {
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    int r, c;
    panel_rc(threadIdx.x, v, r, c);
    P[c][r] = x[v].x, P[c + 1][r] = x[v].y, P[c + 2][r] = x[v].z, P[c + 3][r] = x[v].w;
  }
}

// X L' = C in place for the factor L of the diagonal tile at row q0 of M, whose
// panels are taken as they are finished (flag counts them), so that the solve
// runs beside the factorisation when that is still going on.  All 256
// threads, after a barrier that made C visible.  Per 32-column block b: its
// panel and pivot reciprocals into the panel buffer P[b % 2]; warps 0 .. 3 solve
// it, a thread per row, while warps 4 .. 7 apply block b - 1 to the columns
// past b; then all apply block b to the next 32 columns.  done(b) is called by
// every thread once block b of X is final, and issued(b) behind the barrier
// after that.  Returns false (for all threads) if a wait gave up.
template <class Wait, class Done, class Issued>
__device__ __forceinline__ bool trsm(Tile C, float (*P)[32][kPt], float* rcp, int* s_go, int64_t m, int64_t ldm,
                                     const float* M, const float* dinv, int64_t q0, const int* flag, Wait&& wait,
                                     Done&& done, Issued&& issued) {
  const int tid = threadIdx.x;
  float4 x[4];
  float rc = 1.f;
  bool have = false;  // the panel of this block is already on its way
#pragma unroll 1
  for (int b = 0; b < 4; ++b) {
    const int c0 = 32 * b;
    if (!have) {
      if (tid == 0) s_go[0] = wait(flag, b + 1);
      __syncthreads();
      if (!s_go[0]) return false;
      fetch_panel(x, m, ldm, M, q0, b);
      if (tid < 32) rc = q0 + c0 + tid < m ? __ldcg(dinv + q0 + c0 + tid) : 1.f;
    }
    put_panel(x, P[b & 1]);
    if (tid < 32) rcp[c0 + tid] = rc;
    if (tid == 0) s_go[1] = b < 3 && wait(flag, -(b + 2));  // (without waiting)
    __syncthreads();
    have = s_go[1];
    if (have) {
      fetch_panel(x, m, ldm, M, q0, b + 1);
      if (tid < 32) rc = q0 + c0 + 32 + tid < m ? __ldcg(dinv + q0 + c0 + 32 + tid) : 1.f;
    }
    if (tid < kBig) {
      solve_row(C, P[b & 1], rcp, c0, tid);
    } else if (b > 0) {
#pragma unroll 1
      for (int c = c0 + 32; c < kBig; c += 32) trsm_update<4>(C, P[(b - 1) & 1], c0 - 32, c, tid - kBig);
    }
    __syncthreads();
    if (b < 3) trsm_update<8>(C, P[b & 1], c0, c0 + 32, tid);
    done(b);
    __syncthreads();
    issued(b);
  }
  return true;
}

}  // namespace ft
}  // namespace pdas
