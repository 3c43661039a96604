// syrk_simt.cu -- the normal matrix M = A D A' (Section V: the system
// (A D A') dy = A x) on the SIMT pipes: FP64 for the plain FP64 form and for
// the FP64 re-factorisation of the mixed forms, FP32 for the FP32_IR form.
// Only the lower triangle (p >= q) is formed and written.
//
// Both kernels split M into tiles and, where the tiles alone would leave SMs
// idle, K into S slices per tile (SimtPlan).  Every slice writes its partial
// tile to the workspace; the CTA that finishes a tile last (one ticket per
// tile) adds the S partials in slice order, so the result does not depend on
// the order in which CTAs finish.
#include <algorithm>

#include "syrk_simt.cuh"
#include "tile_core.cuh"

namespace pdas {

namespace {

// ---- FP64 -------------------------------------------------------------------
// Bound by the FP64 pipe (2 multiply-adds per clock and SM): a warp
// instruction holds it for 64 cycles, in which the 2 shared-memory loads per
// multiply-add of a small register tile cost nothing.  So tiles are small, for
// balance over 152 SMs and little work above the diagonal (32 x 32: 3 % of M at
// m = 1000; the 16 x 16 quarter above the diagonal of a diagonal tile is
// skipped), and 16 x 16 where even 32 x 32 tiles leave most SMs idle.  A small
// tile costs more operands per multiply-add, and what they take of that pipe is
// what counts: the product A_pk D_k (1/32 of the multiply-adds with 32 rows)
// stays on it, the widening of a value stored as FP32 or BF16 (2/32) is done on
// the integer pipes.  BF16 A, n = 2 m, 64 x 64 tiles before -> 32 x 32 with the
// conversions -> now: m = 3000 50.6 -> 49.7 -> 46.6 ms, 6000 378 -> 390 -> 362, 8192
// 946 -> 984 -> 916 (FP64 A: 911 -> 915 there).
// Measured against 64 x 64 tiles without a K split: m = 64, n = 128 (one tile):
// 139 -> 9.6 us; 1000 x 2500 (136 tiles on 152 SMs): 2697 -> 2388 us (floor 2000).
template <typename T, int TS>
__global__ void __launch_bounds__(kThreads) k_syrk_fp64(int64_t m, int64_t n, const T* __restrict__ A,
                                                        const double* __restrict__ D, double* __restrict__ M,
                                                        int64_t ldm, int64_t kslice, int slices, double* part,
                                                        unsigned* tickets, const Scalars* sc) {
  constexpr int R = TS / 16;              // outputs per thread and direction
  constexpr int PER = TS * kKc / kThreads;  // elements of each operand per thread and K chunk
  __shared__ double sp[2][kKc][TS + 1], sq[2][kKc][TS + 1];
  __shared__ bool last;
  if (*(volatile const int*)&sc->status != 0) return;
  int64_t ti, tj;
  lower_tile(blockIdx.x, ti, tj);
  const int64_t p0 = ti * TS, q0 = tj * TS;
  const int64_t kbeg = blockIdx.y * kslice, kend = kbeg + kslice < n ? kbeg + kslice : n;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const bool diag = ti == tj;
  double acc[R][R];
#pragma unroll
  for (int i = 0; i < R; ++i)
#pragma unroll
    for (int j = 0; j < R; ++j) acc[i][j] = 0.0;
  double rp[PER], rq[PER], rd[PER];
  auto fetch = [&](int64_t k0) {
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int e = tid + u * kThreads, r = e / kKc;
      const int64_t k = k0 + e % kKc;
      const bool kin = k < kend;
      rd[u] = kin ? __ldg(D + k) : 0.0;
      rp[u] = (kin && p0 + r < m) ? widen_int(A[(p0 + r) * n + k]) : 0.0;
      rq[u] = (kin && q0 + r < m) ? widen_int(A[(q0 + r) * n + k]) : 0.0;
    }
  };
  fetch(kbeg);
  int buf = 0;
  for (int64_t k0 = kbeg; k0 < kend; k0 += kKc, buf ^= 1) {
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int e = tid + u * kThreads;
      sp[buf][e % kKc][e / kKc] = rp[u] * rd[u];  // A_pk D_k in FP64
      sq[buf][e % kKc][e / kKc] = rq[u];
    }
    __syncthreads();  // (two buffers: the previous chunk's readers are past their barrier)
    if (k0 + kKc < kend) fetch(k0 + kKc);
#pragma unroll
    for (int kk = 0; kk < kKc; ++kk) {
      double a[R], b[R];
#pragma unroll
      for (int i = 0; i < R; ++i) a[i] = sp[buf][kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < R; ++j) b[j] = sq[buf][kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < R; ++j)
          if (j <= i || !diag) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
  }
  if (slices > 1) {
    double* dst = part + ((int64_t)blockIdx.x * slices + blockIdx.y) * TS * TS + tid;
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
      for (int j = 0; j < R; ++j) __stcg(dst + (i * R + j) * kThreads, acc[i][j]);
    __threadfence();
    __syncthreads();
    if (tid == 0) {
      last = atomicAdd(tickets + blockIdx.x, 1u) == (unsigned)slices - 1;
      if (last) tickets[blockIdx.x] = 0;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const double* src = part + (int64_t)blockIdx.x * slices * TS * TS + tid;
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
      for (int j = 0; j < R; ++j) acc[i][j] = 0.0;
#pragma unroll 4
    for (int s = 0; s < slices; ++s)
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < R; ++j) acc[i][j] += __ldcg(src + (int64_t)s * TS * TS + (i * R + j) * kThreads);
  }
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int64_t p = p0 + ty + 16 * i;
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int64_t q = q0 + tx + 16 * j;
      if (p < m && q <= p) M[p * ldm + q] = acc[i][j];
    }
  }
}

// ---- FP32 -------------------------------------------------------------------
// Operand planes of the FP32 product, each value formed once per call instead
// of once per tile (an FP64 product per loaded element held the FP64 pipe for
// most of the time of the former kernel): B = fl32(A_pk D_k), the product in
// FP64, and A itself, m x ldk FP32 each, so that the product loads 16 bytes
// whatever the alignment of A's rows.  The planes hold columns c0 .. c0 + ldk - 1
// (zero past column n); only where both would exceed 4 GB is that not all of A.
// The FP64 product and its conversion to FP32 are what the pass costs beyond its
// traffic; the widening of A runs on the integer pipes.  (With D as an FP32 pair
// on the FP32 pipes the whole matrix took 139 us at 1001 x 3003 and 745 at 2000 x
// 6000, now 132 and 713; and D lost 5 of its 53 bits.)  A block takes 16 rows of
// 256 columns.
constexpr int kPlaneRows = 16;
template <typename T>
__global__ void __launch_bounds__(kThreads) k_simt_planes(int64_t m, int64_t n, int64_t c0, int64_t ldk,
                                                          const T* __restrict__ A, const double* __restrict__ D,
                                                          float* __restrict__ Bp, float* __restrict__ Ap,
                                                          const Scalars* sc) {
  if (*(volatile const int*)&sc->status != 0) return;
  const int64_t k = blockIdx.x * (int64_t)kThreads + threadIdx.x;
  if (k >= ldk) return;
  const bool in = c0 + k < n;
  const double d = in ? __ldg(D + c0 + k) : 0.0;
  for (int64_t p0 = (int64_t)blockIdx.y * kPlaneRows; p0 < m; p0 += (int64_t)gridDim.y * kPlaneRows) {
#pragma unroll 8
    for (int r = 0; r < kPlaneRows; ++r) {
      const int64_t p = p0 + r;
      if (p >= m) break;
      const T a = in ? A[p * n + c0 + k] : T(0.f);
      Bp[p * ldk + k] = (float)(widen_int(a) * d);
      Ap[p * ldk + k] = widen32(a);
    }
  }
}

// M = B A' on 128 x 128 tiles, 8 x 8 outputs per thread, K chunks of 16 in two
// shared-memory buffers (next chunk's loads in flight during the products).
// Thread (tx, ty) owns rows 4 ty .. + 3 and 64 + 4 ty .. + 3 and the same of
// columns by tx, so a step reads four 16-byte vectors for 64 multiply-adds.
// Bound by the FP32 pipe.  Measured at 1001 x 3003 (36 tiles): 774 us as 36 CTAs
// with the FP64 products in the loads -> 113 us with the planes and 8 K slices
// (288 CTAs; the multiply-adds alone take 46 us).
constexpr int kPitch = kBig + 4;

__global__ void __launch_bounds__(kThreads, 2) k_syrk_fp32(int64_t m, int64_t ldk, const float* __restrict__ Bp,
                                                           const float* __restrict__ Ap, float* __restrict__ M,
                                                           int64_t ldm, int add, int64_t kslice, int slices, float* part,
                                                           unsigned* tickets, const Scalars* sc) {
  __shared__ __align__(16) float sp[2][kKc][kPitch], sq[2][kKc][kPitch];
  __shared__ bool last;
  if (*(volatile const int*)&sc->status != 0) return;
  int64_t ti, tj;
  lower_tile(blockIdx.x, ti, tj);
  const int64_t p0 = ti * kBig, q0 = tj * kBig;
  const int64_t kbeg = blockIdx.y * kslice, kend = kbeg + kslice < ldk ? kbeg + kslice : ldk;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int lr = tid >> 2, lk = (tid & 3) * 4;  // this thread loads rows lr, lr + 64, elements lk .. lk + 3
  float4 rp[2], rq[2];
  auto fetch = [&](int64_t k0) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int64_t p = p0 + lr + 64 * h, q = q0 + lr + 64 * h;
      const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
      rp[h] = p < m ? __ldg(reinterpret_cast<const float4*>(Bp + p * ldk + k0 + lk)) : z;
      rq[h] = q < m ? __ldg(reinterpret_cast<const float4*>(Ap + q * ldk + k0 + lk)) : z;
    }
  };
  float acc[8][8];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
  fetch(kbeg);
  int buf = 0;
  for (int64_t k0 = kbeg; k0 < kend; k0 += kKc, buf ^= 1) {  // slices are whole chunks of 16
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = lr + 64 * h;
      sp[buf][lk][r] = rp[h].x, sp[buf][lk + 1][r] = rp[h].y, sp[buf][lk + 2][r] = rp[h].z, sp[buf][lk + 3][r] = rp[h].w;
      sq[buf][lk][r] = rq[h].x, sq[buf][lk + 1][r] = rq[h].y, sq[buf][lk + 2][r] = rq[h].z, sq[buf][lk + 3][r] = rq[h].w;
    }
    __syncthreads();
    if (k0 + kKc < kend) fetch(k0 + kKc);
#pragma unroll
    for (int kk = 0; kk < kKc; ++kk) {
      float a[8], b[8];
      *reinterpret_cast<float4*>(a) = *reinterpret_cast<const float4*>(&sp[buf][kk][4 * ty]);
      *reinterpret_cast<float4*>(a + 4) = *reinterpret_cast<const float4*>(&sp[buf][kk][64 + 4 * ty]);
      *reinterpret_cast<float4*>(b) = *reinterpret_cast<const float4*>(&sq[buf][kk][4 * tx]);
      *reinterpret_cast<float4*>(b + 4) = *reinterpret_cast<const float4*>(&sq[buf][kk][64 + 4 * tx]);
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
  }
  if (slices > 1) {
    float4* dst = reinterpret_cast<float4*>(part + ((int64_t)blockIdx.x * slices + blockIdx.y) * kBig * kBig) + tid;
#pragma unroll
    for (int v = 0; v < 16; ++v)
      __stcg(dst + v * kThreads, make_float4(acc[v >> 1][4 * (v & 1)], acc[v >> 1][4 * (v & 1) + 1],
                                             acc[v >> 1][4 * (v & 1) + 2], acc[v >> 1][4 * (v & 1) + 3]));
    __threadfence();
    __syncthreads();
    if (tid == 0) {
      last = atomicAdd(tickets + blockIdx.x, 1u) == (unsigned)slices - 1;
      if (last) tickets[blockIdx.x] = 0;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const float4* src = reinterpret_cast<const float4*>(part + (int64_t)blockIdx.x * slices * kBig * kBig) + tid;
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
    for (int s = 0; s < slices; ++s)
#pragma unroll
      for (int v = 0; v < 16; ++v) {
        const float4 t = __ldcg(src + (int64_t)s * (kBig * kBig / 4) + v * kThreads);
        acc[v >> 1][4 * (v & 1)] += t.x, acc[v >> 1][4 * (v & 1) + 1] += t.y;
        acc[v >> 1][4 * (v & 1) + 2] += t.z, acc[v >> 1][4 * (v & 1) + 3] += t.w;
      }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int64_t p = p0 + 64 * (i >> 2) + 4 * ty + (i & 3);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int64_t q = q0 + 64 * (j >> 2) + 4 * tx + (j & 3);
      if (p < m && q <= p) M[p * ldm + q] = add ? M[p * ldm + q] + acc[i][j] : acc[i][j];
    }
  }
}

int64_t lower_tiles(int64_t m, int64_t ts) {
  const int64_t t = (m + ts - 1) / ts;
  return t * (t + 1) / 2;
}

}  // namespace

SimtPlan simt_plan_fp64(int64_t m, int64_t n) {
  SimtPlan p;
  // 16 x 16 tiles where 32 x 32 tiles with slices of 64 columns are fewer
  // than the SMs
  p.tile = lower_tiles(m, 32) * ((n + 63) / 64) < 152 ? 16 : 32;
  p.tiles = lower_tiles(m, p.tile);
  // Slices of at least one chunk (16 x 16 tiles) or 64 columns, as many as
  // give 8 units of work per SM: with fewer the last wave shows.
  const int64_t least = p.tile == 16 ? kKc : 64;
  int64_t s = std::min((8 * 152 + p.tiles - 1) / p.tiles, n / least);
  s = std::max<int64_t>(1, std::min<int64_t>(s, p.tile == 16 ? 8 : 32));
  p.kslice = ((n + s - 1) / s + kKc - 1) / kKc * kKc;
  p.slices = (int)((n + p.kslice - 1) / p.kslice);
  return p;
}

size_t simt_fp64_part_bytes(int64_t m) {
  const int64_t t32 = lower_tiles(m, 32), t16 = lower_tiles(m, 16);
  size_t b = 0;
  if (t32 < 152) b = sizeof(double) * t16 * 8 * 16 * 16;                        // 16 x 16 tiles, up to 8 slices
  if (t32 < 8 * 152) b = std::max(b, sizeof(double) * (8 * 152 + t32) * 32 * 32);  // 32 x 32 tiles
  return b;
}

int64_t simt_ticket_count(int64_t m) { return lower_tiles(m, 16); }

SimtPlan simt_plan_fp32(int64_t m, int64_t n) {
  SimtPlan p;
  p.tile = kBig;
  p.tiles = lower_tiles(m, kBig);
  // planes of all of A's columns, or of as many as keep both within 4 GB
  const int64_t most = std::max<int64_t>(2048, ((int64_t)1 << 29) / m / kKc * kKc);
  p.ldk = std::min((n + kKc - 1) / kKc * kKc, most);
  // one wave of two CTAs per SM where the tiles alone do not fill it (slices
  // of at least 64 columns)
  int64_t s = std::min<int64_t>(2 * 152 / p.tiles, p.ldk / 64);
  s = std::max<int64_t>(1, std::min<int64_t>(s, 64));
  p.kslice = ((p.ldk + s - 1) / s + kKc - 1) / kKc * kKc;
  p.slices = (int)((p.ldk + p.kslice - 1) / p.kslice);
  p.part_bytes = p.slices > 1 ? sizeof(float) * p.tiles * p.slices * kBig * kBig : 0;
  return p;
}

template <typename T>
cudaError_t launch_syrk_fp64(cudaStream_t st, int64_t m, int64_t n, const T* A, const double* D, double* M,
                             int64_t ldm, void* part, unsigned* tickets, const Scalars* sc) {
  const SimtPlan p = simt_plan_fp64(m, n);
  const dim3 grid((unsigned)p.tiles, (unsigned)p.slices);
  if (p.tile == 16)
    k_syrk_fp64<T, 16><<<grid, kThreads, 0, st>>>(m, n, A, D, M, ldm, p.kslice, p.slices, (double*)part, tickets, sc);
  else
    k_syrk_fp64<T, 32><<<grid, kThreads, 0, st>>>(m, n, A, D, M, ldm, p.kslice, p.slices, (double*)part, tickets, sc);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_syrk_fp32(cudaStream_t st, int64_t m, int64_t n, const T* A, const double* D, float* planes,
                             float* M, int64_t ldm, void* part, unsigned* tickets, const Scalars* sc, int* launches) {
  const SimtPlan p = simt_plan_fp32(m, n);
  float* Ap = planes + m * p.ldk;
  const dim3 pg((unsigned)((p.ldk + kThreads - 1) / kThreads),
                (unsigned)std::min<int64_t>((m + kPlaneRows - 1) / kPlaneRows, 4096));
  const dim3 grid((unsigned)p.tiles, (unsigned)p.slices);
  for (int64_t c0 = 0; c0 < n; c0 += p.ldk) {
    k_simt_planes<T><<<pg, kThreads, 0, st>>>(m, n, c0, p.ldk, A, D, planes, Ap, sc);
    k_syrk_fp32<<<grid, kThreads, 0, st>>>(m, p.ldk, planes, Ap, M, ldm, c0 > 0, p.kslice, p.slices, (float*)part,
                                           tickets, sc);
    *launches += 2;
  }
  return cudaGetLastError();
}

#define PDAS_INST(T)                                                                                               \
  template cudaError_t launch_syrk_fp64<T>(cudaStream_t, int64_t, int64_t, const T*, const double*, double*,       \
                                           int64_t, void*, unsigned*, const Scalars*);                             \
  template cudaError_t launch_syrk_fp32<T>(cudaStream_t, int64_t, int64_t, const T*, const double*, float*, float*, \
                                           int64_t, void*, unsigned*, const Scalars*, int*);
PDAS_INST(double)
PDAS_INST(float)
PDAS_INST(__nv_bfloat16)
#undef PDAS_INST

}  // namespace pdas
