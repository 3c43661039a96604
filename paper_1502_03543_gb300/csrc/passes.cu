// passes.cu -- the passes over A of a handle: A v (the right-hand side r = A x,
// the refinement's residual and operator, Section V) and A'u (ds = -A'dy), in
// FP64 or, for A stored as FP32 or BF16, in double-float on the FP32 pipes.
// Each is one launch, with what follows it in the solve fused in: the
// elementwise end of A'u (D w, dx, ds, the FP32 pairs for the next pass), the
// next search direction of the conjugate gradients before it, and the norm or
// the dot product after A v.
//
// Double-float.  GB300 issues FP64 at 1/64 of its FP32 rate, so an FP64
// multiply-add per entry of A bounds a pass at about 5x the time it takes to
// stream A from HBM.  The vector is split into FP32 pairs v = vh + vl (48
// significant bits), and each term is
//   a vh = ph + pe        exactly (FMA residual),
//   a v  ~ ph + (pe + a vl)        (relative error <= 2^-47),
// summed into an FP32 pair with Knuth's TwoSum on the high part; after at most
// 32 terms the pair is widened exactly (integer pipes) into an FP64
// accumulator.  The error stays within a few units of 2^-44 of sum |a v|.
// Two columns are carried per instruction (f32x2): 11 of them per pair, which
// issue in half the slots of 22 and leave the others for loads and
// conversions.
//
// All sums are deterministic: fixed partitions, fixed trees, and the last CTA of
// a column block (ticket) adds the row chunks in order.
//
// What bounds them: the FP64 passes the FP64 pipe (268M multiply-adds at 8192 x
// 32768: 430 us), the double-float passes the FP32 pipes and HBM alike (76 and
// 80 us there), both at small sizes the latency of two or three dependent
// round trips to L2.  So CTAs are sized for one wave at small sizes, rows are
// reduced by a reduce-scatter (a butterfly per row costs 5 FP64 additions a
// row and warp, 64 cycles each), the next rows are loaded during the work on
// the present ones, and nothing passes through memory between launches that need
// not.  Measured at 8192 x 32768 (BF16): A v in double-float 220 -> 165 us,
// A'u 193 + 16 -> 162 us, in FP64 523 -> 510 and 495 + 16 -> 478 us; a step of the
// conjugate gradients at 512 x 2048 is 4 launches and 45 us instead of 13
// launches, 4 fills and 95 us.
#include <algorithm>

#include "df_util.cuh"
#include "passes.cuh"
#include "reduce_util.cuh"

namespace pdas {

namespace {

// ---- pairs of FP32 numbers in one register pair --------------------------------
using f2 = unsigned long long;
__device__ __forceinline__ f2 pack2(float lo, float hi) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(f2 v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// (hi, lo) += a (vh + vl) for two columns; nvh = -vh, m1 = -1.
__device__ __forceinline__ void df_madd2(f2& hi, f2& lo, f2 a, f2 vh, f2 nvh, f2 vl, f2 m1) {
  const f2 nph = mul2(a, nvh);
  const f2 pl = fma2(a, vl, fma2(a, vh, nph));
  const f2 t = fma2(nph, m1, hi);    // hi + ph
  const f2 nbb = fma2(t, m1, hi);    // -(t - hi)
  const f2 d = fma2(add2(t, nbb), m1, hi);  // hi - (t - bb)
  const f2 f = fma2(nph, m1, nbb);   // ph - bb
  lo = add2(lo, add2(add2(d, f), pl));
  hi = t;
}
__device__ __forceinline__ void df_flush2(double& acc, f2& hi, f2& lo) {  // both lanes into one sum
  float a, b, c, d;
  unpack2(hi, a, b);
  unpack2(lo, c, d);
  const float t = a + b, bb = t - a;  // TwoSum of the high parts: two FP64 additions instead of four
  const float l = (c + d) + ((a - (t - bb)) + (b - bb));
  acc += widen_bits(__float_as_uint(t)) + widen_bits(__float_as_uint(l));
  hi = lo = 0ull;
}
__device__ __forceinline__ void df_flush2(double& a0, double& a1, f2& hi, f2& lo) {  // a sum per lane
  float a, b, c, d;
  unpack2(hi, a, b);
  unpack2(lo, c, d);
  a0 += widen_bits(__float_as_uint(a)) + widen_bits(__float_as_uint(c));
  a1 += widen_bits(__float_as_uint(b)) + widen_bits(__float_as_uint(d));
  hi = lo = 0ull;
}

// ---- 16 bytes of a row of A -------------------------------------------------------
template <typename T>
struct Row16;
template <>
struct Row16<double> {
  static constexpr int N = 2;
  using V = double2;
  __device__ static void widen(const V& v, double (&o)[2]) { o[0] = v.x, o[1] = v.y; }
};
template <>
struct Row16<float> {
  static constexpr int N = 4;
  using V = uint4;
  __device__ static void widen(const V& v, double (&o)[4]) {
    o[0] = widen_bits(v.x), o[1] = widen_bits(v.y), o[2] = widen_bits(v.z), o[3] = widen_bits(v.w);
  }
  __device__ static void pairs(const V& v, f2 (&o)[2]) {
    o[0] = pack2(__uint_as_float(v.x), __uint_as_float(v.y));
    o[1] = pack2(__uint_as_float(v.z), __uint_as_float(v.w));
  }
};
template <>
struct Row16<__nv_bfloat16> {
  static constexpr int N = 8;
  using V = uint4;
  __device__ static void widen(const V& v, double (&o)[8]) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      o[2 * i] = widen_bits(w[i] << 16);
      o[2 * i + 1] = widen_bits(w[i] & 0xffff0000u);
    }
  }
  __device__ static void pairs(const V& v, f2 (&o)[4]) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) o[i] = pack2(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xffff0000u));
  }
};
template <typename T>
__device__ __forceinline__ typename Row16<T>::V load16(const T* p) {
  return __ldg(reinterpret_cast<const typename Row16<T>::V*>(p));
}

constexpr int kWarps = kThreads / 32;

// f(16 bytes of row r, r, count) for r = r0, r0 + 8, ... < nr (rows of n elements
// from a), four rows being loaded while the four before them are worked on: with
// the loads of one group at a time the warps wait for memory for two thirds of
// the pass.
template <typename T, class F>
__device__ __forceinline__ void stream_rows(const T* a, int64_t n, int r0, int nr, F&& f) {
  using V = typename Row16<T>::V;
  constexpr int G = 4;
  V x[G], y[G];
#pragma unroll
  for (int g = 0; g < G; ++g)
    if (r0 + kWarps * g < nr) x[g] = load16(a + (int64_t)(r0 + kWarps * g) * n);
  int it = 0;
#pragma unroll 1
  for (int r = r0; r < nr; r += kWarps * G) {
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const int rn = r + kWarps * (G + g);
      if (rn < nr) y[g] = load16(a + (int64_t)rn * n);
    }
#pragma unroll
    for (int g = 0; g < G; ++g)
      if (r + kWarps * g < nr) f(x[g], r + kWarps * g, it++);
#pragma unroll
    for (int g = 0; g < G; ++g) x[g] = y[g];
  }
}

constexpr int64_t kMaxRows = 512;  // rows of a chunk (its vector is held in shared memory)
constexpr int kScalarCols = 4;     // columns per thread where rows are not 16-byte aligned

// The chunk's vector in shared memory: per row {h, h, l, l} and {-h, -h} (the
// double-float operands of both columns of a pair), or the FP64 value.
struct PassTSmem {
  union {
    struct {
      float4 hl[kMaxRows];
      float2 nh[kMaxRows];
    } df;
    double v[kMaxRows];
  };
  double red[kWarps][256];  // column sums of the warps
  double mx[kWarps];
  int last;
};

// Elementwise end of A'u for column j.
__device__ __forceinline__ void finish_column(int64_t j, double w, int mode, const double* x, const double* D,
                                              double* out0, double* out1, double* out2, float* ph, float* pl,
                                              const double* rd) {
  if (mode == 0) {
    out0[j] = w;
  } else if (mode == 1) {
    const double ds = rd ? rd[j] - w : -w;
    out0[j] = D[j] * (-ds) - x[j];  // dx = D(-ds) - x
    out1[j] = ds;
    if (out2) out2[j] = w;
  } else {
    const double u = D[j] * w;
    if (out0) out0[j] = u;
    if (out2) out2[j] = w;
    if (ph) {
      const float2 q = df_split(u);
      ph[j] = q.x, pl[j] = q.y;
    }
  }
}

// A'u: CTA (cb, ch) sums rows ch rows .. of 32 V columns; warp w takes every
// eighth row, the warps are added in order through shared memory, and the last
// CTA of a column block adds the chunks in order and runs finish_column.  VEC:
// rows are 16-byte aligned and thread l owns V = 16 / sizeof(T) consecutive
// columns; else columns l + 32 k, k < 4, by single loads.
template <typename T, bool DF, bool VEC>
__global__ void __launch_bounds__(kThreads, 3) k_pass_t(int64_t m, int64_t n, const T* __restrict__ A, PassTSrc src,
                                                     int64_t rows, int chunks, double* part, double* maxpart,
                                                     unsigned* ctickets, int mode, const double* __restrict__ x,
                                                     const double* __restrict__ D, double* out0, double* out1,
                                                     double* out2, float* ph, float* pl, Scalars* sc,
                                                     const double* __restrict__ rd) {
  constexpr int V = VEC ? Row16<T>::N : kScalarCols;
  __shared__ PassTSmem sm;
  if (failed(sc)) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t pbeg = (int64_t)blockIdx.y * rows;
  const int nr = (int)(m - pbeg < rows ? m - pbeg : rows);
  // the chunk of the vector
  {
    constexpr int PER = (int)(kMaxRows / kThreads);
    double u[PER], p[PER];  // all loads in flight before the sum below
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int r = tid + k * kThreads;
      u[k] = r < nr ? src.u[pbeg + r] : 0.0;
      p[k] = (r < nr && src.p && !src.first) ? src.p[pbeg + r] : 0.0;
    }
    if (src.p) {  // each warp forms rz by itself
      double rz = 0.0;
      for (int i = lane; i < src.nrz; i += 32) rz += src.rz_part[i];
      rz = warp_sum(rz);
      if (tid == 0 && blockIdx.x == 0 && blockIdx.y == 0) sc->rz[src.par] = rz;
      if (!src.first) {
        const double beta = rz / sc->rz[1 - src.par];
#pragma unroll
        for (int k = 0; k < PER; ++k) u[k] = u[k] + beta * p[k];
      }
    }
    double mx = 0.0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int r = tid + k * kThreads;
      if (r >= nr) continue;
      if (src.p && blockIdx.x == 0) src.p_new[pbeg + r] = u[k];
      if (src.absmax) {
        const double a = fabs(u[k]);
        mx = (a == a) ? fmax(mx, a) : INFINITY;
      }
      if constexpr (DF) {
        const float2 q = df_split(u[k]);
        sm.df.hl[r] = make_float4(q.x, q.x, q.y, q.y);
        sm.df.nh[r] = make_float2(-q.x, -q.x);
      } else {
        sm.v[r] = u[k];
      }
    }
    if (src.absmax && blockIdx.x == 0) {
      mx = warp_max(mx);
      if (lane == 0) sm.mx[warp] = mx;
    }
  }
  __syncthreads();
  if (src.absmax && blockIdx.x == 0 && tid == 0) {
    double g = 0.0;
    for (int w = 0; w < kWarps; ++w) g = fmax(g, sm.mx[w]);
    maxpart[blockIdx.y] = g;
  }
  const int64_t j0 = (int64_t)blockIdx.x * (32 * V);
  double acc[V];
#pragma unroll
  for (int k = 0; k < V; ++k) acc[k] = 0.0;
  if constexpr (VEC) {
    const int64_t j = j0 + (int64_t)lane * V;
    if (j < n) {
      const T* a = A + pbeg * n + j;
      if constexpr (DF) {
        const f2 m1 = pack2(-1.f, -1.f);
        f2 hi[V / 2], lo[V / 2];
#pragma unroll
        for (int k = 0; k < V / 2; ++k) hi[k] = lo[k] = 0ull;
        stream_rows(a, n, warp, nr, [&](const typename Row16<T>::V& x, int r, int it) {
          f2 v[V / 2];
          Row16<T>::pairs(x, v);
          const float4 q = sm.df.hl[r];
          const float2 g = sm.df.nh[r];
          const f2 vh = pack2(q.x, q.y), vl = pack2(q.z, q.w), nvh = pack2(g.x, g.y);
#pragma unroll
          for (int k = 0; k < V / 2; ++k) df_madd2(hi[k], lo[k], v[k], vh, nvh, vl, m1);
          if ((it & 31) == 31 || r + kWarps >= nr) {
#pragma unroll
            for (int k = 0; k < V / 2; ++k) df_flush2(acc[2 * k], acc[2 * k + 1], hi[k], lo[k]);
          }
        });
      } else {
        stream_rows(a, n, warp, nr, [&](const typename Row16<T>::V& x, int r, int) {
          double v[V];
          Row16<T>::widen(x, v);
          const double u = sm.v[r];
#pragma unroll
          for (int k = 0; k < V; ++k) acc[k] = fma(v[k], u, acc[k]);
        });
      }
    }
  } else {
    const T* a = A + pbeg * n + j0 + lane;
    bool in[V];
#pragma unroll
    for (int k = 0; k < V; ++k) in[k] = j0 + lane + 32 * k < n;
    if constexpr (DF) {
      float hi[V], lo[V];
#pragma unroll
      for (int k = 0; k < V; ++k) hi[k] = lo[k] = 0.f;
      int it = 0;
#pragma unroll 4
      for (int r = warp; r < nr; r += kWarps) {
        const float4 q = sm.df.hl[r];
#pragma unroll
        for (int k = 0; k < V; ++k)
          df_madd(hi[k], lo[k], in[k] ? widen32(a[(int64_t)r * n + 32 * k]) : 0.f, q.x, q.z);
        if ((++it & 31) == 0) {
#pragma unroll
          for (int k = 0; k < V; ++k) df_flush(acc[k], hi[k], lo[k]);
        }
      }
#pragma unroll
      for (int k = 0; k < V; ++k) df_flush(acc[k], hi[k], lo[k]);
    } else {
#pragma unroll 4
      for (int r = warp; r < nr; r += kWarps) {
        const double u = sm.v[r];
#pragma unroll
        for (int k = 0; k < V; ++k) acc[k] = fma(in[k] ? widen(a[(int64_t)r * n + 32 * k]) : 0.0, u, acc[k]);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < V; ++k) sm.red[warp][VEC ? lane * V + k : lane + 32 * k] = acc[k];
  __syncthreads();
  const int64_t j = j0 + tid;
  const bool mine = tid < 32 * V && j < n;
  double w = 0.0;
  if (mine) {
#pragma unroll
    for (int k = 0; k < kWarps; ++k) w += sm.red[k][tid];
  }
  if (chunks > 1) {
    if (mine) __stcg(part + (int64_t)blockIdx.y * n + j, w);
    __threadfence();
    __syncthreads();
    if (tid == 0) {
      sm.last = atomicAdd(ctickets + blockIdx.x, 1u) == (unsigned)chunks - 1;
      if (sm.last) ctickets[blockIdx.x] = 0;
    }
    __syncthreads();
    if (!sm.last) return;
    __threadfence();
    if (mine) {
      w = 0.0;
#pragma unroll 8
      for (int c = 0; c < chunks; ++c) w += __ldcg(part + (int64_t)c * n + j);
    }
  }
  if (mine) finish_column(j, w, mode, x, D, out0, out1, out2, ph, pl, rd);
  if (src.absmax && blockIdx.x == 0 && tid == 0) {
    double g = 0.0;
    for (int c = 0; c < chunks; ++c) g = fmax(g, __ldcg(maxpart + c));
    sc->dynorm = g;
  }
}

// v[0 .. R - 1] summed over the warp by halving exchanges: lane l returns the
// sum of entry l / (32 / R).  R - 1 + log2(32 / R) additions.
template <int R>
__device__ __forceinline__ double warp_sum_rows(double (&v)[R], int lane) {
  int off = 16;
#pragma unroll
  for (int h = R / 2; h >= 1; h >>= 1, off >>= 1) {
    const bool up = lane & off;
#pragma unroll
    for (int i = 0; i < R / 2; ++i)
      if (i < h) {
        const double keep = up ? v[i + h] : v[i], give = up ? v[i] : v[i + h];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, give, off);
      }
  }
  double s = v[0];
  for (; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  return s;
}

// A v: R rows per CTA, every thread a strided slice of their columns.
template <typename T, int R, bool DF>
__global__ void __launch_bounds__(kThreads, DF ? 2 : sizeof(T) == 8 ? 5 : 3) k_pass(int64_t m, int64_t n, const T* __restrict__ A,
                                                   const double* __restrict__ v, const float* __restrict__ vh,
                                                   const float* __restrict__ vl, const double* __restrict__ base,
                                                   double* __restrict__ out, int vec, double* part,
                                                   unsigned* tickets, Scalars* sc, int norm_slot,
                                                   const double* __restrict__ dot) {
  __shared__ double sm[32];
  __shared__ double rsum[kWarps][R];
  if (failed(sc)) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t p0 = (int64_t)blockIdx.x * R;
  const int nr = (int)(m - p0 < R ? m - p0 : R);
  const T* rows[R];
#pragma unroll
  for (int r = 0; r < R; ++r) rows[r] = A + (p0 + (r < nr ? r : 0)) * n;  // (a row past m reads the CTA's first and is dropped)
  double acc[R];
#pragma unroll
  for (int r = 0; r < R; ++r) acc[r] = 0.0;
  constexpr int V = Row16<T>::N;
  if (vec) {
    if constexpr (DF) {
      const f2 m1 = pack2(-1.f, -1.f);
      f2 hi[R], lo[R];
#pragma unroll
      for (int r = 0; r < R; ++r) hi[r] = lo[r] = 0ull;
      int it = 0;
      constexpr int64_t step = (int64_t)kThreads * V;
      typename Row16<T>::V a[R], b[R];  // the next step's rows are loaded during this one's work
      int64_t j = (int64_t)tid * V;
      if (j < n) {
#pragma unroll
        for (int r = 0; r < R; ++r) a[r] = load16(rows[r] + j);
      }
#pragma unroll 1
      for (; j < n; j += step) {
        float4 qh[V / 4], ql[V / 4];
#pragma unroll
        for (int k = 0; k < V / 4; ++k) {
          qh[k] = __ldg(reinterpret_cast<const float4*>(vh + j) + k);
          ql[k] = __ldg(reinterpret_cast<const float4*>(vl + j) + k);
        }
        if (j + step < n) {
#pragma unroll
          for (int r = 0; r < R; ++r) b[r] = load16(rows[r] + j + step);
        }
        f2 h2[V / 2], l2[V / 2], n2[V / 2];
#pragma unroll
        for (int k = 0; k < V / 4; ++k) {
          h2[2 * k] = pack2(qh[k].x, qh[k].y), h2[2 * k + 1] = pack2(qh[k].z, qh[k].w);
          n2[2 * k] = pack2(-qh[k].x, -qh[k].y), n2[2 * k + 1] = pack2(-qh[k].z, -qh[k].w);
          l2[2 * k] = pack2(ql[k].x, ql[k].y), l2[2 * k + 1] = pack2(ql[k].z, ql[k].w);
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
          f2 q[V / 2];
          Row16<T>::pairs(a[r], q);
#pragma unroll
          for (int k = 0; k < V / 2; ++k) df_madd2(hi[r], lo[r], q[k], h2[k], n2[k], l2[k], m1);
          a[r] = b[r];
        }
        if ((++it & 7) == 0 || j + step >= n) {  // 4 (BF16) or 2 terms per lane and step
#pragma unroll
          for (int r = 0; r < R; ++r) df_flush2(acc[r], hi[r], lo[r]);
        }
      }
    } else {
      // FP64-stored A: 4 rows x 16 bytes a step are 20 instructions' work, and
      // warps hide the loads better than a second buffer does (45 against 57 us
      // at 2048 x 8192)
      constexpr bool kAhead = sizeof(T) < 8;
      constexpr int64_t step = (int64_t)kThreads * V;
      typename Row16<T>::V a[R], b[R];
      int64_t j = (int64_t)tid * V;
      if (kAhead && j < n) {
#pragma unroll
        for (int r = 0; r < R; ++r) a[r] = load16(rows[r] + j);
      }
#pragma unroll 1
      for (; j < n; j += step) {
        double vv[V];
#pragma unroll
        for (int k = 0; k < V; k += 2) {
          const double2 q = __ldg(reinterpret_cast<const double2*>(v + j + k));
          vv[k] = q.x, vv[k + 1] = q.y;
        }
        if (!kAhead) {
#pragma unroll
          for (int r = 0; r < R; ++r) a[r] = load16(rows[r] + j);
        } else if (j + step < n) {
#pragma unroll
          for (int r = 0; r < R; ++r) b[r] = load16(rows[r] + j + step);
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
          double w[V];
          Row16<T>::widen(a[r], w);
#pragma unroll
          for (int k = 0; k < V; ++k) acc[r] = fma(w[k], vv[k], acc[r]);
          if (kAhead) a[r] = b[r];
        }
      }
    }
  } else {
    if constexpr (DF) {
      float hi[R], lo[R];
#pragma unroll
      for (int r = 0; r < R; ++r) hi[r] = lo[r] = 0.f;
      int it = 0;
#pragma unroll 2
      for (int64_t j = tid; j < n; j += kThreads) {
        const float h = __ldg(vh + j), l = __ldg(vl + j);
#pragma unroll
        for (int r = 0; r < R; ++r) df_madd(hi[r], lo[r], widen32(rows[r][j]), h, l);
        if ((++it & 31) == 0) {
#pragma unroll
          for (int r = 0; r < R; ++r) df_flush(acc[r], hi[r], lo[r]);
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r) df_flush(acc[r], hi[r], lo[r]);
    } else {
#pragma unroll 2
      for (int64_t j = tid; j < n; j += kThreads) {
        const double vj = __ldg(v + j);
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r] = fma(widen(rows[r][j]), vj, acc[r]);
      }
    }
  }
  const double s = warp_sum_rows<R>(acc, lane);
  constexpr int W = 32 / R;  // lanes per row
  if (lane % W == 0) rsum[warp][lane / W] = s;
  __syncthreads();
  double mx = 0.0, pq = 0.0;
  if (tid < R && tid < nr) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) t += rsum[w][tid];
    const int64_t p = p0 + tid;
    const double o = base ? base[p] - t : t;
    out[p] = o;
    mx = isfinite(o) ? fabs(o) : INFINITY;
    if (dot) pq = dot[p] * o;
  }
  if (norm_slot < 0 && !dot) return;
  if (warp == 0) {
    if (dot) mx = warp_sum(pq);
    else mx = warp_max(mx);
    if (lane == 0) part[blockIdx.x] = mx;
  }
  if (!last_block(tickets + T_NORM)) return;
  const double g = dot ? combine<0>(part, gridDim.x, sm) : combine<1>(part, gridDim.x, sm);
  if (tid == 0) {
    if (dot) sc->dot_b = g;
    else if (norm_slot == 0) sc->rnorm = g;
    else sc->rho_norm = g;
    tickets[T_NORM] = 0;
  }
}

__global__ void k_split_pairs(int64_t n, const double* __restrict__ v, float* __restrict__ ph, float* __restrict__ pl) {
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
    const float2 q = df_split(v[j]);
    ph[j] = q.x, pl[j] = q.y;
  }
}

}  // namespace

PassTPlan pass_t_plan(int64_t m, int64_t n, int elem_bytes, bool vec) {
  PassTPlan p;
  const int64_t cols = 32 * (vec ? 16 / elem_bytes : kScalarCols);
  p.cblocks = (n + cols - 1) / cols;
  // One wave of 4 CTAs per SM while that leaves 32 rows or more to a chunk (4 a
  // warp, all loads in flight at once); chunks of at most 512 rows beyond.
  const int64_t one_wave = std::max<int64_t>(1, 4 * 152 / p.cblocks);
  int64_t rows = std::max<int64_t>(32, (m + one_wave - 1) / one_wave);
  rows = std::min<int64_t>(kMaxRows, (rows + kWarps - 1) / kWarps * kWarps);
  p.chunks = (int)((m + rows - 1) / rows);
  p.rows = rows;
  return p;
}

int64_t pass_t_part_doubles(int64_t m, int64_t n, int elem_bytes) {
  return std::max(pass_t_plan(m, n, elem_bytes, true).chunks, pass_t_plan(m, n, elem_bytes, false).chunks) * n;
}

int64_t pass_t_tickets(int64_t n) { return (n + 63) / 64 + 1; }

template <typename T>
cudaError_t launch_pass_t(cudaStream_t st, int64_t m, int64_t n, const T* A, bool df, const PassTSrc& src,
                          double* part, double* maxpart, unsigned* ctickets, int mode, const double* x, const double* D,
                          double* out0, double* out1, double* out2, float* pairs, Scalars* sc, const double* rd) {
  const bool vec = vec_aligned(A, n);
  const PassTPlan p = pass_t_plan(m, n, sizeof(T), vec);
  const dim3 grid((unsigned)p.cblocks, (unsigned)p.chunks);
  float* pl = pairs ? pairs + pairs_pitch(n) : nullptr;
#define PASS_T(DF, VEC)                                                                                         \
  k_pass_t<T, DF, VEC><<<grid, kThreads, 0, st>>>(m, n, A, src, p.rows, p.chunks, part, maxpart, ctickets, mode, x, \
                                                  D, out0, out1, out2, pairs, pl, sc, rd)
  if constexpr (sizeof(T) < 8) {
    if (df) {
      if (vec) PASS_T(true, true);
      else PASS_T(true, false);
      return cudaGetLastError();
    }
  }
  if (vec) PASS_T(false, true);
  else PASS_T(false, false);
#undef PASS_T
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_pass(cudaStream_t st, int64_t m, int64_t n, const T* A, const double* v, const float* pairs,
                        const double* base, double* out, double* part, unsigned* tickets, Scalars* sc, int norm_slot,
                        const double* dot) {
  constexpr int R = 4;  // (8 rows halve the reads of the vector but leave one CTA per SM: 209 against 165 us at 8192 x 32768)
  const int64_t grid = (m + R - 1) / R;
  if ((norm_slot >= 0 || dot) && grid > kPartMax) return cudaErrorInvalidConfiguration;
  const int vec = vec_aligned(A, n) && (uintptr_t)v % 16 == 0;
  const float* vl = pairs ? pairs + pairs_pitch(n) : nullptr;
#define PASS(DF)                                                                                                 \
  k_pass<T, R, DF><<<(unsigned)grid, kThreads, 0, st>>>(m, n, A, v, pairs, vl, base, out, vec, part, tickets, sc, \
                                                         norm_slot, dot)
  if constexpr (sizeof(T) < 8) {
    if (pairs) {
      PASS(true);
      return cudaGetLastError();
    }
  }
  PASS(false);
#undef PASS
  return cudaGetLastError();
}

cudaError_t launch_split_pairs(cudaStream_t st, int64_t n, const double* v, float* pairs) {
  k_split_pairs<<<grid_for(n, 4), kThreads, 0, st>>>(n, v, pairs, pairs + pairs_pitch(n));
  return cudaGetLastError();
}

#define PDAS_INST(T)                                                                                                 \
  template cudaError_t launch_pass_t<T>(cudaStream_t, int64_t, int64_t, const T*, bool, const PassTSrc&, double*,    \
                                        double*, unsigned*, int, const double*, const double*, double*, double*,     \
                                        double*, float*, Scalars*, const double*);                                   \
  template cudaError_t launch_pass<T>(cudaStream_t, int64_t, int64_t, const T*, const double*, const float*,         \
                                      const double*, double*, double*, unsigned*, Scalars*, int, const double*);
PDAS_INST(double)
PDAS_INST(float)
PDAS_INST(__nv_bfloat16)
#undef PDAS_INST

}  // namespace pdas
