// trsv_blk.cu -- the two triangular solves of the normal equations with the
// FP32 factor of the mixed forms (Section V-A: L z = A x, then L' dy = z),
// in 128-row blocks.  The factor launch leaves U_b = L_bb^{-T} for every
// diagonal tile, so a block applies U_b' (forward) or U_b (backward) as a
// 128 x 128 product instead of a 128-step substitution; the dependency chain
// from block to block is then one tile product with the newest neighbour
// block and one with U_b.  The FP32 factor is a preconditioner here (the
// mixed forms refine in FP64 afterwards), so the explicit inverse of each
// diagonal tile is accurate enough; the plain FP64 form keeps substitution.
//
// One launch per solve, in clusters of 8 blocks.  Clusters take 8 block rows at
// a time from a ticket counter and wait (bounded: 2 s, or the handle's own limit)
// for the solution blocks they depend on, which were handed out earlier: no
// deadlock.  Inside a cluster a block writes its solution straight into the
// shared memory of the blocks behind it (st.async on their mbarriers).  Between
// clusters it goes through L2: a solution vector not yet written holds an all-ones
// bit pattern (a value the solves cannot produce: each entry is an FP32 sum
// widened to FP64, whose low 29 bits are zero), and one warp of the consumer polls
// the entries until none holds it.  The forward solve fills the backward
// solve's output with the pattern and the backward solve refills the forward
// one's as it reads it, so no fill runs between the launches.
//
// What bounds a solve is the latency of its chain of nb links.  Per link: the
// hand-off, a 128 x 128 product whose tile is already in registers, a
// reduce-scatter over lanes, and the product with U_b, whose entries every
// thread holds in registers, too.  Measured at m = 2048 (16 links), forward and
// backward: 48 and 26 us with every warp of every waiting block polling L2,
// 29 and 37 us with one warp polling and U_b in registers, 20-27 and 29 us in
// clusters; at m = 8192 187 and 106, now 101 and 125 us.
//
// The conjugate gradients of the refinement ride along: the forward solve's
// block first takes its rows of the step (dy += a p, rho -= a q) and leaves the
// largest magnitudes, which the backward solve's last block combines while it
// waits; the backward solve leaves the partial sums of rho'z.
#include "reduce_util.cuh"
#include "sync_util.cuh"
#include "tc_util.cuh"
#include "tile_core.cuh"

namespace pdas {

namespace {

constexpr int kClu = 8;  // blocks per cluster (the portable limit)

struct TrsvSmem {
  __align__(16) float zc[kClu][kBig];  // solution blocks of this cluster
  __align__(16) float zs[2][kBig];     // the solution block in use of another cluster, and the next
  __align__(16) float rhs[kBig];
  __align__(16) float red[8][kBig];
  unsigned long long bar[kClu];  // arrival of zc
  double mx[8][2];
  unsigned cluster;
  int ok[2];
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t peer_addr(const void* p, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(tc::smem_u32(p)), "r"(rank));
  return r;
}

// This block's place in the order of the chain.  All threads; sets up the
// arrival barriers of the blocks before it in its cluster.
__device__ __forceinline__ int64_t chain_position(TrsvSmem& sm, unsigned* ticket) {
  const uint32_t rank = cluster_rank();
  if (threadIdx.x == 0) {
    for (uint32_t k = 0; k < rank; ++k) {
      tc::mbar_init(tc::smem_u32(&sm.bar[k]), 1);
      tc::mbar_expect_tx(tc::smem_u32(&sm.bar[k]), sizeof(float) * kBig);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (rank == 0) {
      const unsigned t = atomicAdd(ticket, 1u);
      if (t == gridDim.x / kClu - 1) *ticket = 0;  // every cluster has its own
      for (uint32_t k = 0; k < kClu; ++k)
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(peer_addr(&sm.cluster, k)), "r"(t) : "memory");
    }
  }
  cluster_barrier();
  return (int64_t)sm.cluster * kClu + rank;
}

// The solution entry of row i = tid / 2 (in both lanes of a pair) to the blocks
// behind this one in its cluster, of `behind` in all.
__device__ __forceinline__ void send_entry(TrsvSmem& sm, float v, int64_t behind) {
  const uint32_t rank = cluster_rank(), i = threadIdx.x >> 1;
  for (uint32_t k = rank + 1 + (threadIdx.x & 1); k < kClu && (int64_t)(k - rank) <= behind; k += 2)
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(
                     peer_addr(&sm.zc[rank][i], k)),
                 "r"(__float_as_uint(v)), "r"(peer_addr(&sm.bar[rank], k))
                 : "memory");
}

// No block leaves while another may write to its shared memory: it has waited
// for all blocks before it, or (ok false) gives what they may have sent 50 us
// to land once they are all done.
__device__ __forceinline__ void leave(TrsvSmem& sm, bool ok) {
  cluster_barrier();
  if (ok) return;
  const uint64_t t0 = global_ns();
  for (uint32_t k = 0; k < cluster_rank(); ++k)
    while (!tc::mbar_try(tc::smem_u32(&sm.bar[k]), 0) && global_ns() - t0 < 50000) {
    }
}

// Bounded wait for block k of this cluster; false on a timeout or a failed status.
__device__ __forceinline__ bool wait_peer(TrsvSmem& sm, int k, Scalars* sc) {
  const uint32_t bar = tc::smem_u32(&sm.bar[k]);
  if (tc::mbar_try(bar, 0)) return true;
  const uint64_t t0 = global_ns(), limit = wait_limit_ns(sc);
  for (;;) {
    if (tc::mbar_try(bar, 0)) return true;
    if (dev_failed(sc)) return false;
    if (global_ns() - t0 > limit) {
      atomicCAS(&sc->status, 0, (int)PDAS_ERR_TIMEOUT);
      return false;
    }
  }
}

// 16 per-lane partial sums reduced across the warp by exchanging halves:
// lane l ends with the total of entry (l >> 1) & 15 (16 shuffles in all).
__device__ __forceinline__ float reduce16(float (&v)[16], int lane) {
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const bool up = lane & 16;
    const float keep = up ? v[k + 8] : v[k], send = up ? v[k] : v[k + 8];
    v[k] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const bool up = lane & 8;
    const float keep = up ? v[k + 4] : v[k], send = up ? v[k] : v[k + 4];
    v[k] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const bool up = lane & 4;
    const float keep = up ? v[k + 2] : v[k], send = up ? v[k] : v[k + 2];
    v[k] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
  }
  {
    const bool up = lane & 2;
    const float keep = up ? v[1] : v[0], send = up ? v[0] : v[1];
    v[0] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
  }
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

constexpr unsigned long long kUnset = ~0ull;  // a solution entry not yet written

__device__ __forceinline__ double ld_relaxed_f64(const double* p) {
  double v;
  asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed_f64(double* p, double v) {
  asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" ::"l"(p), "d"(v) : "memory");
}

// The warp waits (bounded) until none of the entries p[4 lane .. + 3] (those
// below left; the others read as 0) holds kUnset.  Returns false on a timeout
// or a failed status.  far: the block is not next in the chain and polls less often.
__device__ __forceinline__ bool poll_entries(const double* p, int left, float (&out)[4], bool far, Scalars* sc) {
  const int lane = threadIdx.x & 31;
  const uint64_t t0 = global_ns(), limit = wait_limit_ns(sc);
  for (;;) {
    bool mine = true;
    const bool failed = dev_failed(sc);  // (in flight with the entries)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const double v = 4 * lane + k < left ? ld_relaxed_f64(p + 4 * lane + k) : 0.0;
      mine = mine && __double_as_longlong(v) != (long long)kUnset;
      out[k] = (float)v;
    }
    if (__all_sync(0xffffffffu, mine)) return true;
    if (__any_sync(0xffffffffu, failed)) return false;
    if (__any_sync(0xffffffffu, global_ns() - t0 > limit)) {
      if (lane == 0) atomicCAS(&sc->status, 0, (int)PDAS_ERR_TIMEOUT);
      return false;
    }
    if (far) __nanosleep(200);
  }
}

// Warp 0 fetches solution block k of v (m entries) into sm.zs[buf]; the others
// learn the outcome behind the caller's next barrier.
__device__ __forceinline__ void fetch_block(TrsvSmem& sm, const double* v, int64_t m, int64_t k, int buf, bool far,
                                            Scalars* sc) {
  if (threadIdx.x < 32) {
    const int64_t left = m - k * kBig;
    float e[4];
    const bool ok = poll_entries(v + k * kBig, left < kBig ? (int)left : kBig, e, far, sc);
    *reinterpret_cast<float4*>(&sm.zs[buf][4 * threadIdx.x]) = make_float4(e[0], e[1], e[2], e[3]);
    if (threadIdx.x == 0) sm.ok[buf] = ok;
  }
}

__device__ __forceinline__ float dot64(const float4 (&u)[16], const float* v) {  // v: 64 floats in shared memory
  float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const float4 q = *reinterpret_cast<const float4*>(v + 4 * k);
    s[0] = fmaf(u[k].x, q.x, s[0]), s[1] = fmaf(u[k].y, q.y, s[1]);
    s[2] = fmaf(u[k].z, q.z, s[2]), s[3] = fmaf(u[k].w, q.w, s[3]);
  }
  return (s[0] + s[1]) + (s[2] + s[3]);
}

// L z = v: z_b = U_b' (v_b - sum_{j<b} L_bj z_j).  upd: v takes a step of the
// conjugate gradients first (CgStep) and the largest magnitudes of v and dy go
// to npart.  fill: the backward solve's output.
template <bool UPD>
__device__ __forceinline__ bool trsv_lower_block(TrsvSmem& sm, int64_t b, int64_t nblk, int64_t m, int64_t ldm,
                                                 const float* __restrict__ L, const float* __restrict__ Uinv,
                                                 double* v, double* z, double* fill, const CgStep& upd, double* npart,
                                                 Scalars* sc) {
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int64_t own = b - cluster_rank();  // the cluster's first block
  if (b >= nblk) return true;
  if (__syncthreads_or(dev_failed(sc))) return false;
  const int64_t r0 = b * kBig;
  const int rb = (int)(m - r0 < kBig ? m - r0 : kBig);
  if (tid < rb) fill[r0 + tid] = __longlong_as_double((long long)kUnset);
  const int myrow = 16 * w + ((lane >> 1) & 15);  // the row this lane pair finishes after the reduction
  float vmine = 0.f;
  double mr = 0.0, my = 0.0;
  if ((lane & 1) == 0 && myrow < rb) {
    double r = v[r0 + myrow];
    if constexpr (UPD) {
      double a, y = upd.dy[r0 + myrow];
      if (cg_step_length(*upd.rz, sc->dot_b, &a)) {
        y = y + a * upd.p[r0 + myrow];
        r = r - a * upd.q[r0 + myrow];
        upd.dy[r0 + myrow] = y;
        v[r0 + myrow] = r;
      }
      mr = r == r ? fabs(r) : INFINITY;
      my = y == y ? fabs(y) : INFINITY;
    }
    vmine = (float)r;
  }
  if constexpr (UPD) {
    mr = warp_max(mr);
    my = warp_max(my);
    if (lane == 0) sm.mx[w][0] = mr, sm.mx[w][1] = my;
    __syncthreads();
    if (tid == 0) {
      for (int k = 0; k < 8; ++k) mr = fmax(mr, sm.mx[k][0]), my = fmax(my, sm.mx[k][1]);
      npart[2 * b] = mr, npart[2 * b + 1] = my;
    }
  }
  float part[16];
#pragma unroll
  for (int rr = 0; rr < 16; ++rr) part[rr] = 0.f;
  bool ok = true;
  // Two buffers: tile j + 1 is on its way while tile j waits for its block of z.
  // A tile is rows 16 w .. 16 w + 15, columns 4 lane .. + 3; "tile b" is this
  // thread's share of U_b: column c = tid / 2, rows 64 (tid % 2) .. + 63.
  float4 lv[2][16];
  auto fetch = [&](int64_t j, float4 (&t)[16]) {
    if (j < b) {
#pragma unroll
      for (int rr = 0; rr < 16; ++rr) {
        const int64_t row = r0 + 16 * w + rr;
        t[rr] = row < m ? __ldg(reinterpret_cast<const float4*>(L + row * ldm + j * kBig + 4 * lane))
                        : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    } else {
      const float* Ub = Uinv + (int64_t)b * kBig * kBig + (int64_t)(64 * (tid & 1)) * kBig + (tid >> 1);
#pragma unroll
      for (int r = 0; r < 16; ++r)
        t[r] = make_float4(__ldg(Ub + 4 * r * kBig), __ldg(Ub + (4 * r + 1) * kBig), __ldg(Ub + (4 * r + 2) * kBig),
                           __ldg(Ub + (4 * r + 3) * kBig));
    }
  };
  auto consume = [&](int64_t j, const float4 (&t)[16]) {
    const float* zj = sm.zs[j & 1];
    if (j >= own) {
      if (__syncthreads_or(!wait_peer(sm, (int)(j - own), sc))) return false;
      zj = sm.zc[j - own];
    } else {
      fetch_block(sm, z, m, j, j & 1, j + 3 < own, sc);
      __syncthreads();
      if (!sm.ok[j & 1]) return false;
    }
    const float4 q = *reinterpret_cast<const float4*>(&zj[4 * lane]);
#pragma unroll
    for (int rr = 0; rr < 16; ++rr)
      part[rr] = fmaf(t[rr].x, q.x, fmaf(t[rr].y, q.y, fmaf(t[rr].z, q.z, fmaf(t[rr].w, q.w, part[rr]))));
    return true;
  };
  fetch(0, lv[0]);
  for (int64_t j = 0; j < b && ok; j += 2) {
    fetch(j + 1, lv[1]);
    ok = consume(j, lv[0]);
    if (!ok || j + 1 >= b) break;
    fetch(j + 2, lv[0]);
    ok = consume(j + 1, lv[1]);
  }
  if (!ok) return false;  // a wait gave up: the status says why
  const float tot = reduce16(part, lane);
  if ((lane & 1) == 0) sm.rhs[myrow] = myrow < rb ? vmine - tot : 0.f;
  __syncthreads();
  const float* half = &sm.rhs[64 * (tid & 1)];
  float s = (b & 1) ? dot64(lv[1], half) : dot64(lv[0], half);  // z_c = sum_r U_rc rhs_r
  s += __shfl_xor_sync(0xffffffffu, s, 1);
  send_entry(sm, s, nblk - 1 - b);
  if ((tid & 1) == 0 && (tid >> 1) < rb) st_relaxed_f64(z + r0 + (tid >> 1), (double)s);
  return true;
}

template <bool UPD>
__global__ void __launch_bounds__(kThreads, 1) k_trsv_lower_blk(int64_t m, int64_t ldm, int64_t nblk,
                                                                const float* __restrict__ L,
                                                                const float* __restrict__ Uinv, double* v, double* z,
                                                                double* fill, CgStep upd, double* npart,
                                                                unsigned* ticket, Scalars* sc) {
  __shared__ TrsvSmem sm;
  const int64_t b = chain_position(sm, ticket);
  leave(sm, trsv_lower_block<UPD>(sm, b, nblk, m, ldm, L, Uinv, v, z, fill, upd, npart, sc));
}

// L' y = z: y_b = U_b (z_b - sum_{k>b} L_kb' y_k); blocks go from the last.
// dpart != null: the block's part of rho'y goes to dpart[b].  npart != null: the
// last block of the chain combines the forward solve's magnitudes.
__device__ __forceinline__ bool trsv_upper_block(TrsvSmem& sm, int64_t pos, int64_t nblk, int64_t m, int64_t ldm,
                                                 const float* __restrict__ L, const float* __restrict__ Uinv,
                                                 double* zin, double* y, const double* __restrict__ rho,
                                                 double* dpart, const double* __restrict__ npart, Scalars* sc) {
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int64_t own = pos - cluster_rank();  // the cluster's first place in the chain
  if (pos >= nblk) return true;
  if (__syncthreads_or(dev_failed(sc))) return false;
  const int64_t b = nblk - 1 - pos;
  const int64_t r0 = b * kBig;
  const int rb = (int)(m - r0 < kBig ? m - r0 : kBig);
  if (npart && b == 0 && w == 0) {
    double gr = 0.0, gy = 0.0;
    for (int64_t i = lane; i < nblk; i += 32) gr = fmax(gr, npart[2 * i]), gy = fmax(gy, npart[2 * i + 1]);
    gr = warp_max(gr);
    gy = warp_max(gy);
    if (lane == 0) sc->rho_norm = gr, sc->dynorm = gy;
  }
  float zmine = 0.f;
  if (tid < rb) {
    zmine = (float)zin[r0 + tid];
    zin[r0 + tid] = __longlong_as_double((long long)kUnset);  // for the next forward solve
  }
  float colp[4] = {0.f, 0.f, 0.f, 0.f};  // columns 4 lane .. 4 lane + 3 of tile b, this warp's rows
  bool ok = true;
  // Two buffers, as in the forward solve; after the tiles this thread's share of
  // U_b: row r = tid / 2, columns 64 (tid % 2) .. + 63.
  float4 lv[2][16];
  auto fetch = [&](int64_t k, float4 (&t)[16]) {
    if (k > b) {
#pragma unroll
      for (int rr = 0; rr < 16; ++rr) {
        const int64_t row = k * kBig + 16 * w + rr;
        t[rr] = row < m ? __ldg(reinterpret_cast<const float4*>(L + row * ldm + r0 + 4 * lane))
                        : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    } else {
      const float4* Ub = reinterpret_cast<const float4*>(Uinv + (int64_t)b * kBig * kBig + (int64_t)(tid >> 1) * kBig +
                                                         64 * (tid & 1));
#pragma unroll
      for (int r = 0; r < 16; ++r) t[r] = __ldg(Ub + r);
    }
  };
  auto consume = [&](int64_t k, const float4 (&t)[16]) {
    const int64_t at = nblk - 1 - k;  // its place in the chain
    const float* yk = sm.zs[k & 1];
    if (at >= own) {
      if (__syncthreads_or(!wait_peer(sm, (int)(at - own), sc))) return false;
      yk = sm.zc[at - own];
    } else {
      fetch_block(sm, y, m, k, k & 1, at + 3 < own, sc);
      __syncthreads();
      if (!sm.ok[k & 1]) return false;
    }
#pragma unroll
    for (int rr = 0; rr < 16; rr += 4) {
      const float4 q = *reinterpret_cast<const float4*>(&yk[16 * w + rr]);
      const float yv[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        colp[0] = fmaf(t[rr + e].x, yv[e], colp[0]);
        colp[1] = fmaf(t[rr + e].y, yv[e], colp[1]);
        colp[2] = fmaf(t[rr + e].z, yv[e], colp[2]);
        colp[3] = fmaf(t[rr + e].w, yv[e], colp[3]);
      }
    }
    return true;
  };
  const int64_t nk = nblk - 1 - b;  // tiles: k = nblk - 1 - i, i < nk
  fetch(nblk - 1, lv[0]);
  for (int64_t i = 0; i < nk && ok; i += 2) {
    fetch(nblk - 2 - i, lv[1]);
    ok = consume(nblk - 1 - i, lv[0]);
    if (!ok || i + 1 >= nk) break;
    fetch(nblk - 3 - i, lv[0]);
    ok = consume(nblk - 2 - i, lv[1]);
  }
  if (!ok) return false;  // a wait gave up: the status says why
  *reinterpret_cast<float4*>(&sm.red[w][4 * lane]) = make_float4(colp[0], colp[1], colp[2], colp[3]);
  __syncthreads();
  if (tid < kBig) {
    float t = 0.f;
#pragma unroll
    for (int ww = 0; ww < 8; ++ww) t += sm.red[ww][tid];
    sm.rhs[tid] = tid < rb ? zmine - t : 0.f;
  }
  __syncthreads();
  const float* half = &sm.rhs[64 * (tid & 1)];
  float s = (nk & 1) ? dot64(lv[1], half) : dot64(lv[0], half);  // y_r = sum_c U_rc rhs_c
  s += __shfl_xor_sync(0xffffffffu, s, 1);
  send_entry(sm, s, b);
  const int r = tid >> 1;
  const bool mine = (tid & 1) == 0 && r < rb;
  if (mine) st_relaxed_f64(y + r0 + r, (double)s);
  if (dpart) {
    const double d = warp_sum(mine ? rho[r0 + r] * (double)s : 0.0);
    if (lane == 0) sm.mx[w][0] = d;
    __syncthreads();
    if (tid == 0) {
      double g = 0.0;
      for (int k = 0; k < 8; ++k) g += sm.mx[k][0];
      dpart[b] = g;
    }
  }
  return true;
}

__global__ void __launch_bounds__(kThreads, 1) k_trsv_upper_blk(int64_t m, int64_t ldm, int64_t nblk,
                                                                const float* __restrict__ L,
                                                                const float* __restrict__ Uinv, double* zin, double* y,
                                                                const double* __restrict__ rho, double* dpart,
                                                                const double* __restrict__ npart, unsigned* ticket,
                                                                Scalars* sc) {
  __shared__ TrsvSmem sm;
  const int64_t pos = chain_position(sm, ticket);
  leave(sm, trsv_upper_block(sm, pos, nblk, m, ldm, L, Uinv, zin, y, rho, dpart, npart, sc));
}

template <class... Params, class... Args>
cudaError_t launch_clusters(cudaStream_t st, int64_t nblk, void (*kernel)(Params...), Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((nblk + kClu - 1) / kClu * kClu));
  cfg.blockDim = dim3(kThreads);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kClu;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

}  // namespace

cudaError_t trsv_blk_solve(cudaStream_t st, int64_t m, int64_t ldm, const float* L, const float* Uinv, double* rhs,
                           double* z, double* out, const CgStep* upd, double* dpart, double* npart, unsigned* ticket,
                           Scalars* sc) {
  const int64_t nblk = (m + kBig - 1) / kBig;
  cudaError_t e = launch_clusters(st, nblk, upd ? k_trsv_lower_blk<true> : k_trsv_lower_blk<false>, m, ldm, nblk, L,
                                  Uinv, rhs, z, out, upd ? *upd : CgStep{}, npart, ticket, sc);
  if (e == cudaSuccess)
    e = launch_clusters(st, nblk, k_trsv_upper_blk, m, ldm, nblk, L, Uinv, z, out, rhs, dpart,
                        upd ? npart : (double*)nullptr, ticket, sc);
  return e;
}

}  // namespace pdas
