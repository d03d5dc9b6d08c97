// Helpers of the plane-marching FP32 kernels (march.cu, cg.cu): asynchronous
// copies, a thread's 4 x 2 patch of sites and its neighbour sums, and the
// fixed-order sums over a launch's blocks.
#pragma once

#include "hca_internal.cuh"
#include "tc.cuh"

namespace hca {

constexpr int kMT = 256;              // most threads per block (instances: 64, 128, 256)
constexpr int kMaxSeg = 8;            // most z segments of a slab (reduction slots)
constexpr int blocks_per_sm(int nt) { return nt >= 256 ? 2 : 512 / nt; }

__device__ __forceinline__ void cp16(unsigned sdst, const float* gsrc, int n) {   // n = 0: zero fill
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sdst), "l"(gsrc), "r"(n) : "memory");
}

// Planes of a tile arrive by tensor copies: one thread issues, per plane and
// input array, the box of the tile's rows (halo included, zeros outside the
// level), completing on the stage's mbarrier.  (Per-thread 16-byte cp.async
// copies of the patches took 14 shared-memory cycles a warp instruction: the
// pipe the sweeps' own exchanges need.)
constexpr int kTmaWaitLimit = 1 << 20;
// The lattice's maps, from MGLevel::map0 of its pass A tiling: z, p, p_alt, dx,
// d; a, b, perfusion, V, K_prev; x_hi and x_lo of each operator.
constexpr int kMapReac = 5, kMapFields = 10;
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc::smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void tma_load_3d(void* sdst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::
          "r"(tc::smem_u32(sdst)),
      "l"((unsigned long long)map), "r"(x), "r"(y), "r"(z), "r"(tc::smem_u32(bar))
      : "memory");
}
// The maps are in global memory, written by a copy at creation; the acquire
// also drops what the descriptor cache may hold of an earlier handle at the
// same address.
__device__ __forceinline__ void maps_acquire(const CUtensorMap* maps, int n) {
  for (int m = 0; m < n; ++m)
    asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"((unsigned long long)&maps[m])
                 : "memory");
}
// The stages' barriers, and the maps the block uses (one thread).
__device__ __forceinline__ void mbars_init(uint64_t* bar, int n, const CUtensorMap* maps, int n_maps) {
  if (threadIdx.x == 0) {
    maps_acquire(maps, n_maps);
    for (int s = 0; s < n; ++s) tc::mbar_init(&bar[s], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
}
__device__ __forceinline__ float4* align128(void* p) {
  return reinterpret_cast<float4*>((reinterpret_cast<uintptr_t>(p) + 127) & ~uintptr_t(127));
}
// A copy did not complete in time: record it and let this block's copies in
// flight (uses n .. issued - 1 of a ring of `ring` stages) land before its
// shared memory is released.
__device__ __forceinline__ void tma_abort(const Ctx& c, uint64_t* bar, int ring, int n, int issued) {
  if (threadIdx.x == 0) {
    c.sync->error = SYNC_ERR_TIMEOUT;
    for (int k = n; k < issued; ++k) (void)tc::mbar_wait(&bar[k % ring], (uint32_t)((k / ring) & 1), kTmaWaitLimit);
  }
  __syncthreads();
}
__device__ __forceinline__ void cp4(unsigned sdst, const float* gsrc, int n) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(sdst), "l"(gsrc), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// The patch's 4 x 2 values on one plane as pairs along x: the sums and
// products below use the two-wide FP32 instructions (one issue for two
// sites; every product and sum rounded as in the scalar form).
struct P8 {
  float2 v[2][2];   // [row][sites 0, 1 | 2, 3]
};
__device__ __forceinline__ float2 dup(float a) { return make_float2(a, a); }
__device__ __forceinline__ void get_row(float2 (&v)[2], const float4* s) {
  const float4 q = *s;
  v[0] = make_float2(q.x, q.y);
  v[1] = make_float2(q.z, q.w);
}

// 1 / d (0 where d = 0: padding, outside the level, an isolated empty site);
// a smoothing weight, so the hardware reciprocal (1 ulp) serves
__device__ __forceinline__ float inv_d(float d) {
  float w;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(w) : "f"(d));
  return d > 0.f ? w : 0.f;
}
__device__ __forceinline__ float2 inv_d(float2 d) { return make_float2(inv_d(d.x), inv_d(d.y)); }

// This thread's place in its block's tile.  Every tile carries its halo, also
// at the level's edges (zeros there), so no neighbour needs a bounds check;
// neighbours beyond the tile (of outermost halo patches, unused) read the
// thread's own values.
struct Patch {
  int tid, lane, x0, y0;   // first site of the patch
  int tx0, ty0;        // first site and row of the tile's box
  int r0, r1;          // the patch's rows in a staged box (16-byte units)
  int nx, nz;
  int im, ip;          // row buffer slots of the rows below and above the patch
  bool l0, l31;        // the x neighbour is in another warp
  bool rok[2];         // the patch's rows inside the level (and the group)
  bool in[2];          // the rows that belong to the tile's interior
  bool out;            // either does
  bool part;           // the group has padding sites
  unsigned e, sy, sz;  // element of (x0, y0, plane 0), strides (a field has fewer than 2^32 elements)
};

// HY: halo rows below and above the tile's interior (2: patches start on even
// rows, as the transfers to the next level need; 1: one more row of interior
// for the same patches).
template <int NT, int HY>
__device__ __forceinline__ Patch patch_of(const MGLevel& L, int4 b) {
  Patch p;
  p.tid = threadIdx.x;
  p.lane = p.tid & 31;
  const int cols = L.cols, pairs = L.pairs;
  const int pr = p.tid / cols, col = p.tid - pr * cols;
  p.nx = L.nx;
  p.nz = L.nz;
  const int ty = b.y / L.tx, tx = b.y - ty * L.tx;
  const int g = tx * L.ox - 1 + col;
  p.x0 = 4 * g;
  p.y0 = ty * L.oy - HY + 2 * pr;
  p.tx0 = 4 * (tx * L.ox - 1);
  p.ty0 = ty * L.oy - HY;
  p.r0 = pr < pairs ? 2 * pr * cols + col : 0;
  p.r1 = p.r0 + (pr < pairs ? cols : 0);
  const bool gok = g >= 0 && p.x0 < p.nx && pr < pairs, cin = col >= 1 && col <= L.ox;
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const int t = 2 * pr + a - HY;   // row of the interior
    p.rok[a] = gok && p.y0 + a >= 0 && p.y0 + a < L.ny;
    p.in[a] = p.rok[a] && cin && t >= 0 && t < L.oy;
  }
  p.out = p.in[0] || p.in[1];
  p.part = p.x0 + 4 > p.nx;
  p.im = NT + p.tid - (pr > 0 ? cols : 0);
  p.ip = p.tid + (pr < pairs - 1 ? cols : 0);
  p.l0 = p.lane == 0 && p.tid > 0;
  p.l31 = p.lane == 31 && p.tid + 1 < NT;
  p.sy = (unsigned)L.pitch;
  p.sz = (unsigned)L.pitch * (unsigned)L.ny;
  p.e = p.rok[0] || p.rok[1] ? (unsigned)p.x0 + p.sy * (unsigned)p.y0 : 0u;   // (row -1: wraps, its own row is not used)
  return p;
}

// The sum over the neighbours of the patch on its own plane and the one
// below: uc the plane (its rows also in row buffer B: [row of the
// pair][thread]), um the plane below; S may be um.
template <int NT>
__device__ __forceinline__ void nb_patch(const Patch& p, const float4* __restrict__ B, const P8& uc, const P8& um,
                                         P8& S) {
  const float4 ym = B[p.im], yp = B[p.ip];
  const float2 ymv[2] = {make_float2(ym.x, ym.y), make_float2(ym.z, ym.w)};
  const float2 ypv[2] = {make_float2(yp.x, yp.y), make_float2(yp.z, yp.w)};
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const float2 u0 = uc.v[a][0], u1 = uc.v[a][1];
    float lft = __shfl_up_sync(0xffffffffu, u1.y, 1), rgt = __shfl_down_sync(0xffffffffu, u0.x, 1);
    const float* Bf = reinterpret_cast<const float*>(B + a * NT + p.tid);
    if (p.l0) lft = Bf[-1];
    if (p.l31) rgt = Bf[4];
    const float2 x[2] = {make_float2(lft + u0.y, u0.x + u1.x), make_float2(u0.y + u1.y, u1.x + rgt)};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float2 m = a == 0 ? __fadd2_rn(ymv[h], uc.v[1][h]) : __fadd2_rn(uc.v[0][h], ypv[h]);
      S.v[a][h] = __fadd2_rn(__fadd2_rn(x[h], m), um.v[a][h]);
    }
  }
}

template <int NT>
__device__ __forceinline__ void put_patch(const Patch& p, float4* __restrict__ B, const P8& u) {
#pragma unroll
  for (int a = 0; a < 2; ++a) B[a * NT + p.tid] = make_float4(u.v[a][0].x, u.v[a][0].y, u.v[a][1].x, u.v[a][1].y);
}

__device__ __forceinline__ void zero_patch(P8& u) {
#pragma unroll
  for (int a = 0; a < 2; ++a) u.v[a][0] = u.v[a][1] = make_float2(0.f, 0.f);
}

// The end of a marching kernel that sums into slots: the last block of the
// replicate (nblk blocks) to arrive adds its n slots in an order that is the
// same whatever the launch (64 lanes take every 64th slot, then a fixed
// tree) and hands the sum to fin, called by one thread.  count: how many of
// the nblk blocks this one stands for.
template <class Fin>
__device__ __forceinline__ void march_finish(const Ctx& c, int rep, int nblk, const double* slots, int n, Fin fin,
                                             int count = 1) {
  __shared__ int s_last;
  __shared__ double s_half[2];
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(&c.mcnt[rep], count) == nblk - count;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (threadIdx.x < 64) {
    double t = 0.0;
#pragma unroll 8
    for (int i = threadIdx.x; i < n; i += 64) t += __ldcg(&slots[i]);
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) s_half[threadIdx.x >> 5] = t;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    fin(s_half[0] + s_half[1]);
    c.mcnt[rep] = 0;
  }
}

}  // namespace hca
