// FP64 Jacobi-PCG on small lattices: a whole solve in one launch.
//
// FP64 lattices of up to ~300 000 sites (the 48^3 configuration) are bound by
// latency, not bytes: as two kernels an iteration, each pass took 21 us for
// 110 592 sites (launch, loads, three levels of arrivals for the sums).  Here
// a replicate's solve runs in a group of co-resident blocks (cooperative
// launch): a thread keeps its sites' x, r, z = r / d, d, 1/d, p and c S(p) (S
// the neighbour sum) in registers for the whole solve; only z is exchanged,
// through L2, since S(p) = S(z) + beta S(p_old), and an iteration needs two
// barriers of the group, which are the exchanges of the blocks' partial sums.  FP64 runs
// at 1/64 of the FP32 rate on this GPU (measured: a warp instruction occupies
// its quarter of the multiprocessor for 76 cycles, 64 to its result), so
// operations count, 15 a site and iteration, and chains of them in the sums.
// S(p) by recurrence drifts from the neighbour sum of p by rounding, and z is a
// product with a rounded 1 / d, beta one with a rounded reciprocal: the solve
// stops on the recurred residual, as CG does, and the residual that the
// statistics report is recomputed from x.
// Measured at 48^3 (379 iterations a step): 41 -> 12.3 us an iteration, a
// third of it FP64 arithmetic, the rest the two exchanges (four trips through
// L2); a step 15.3 -> 5.9 ms.
//
// The sums' order depends on the replicate's own lattice alone (sites to
// blocks, threads, lanes), so a batch gives each replicate its own bits.
// Waits are bounded (SYNC_ERR_TIMEOUT); every block of a group runs the
// same scalar recurrences on the same sums, so all leave together.
#include <algorithm>
#include <vector>

#include "hca_internal.cuh"

namespace hca {

namespace {

constexpr int kT64 = 512;
constexpr int kMaxNG = 2;   // 2-site groups a thread holds

__device__ __forceinline__ double2 ldcg2(const double* p) { return __ldcg(reinterpret_cast<const double2*>(p)); }

// A block's partial sum travels in a slot of two 64-bit words, each half of
// the value beside the 32-bit epoch of the exchange, so a reader that sees
// the epoch in both words has the value (no counter, no second round trip).
__device__ __forceinline__ void put_slot(ulonglong2* s, double v, unsigned epoch) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v), t = (unsigned long long)epoch << 32;
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(&s->x), "l"(t | (b & 0xffffffffull)) : "memory");
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(&s->y), "l"(t | (b >> 32)) : "memory");
}
__device__ __forceinline__ bool get_slot(const ulonglong2* s, unsigned epoch, double& v) {
  unsigned long long x, y;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(x) : "l"(&s->x) : "memory");
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(y) : "l"(&s->y) : "memory");
  v = __longlong_as_double((long long)((x & 0xffffffffull) | (y << 32)));
  return (unsigned)(x >> 32) == epoch && (unsigned)(y >> 32) == epoch;
}

// m values in shared memory summed in a fixed order by W warps (this one is
// number w of them): a lane adds every 32 W-th value, then a tree.  An FP64
// instruction occupies its quarter of the multiprocessor for ~76 cycles (64
// to its result), so the sums use four warps, one a quarter, and short chains.
__device__ __forceinline__ void warp_part(const double* v, int m, int W, int w, double* out) {
  const int lane = threadIdx.x & 31;
  double t = 0.0;
  int i = 32 * w + lane;
  if (i < m) t = v[i];
  for (i += 32 * W; i < m; i += 32 * W) t += v[i];
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (lane == 0) out[w] = t;
}

// One exchange of the group's n blocks (N n <= kT64): the sums of v[0 .. N -
// 1] over all of them, in a fixed order, go through next(v) in thread 0 of
// block 0, and what it returns comes back in every thread of every block.
// Block 0 alone polls the blocks' slots (all of them polling took twice as
// long: the slots' few cache lines were the bottleneck) and hands the result
// out in one slot more.  It is a barrier of the group: nobody passes before
// every block has put its sums.  DATA: the blocks' global stores before the
// call are visible after it.  NaN when a bounded wait gave up.
__device__ __forceinline__ bool wait_slot(const Ctx& c, const ulonglong2* s, unsigned epoch, double& u) {
  int tries = 0;
  unsigned long long t0 = 0;
  while (!get_slot(s, epoch, u)) {
    if ((++tries & 255) == 0) {
      const unsigned long long now = device_ns();
      if (!t0) t0 = now;
      if (now - t0 > kBarrierTimeoutNs || *(volatile int*)&c.sync->error == SYNC_ERR_TIMEOUT) {
        atomicExch(&c.sync->error, SYNC_ERR_TIMEOUT);
        u = __longlong_as_double(0x7ff8000000000000ll);
        return false;
      }
    }
  }
  return true;
}

template <int N, bool DATA, class Next>
__device__ __forceinline__ double exchange(const Ctx& c, double (&v)[N], int nt, ulonglong2* slots, int idx, int n,
                                           unsigned epoch, Next next) {
  constexpr int W = 4 / N;
  __shared__ double s_w[N][kT64], s_p[N][W], s_out;
  const int tid = threadIdx.x, warp = tid >> 5;
  auto total = [&](int k) {
    return W == 4 ? (s_p[k][0] + s_p[k][1]) + (s_p[k][2 % W] + s_p[k][3 % W]) : s_p[k][0] + s_p[k][1 % W];
  };
#pragma unroll
  for (int k = 0; k < N; ++k) s_w[k][tid] = v[k];
  __syncthreads();
  if (warp < 4) warp_part(s_w[warp / W], nt, W, warp % W, s_p[warp / W]);
  __syncthreads();
  if (tid < N) {
    const double t = total(tid);
    if (DATA) __threadfence();
    put_slot(&slots[tid * n + idx], t, epoch);
  }
  ulonglong2* result = slots + N * n;
  if (idx == 0) {
    if (tid < N * n) {
      double u;
      wait_slot(c, &slots[tid], epoch, u);
      if (DATA) __threadfence();
      s_w[tid / n][tid % n] = u;   // (this block's values were read before the second barrier above)
    }
    __syncthreads();
    if (warp < 4) warp_part(s_w[warp / W], n, W, warp % W, s_p[warp / W]);
    __syncthreads();
    if (tid == 0) {
#pragma unroll
      for (int k = 0; k < N; ++k) v[k] = total(k);
      const double out = next(v);
      if (DATA) __threadfence();
      put_slot(result, out, epoch);
      s_out = out;
    }
  } else if (tid == 0) {
    double u;
    wait_slot(c, result, epoch, u);
    if (DATA) __threadfence();
    s_out = u;
  }
  __syncthreads();
  return s_out;
}

template <int NG>
__device__ void solve_group(const Ctx& c, int which, double* __restrict__ xfield, const Cg64Block& b) {
  const int rep = b.rep, n = b.n, nt = b.nt;
  const RepDesc& rd = c.reps[rep];
  const RepSolve sv = c.solve[rep];
  if (!sv.active) return;
  const double cpl = op_coupling(rd, which);
  double* __restrict__ zz = (double*)c.z + rd.off;
  const double* __restrict__ dd = (const double*)c.d + rd.off;
  double* __restrict__ xx = xfield + rd.off;
  ulonglong2* slots = c.slot64 + b.slot;   // sigma (n), alpha, rho (n), |r|^2 (n), beta
  __shared__ double s_rho, s_inv;   // block 0: rho (kept by thread 0) and its reciprocal
  unsigned epoch = *(volatile unsigned*)&c.epoch64[rep];   // of the last exchange
  const int gpr = rd.nxp >> 1;
  const int total = gpr * rd.ny * rd.nz;
  const int sy = rd.nxp, sz = rd.nxp * rd.ny;
  bool live[NG], has[NG][6];
  int e[NG];
  double2 x[NG], r[NG], z[NG], d[NG], w[NG], p[NG], S[NG];
#pragma unroll
  for (int i = 0; i < NG; ++i) {
    const int g = (b.idx * NG + i) * nt + (int)threadIdx.x;
    live[i] = (int)threadIdx.x < nt && g < total;
    const int row = live[i] ? g / gpr : 0;
    const int j = live[i] ? g - row * gpr : 0;
    const int zc = row / rd.ny, y = row - zc * rd.ny;
    e[i] = 2 * j + sy * row;
    has[i][0] = live[i] && j > 0;
    has[i][1] = live[i] && j + 1 < gpr;
    has[i][2] = live[i] && y > 0;
    has[i][3] = live[i] && y < rd.ny - 1;
    has[i][4] = live[i] && zc > 0;
    has[i][5] = live[i] && zc < rd.nz - 1;
    const double2 o = make_double2(0.0, 0.0);
    x[i] = live[i] ? *reinterpret_cast<const double2*>(xx + e[i]) : o;
    z[i] = live[i] ? ldcg2(zz + e[i]) : o;
    d[i] = live[i] ? ldcg2(dd + e[i]) : o;
    w[i] = make_double2(d[i].x != 0.0 ? 1.0 / d[i].x : 0.0, d[i].y != 0.0 ? 1.0 / d[i].y : 0.0);
    r[i] = make_double2(d[i].x * z[i].x, d[i].y * z[i].y);
    p[i] = S[i] = o;
  }
  // the scalars of the recurrences are thread 0 of block 0's; the others get
  // alpha and beta (NaN: stop)
  const double nan = __longlong_as_double(0x7ff8000000000000ll);
  const double stop = sv.rtol * sqrt(sv.bnorm2), stop2 = stop * stop;
  double rho = sv.rho, rr = sv.rnorm2, beta = 0.0;
  int iters = 0, error = 0;
  bool done = false;
  if (threadIdx.x == 0) s_rho = rho;   // (read after the first exchange's barriers)
  for (;;) {
    // p = z + beta p and c S(p) = c S(z) + beta c S(p_old); q = d p - c S(p) = A p
    double s1[1] = {0.0};
    double2 q[NG];
#pragma unroll
    for (int i = 0; i < NG; ++i) {
      const double2 o = make_double2(0.0, 0.0);
      const double zl = has[i][0] ? __ldcg(zz + e[i] - 1) : 0.0, zr = has[i][1] ? __ldcg(zz + e[i] + 2) : 0.0;
      const double2 ym = has[i][2] ? ldcg2(zz + e[i] - sy) : o, yp = has[i][3] ? ldcg2(zz + e[i] + sy) : o;
      const double2 zm = has[i][4] ? ldcg2(zz + e[i] - sz) : o, zp = has[i][5] ? ldcg2(zz + e[i] + sz) : o;
      p[i].x = fma(beta, p[i].x, z[i].x);
      p[i].y = fma(beta, p[i].y, z[i].y);
      S[i].x = fma(beta, S[i].x, cpl * (((zl + z[i].y) + (ym.x + yp.x)) + (zm.x + zp.x)));
      S[i].y = fma(beta, S[i].y, cpl * (((z[i].x + zr) + (ym.y + yp.y)) + (zm.y + zp.y)));
      q[i].x = fma(d[i].x, p[i].x, -S[i].x);
      q[i].y = fma(d[i].y, p[i].y, -S[i].y);
      s1[0] = fma(p[i].x, q[i].x, s1[0]);   // padding: p = 0
      s1[0] = fma(p[i].y, q[i].y, s1[0]);
    }
    const double alpha = exchange<1, false>(c, s1, nt, slots, b.idx, n, ++epoch, [&](const double (&t)[1]) {
      if (t[0] > 0.0 && isfinite(t[0])) return rho / t[0];
      error = !isfinite(t[0]);
      done = true;
      return nan;
    });
    if (alpha != alpha) break;
    if (b.idx == 0 && threadIdx.x == kT64 - 1) s_inv = 1.0 / s_rho;   // beta is then a product
    double s2[2] = {0.0, 0.0};
#pragma unroll
    for (int i = 0; i < NG; ++i) {
      x[i].x = fma(alpha, p[i].x, x[i].x);
      x[i].y = fma(alpha, p[i].y, x[i].y);
      if (d[i].x != 0.0) r[i].x = fma(-alpha, q[i].x, r[i].x);   // padding keeps r = 0
      if (d[i].y != 0.0) r[i].y = fma(-alpha, q[i].y, r[i].y);
      z[i].x = w[i].x * r[i].x;
      z[i].y = w[i].y * r[i].y;
      s2[0] = fma(r[i].x, z[i].x, s2[0]);
      s2[0] = fma(r[i].y, z[i].y, s2[0]);
      s2[1] = fma(r[i].x, r[i].x, s2[1]);
      s2[1] = fma(r[i].y, r[i].y, s2[1]);
      if (live[i]) __stcg(reinterpret_cast<double2*>(zz + e[i]), z[i]);
    }
    beta = exchange<2, true>(c, s2, nt, slots + n + 1, b.idx, n, ++epoch, [&](const double (&t)[2]) {
      ++iters;
      error = !isfinite(t[0]) || !isfinite(t[1]);
      if (error) {
        done = true;
        return nan;
      }
      const double bt = t[0] * s_inv;
      s_rho = rho = t[0];
      rr = t[1];
      done = rr <= stop2 || iters >= sv.maxit;
      return done ? nan : bt;
    });
    if (beta != beta) break;
  }
#pragma unroll
  for (int i = 0; i < NG; ++i)
    if (live[i]) *reinterpret_cast<double2*>(xx + e[i]) = x[i];
  if (threadIdx.x == 0) {
    // the next launch's exchanges continue past this one's epochs (far past
    // them after a timeout, whose blocks left at different ones)
    if (*(volatile int*)&c.sync->error == SYNC_ERR_TIMEOUT) {
      atomicMax(&c.epoch64[rep], epoch + (1u << 16));
    } else if (b.idx == 0 && done) {
      c.epoch64[rep] = epoch;
      RepSolve& s = c.solve[rep];
      s.iters = iters;
      s.rho = rho;
      s.rnorm2 = rr;
      s.active = 0;
      if (error) c.sync->error = 1;
    }
  }
}

__global__ void __launch_bounds__(kT64, 1) k_cg64(Ctx c, int which, double* xfield, const Cg64Block* table, int rounds) {
  HCA_COUNT_KERNEL(c);
  for (int r = 0; r < rounds; ++r) {
    const Cg64Block b = table[r * gridDim.x + blockIdx.x];
    if (b.rep < 0) continue;
    if (*(volatile int*)&c.sync->error == SYNC_ERR_TIMEOUT) return;
    if (b.ng == 1) solve_group<1>(c, which, xfield, b);
    else solve_group<2>(c, which, xfield, b);
    __syncthreads();
  }
}

// The replicates still iterating after k_cg64 (those too large for it).
__global__ void k_cg64_done(Ctx c, CondArg cnd) {
  HCA_COUNT_KERNEL(c);
  if (threadIdx.x) return;
  int n = 0;
  for (int r = 0; r < c.n_reps; ++r) n += c.solve[r].active;
  c.sync->active_count = n;
  set_cond(cnd, n > 0);
}

}  // namespace

// Blocks of the small replicates' solves: table [round][block] of a launch of
// `blocks` co-resident blocks; a replicate's group of blocks follows its
// lattice alone.  Returns the number of rounds (0: no replicate is small, or
// no cooperative launch); *large: replicates left to the pass kernels.
int cg64_plan(const std::vector<RepDesc>& reps, int sm_count, std::vector<Cg64Block>& table, int* blocks, int* large,
              long long* slots) {
  *blocks = 0;
  *slots = 0;
  *large = (int)reps.size();
  int dev = 0, coop = 0, per = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess ||
      !coop || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_cg64, kT64, 0) != cudaSuccess || per < 1) {
    (void)cudaGetLastError();
    return 0;
  }
  std::vector<std::vector<Cg64Block>> rounds;
  for (size_t i = 0; i < reps.size(); ++i) {
    const long long g = (long long)(reps[i].nxp / 2) * reps[i].ny * reps[i].nz;
    // an even share of the 2-site groups per multiprocessor (the FP64 pipe is
    // the bound of the arithmetic), at least two warps a block
    const int ng = g <= (long long)kT64 * sm_count ? 1 : kMaxNG;
    const long long share = ((g + sm_count - 1) / sm_count + ng - 1) / ng;
    const int nt = (int)std::max(64LL, (share + 31) / 32 * 32);
    const long long nb = (g + (long long)nt * ng - 1) / ((long long)nt * ng);
    if (nt > kT64 || nb > sm_count || 2 * nb > kT64) continue;
    --*large;
    size_t r = 0;
    while (r < rounds.size() && (long long)rounds[r].size() + nb > sm_count) ++r;
    if (r == rounds.size()) rounds.emplace_back();
    for (int k = 0; k < (int)nb; ++k) rounds[r].push_back(Cg64Block{(int)i, k, (int)nb, ng, nt, 0, *slots});
    *slots += 3 * nb + 2;
  }
  for (auto& r : rounds) *blocks = std::max(*blocks, (int)r.size());
  for (auto& r : rounds) {
    r.resize(*blocks, Cg64Block{-1, 0, 0, 0, 0, 0, 0});
    table.insert(table.end(), r.begin(), r.end());
  }
  return (int)rounds.size();
}

void launch_cg64(const Ctx& c, int which, void* xfield, CondArg cnd) {
  Ctx cc = c;
  int wh = which, rounds = c.rounds64;
  double* x = (double*)xfield;
  const Cg64Block* t = c.blk64;
  void* args[] = {&cc, &wh, &x, &t, &rounds};
  (void)cudaLaunchCooperativeKernel((const void*)k_cg64, dim3(c.n_blk64), dim3(kT64), args, 0, c.stream);
  k_cg64_done<<<1, 32, 0, c.stream>>>(c, cnd);
}

}  // namespace hca
