// The FP32 CG passes (both preconditioners, single lattices and batches):
//
//   pass A  p = z + beta p_old, q = A p, sigma = p.q -> alpha
//   pass B  r -= alpha q, |r|^2  (V-cycle form; Jacobi form: the carried
//           z = r / d, z -= alpha q / d, rho = sum d z^2, |r|^2 = sum (d z)^2)
//
// x += alpha p moves from pass B to the next pass A, which reads p_old
// anyway: the first iteration of a solve touches no x at all, the last step
// is added by the defect correction's update (k_dc_update).  Traffic per site:
// pass A reads z, d (+ p_old, dx) and writes p, q (+ dx): 16 B in a solve's
// first iteration, 24 in its second, 28 from then on; pass B reads r, q and
// writes r: 12 B (Jacobi form: also d); the update reads p besides dx.  A
// plain FP32 solve (no defect correction) keeps x += alpha p in pass B.
//
// Pass A marches up z like the V-cycle's sweeps (march.cu): patches of 4 x 2
// sites, inputs staged two planes ahead by tensor copies, p of
// the plane's rows exchanged through shared memory, z neighbours in
// registers.  Pass B is a stream of 4-site groups through a cp.async ring.
// Both leave the split of the L1 where the V-cycle's kernels need it: row
// kernels that load through a large L1 ran at 77 us each at 256^3, but every
// switch between them and those kernels cost ~12 us (with the split pinned
// for all of them, pass A 102 us and pass B 89 us).  Measured at 256^3: pass
// A 75 us (an average of 22 B a site; 87 with per-thread copies), pass B 48 us;
// a step 15.2 -> 13.6 ms by the passes themselves.
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "march.cuh"

namespace hca {

void march_tile(MGLevel& L, int halo_rows);
int march_threads(const std::vector<MGLevel*>& lv);
void march_blocks(std::vector<MGLevel*>& lv, const std::vector<int>& reps, int sm_count, int extra, std::vector<int4>& out);

namespace {

constexpr int kARing = 3;             // planes k .. k + 2 of z, p_old and dx, k - 1 .. k + 1 of d
constexpr size_t a_smem(int nt) { return (size_t)(kARing * 8 + 4) * nt * 16 + (size_t)kMaxSeg * (nt / 32) * 8 + 128; }

// ----------------------------------------------------------------- pass A --
// One thread, with sigma = p.q of replicate rep.
__device__ __forceinline__ void alpha_of(const Ctx& c, int rep, double sigma) {
  RepSolve& s = c.solve[rep];
  if (!(sigma > 0.0) || !isfinite(sigma)) {
    if (!isfinite(sigma)) c.sync->error = 1;
    s.active = 0;
    s.pend = 0;   // this launch added the last step
    return;
  }
  s.alpha = s.rho / sigma;
}

template <int NT, bool DEFER>
__global__ void __launch_bounds__(NT, blocks_per_sm(NT)) k_cg_a(Ctx c, int which) {
  extern __shared__ __align__(16) float4 msm[];
  const int4 b = c.ablk[blockIdx.x];
  const int rep = b.x;
  const MGLevel& L = c.cg_lv[rep];
  const RepDesc& rd = c.reps[rep];
  const Patch p = patch_of<NT, 1>(L, b);
  const int zb = b.z, ze = b.w;
  const float cpl = rd.cpl32[which];
  const long long off = rd.off;
  __shared__ __align__(8) uint64_t bar[kARing];
  const CUtensorMap* maps = c.tmaps + L.map0;   // z, p, p_alt, dx, d
  mbars_init(bar, kARing, maps, 5);
  HCA_COUNT_KERNEL(c);
  const RepSolve sv = c.solve[rep];
  if (!sv.active) return;
  const int par = c.sync->parity;
  float* __restrict__ pn = (float*)(par ? c.p : c.p_alt) + off;
  const CUtensorMap* map_p = &maps[par ? 2 : 1];
  const uint32_t box = 32u * (uint32_t)(L.cols * L.pairs);
  float* __restrict__ qq = (float*)c.q + off;
  float* __restrict__ xx = (float*)c.dx + off;
  const float2 beta = dup((float)sv.beta), alpha = dup((float)sv.alpha);
  const bool add = DEFER && sv.pend;                 // the step of the iteration before
  const bool use_p = sv.beta != 0.0 || add, use_x = add && sv.iters > 1;
  // the first iteration of a rescaled inner solve starts from scale * z (the
  // V-cycle scales r itself before it forms z)
  const float2 zs = dup((sv.iters == 0 && !c.mg) ? (float)sv.scale : 1.f);
  float4* ring = align128(msm);            // [phase][z, p, x, d (of the plane before)][row][group]
  float4* pb = ring + kARing * 8 * NT;     // [plane & 1][row of the pair][thread]
  float2* segs = reinterpret_cast<float2*>(pb + 4 * NT);
  auto fetch = [&](int k, int slot) {
    float4* s = ring + slot * 8 * NT;
    mbar_expect_tx(&bar[slot], (2u + use_p + use_x) * box);
    tma_load_3d(s, &maps[0], p.tx0, p.ty0, k, &bar[slot]);
    if (use_p) tma_load_3d(s + 2 * NT, map_p, p.tx0, p.ty0, k, &bar[slot]);
    if (use_x) tma_load_3d(s + 4 * NT, &maps[3], p.tx0, p.ty0, k, &bar[slot]);
    tma_load_3d(s + 6 * NT, &maps[4], p.tx0, p.ty0, k - 1, &bar[slot]);
  };
  P8 u[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) zero_patch(u[i]);
  FF acc{0.f, 0.f};
  const int k0 = zb - 1, k1 = ze;   // planes whose p is formed
  int issued = 2;   // (thread 0)
  if (p.tid == 0) {
    fetch(k0, 0);
    fetch(k0 + 1, 1);
  }
  int seg = 0;
  uint32_t phase = 0;
  const int seglen = L.seg;
  auto step = [&](auto ph, int k) {
    constexpr int P0 = decltype(ph)::value, P1 = (P0 + 2) % 3, P2 = (P0 + 1) % 3;
    if (p.tid == 0 && k + 2 <= k1) {
      fetch(k + 2, P1);
      ++issued;
    }
    const bool ok = tc::mbar_wait(&bar[P0], phase, kTmaWaitLimit);
    const float4* rs = ring + P0 * 8 * NT;
    float2 z[2][2], po[2][2];
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      get_row(z[a], rs + (a ? p.r1 : p.r0));
      if (use_p) get_row(po[a], rs + 2 * NT + (a ? p.r1 : p.r0));
      else po[a][0] = po[a][1] = make_float2(0.f, 0.f);
    }
    nb_patch<NT>(p, pb + ((k & 1) ^ 1) * 2 * NT, u[P1], u[P2], u[P2]);
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int h = 0; h < 2; ++h) u[P0].v[a][h] = __ffma2_rn(beta, po[a][h], __fmul2_rn(zs, z[a][h]));
    put_patch<NT>(p, pb + (k & 1) * 2 * NT, u[P0]);
    if (add && k >= zb && k < ze) {
      const unsigned e = p.e + (unsigned)k * p.sz;
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        if (!p.in[a]) continue;
        float2 x[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        if (use_x) get_row(x, rs + 4 * NT + (a ? p.r1 : p.r0));
#pragma unroll
        for (int h = 0; h < 2; ++h) x[h] = __ffma2_rn(alpha, po[a][h], x[h]);
        *reinterpret_cast<float4*>(xx + (e + a * p.sy)) = make_float4(x[0].x, x[0].y, x[1].x, x[1].y);
      }
    }
    if (k > zb) {
      const unsigned e = p.e + (unsigned)(k - 1) * p.sz;
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        if (!p.in[a]) continue;
        float2 d[2], q[2];
        get_row(d, rs + 6 * NT + (a ? p.r1 : p.r0));
        float g_s = 0.f;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float2 S = __fadd2_rn(u[P2].v[a][h], u[P0].v[a][h]);
          const float2 m = __fmul2_rn(dup(cpl), S);
          q[h] = __ffma2_rn(d[h], u[P1].v[a][h], make_float2(-m.x, -m.y));
          if (p.part) {   // padding sites hold 0
            if (p.x0 + 2 * h >= p.nx) q[h].x = 0.f;
            if (p.x0 + 2 * h + 1 >= p.nx) q[h].y = 0.f;
          }
          g_s = cg_madd(u[P1].v[a][h].x, q[h].x, g_s);
          g_s = cg_madd(u[P1].v[a][h].y, q[h].y, g_s);
        }
        const float2* w = u[P1].v[a];
        *reinterpret_cast<float4*>(pn + (e + a * p.sy)) = make_float4(w[0].x, w[0].y, w[1].x, w[1].y);
        *reinterpret_cast<float4*>(qq + (e + a * p.sy)) = make_float4(q[0].x, q[0].y, q[1].x, q[1].y);
        acc = ff_add(acc, g_s);
      }
      const int z1 = k - 1;
      if (((z1 + 1) % seglen) == 0 || z1 == ze - 1) {
        const FF s = row_reduce_ff(acc, 32);
        if (p.lane == 0) segs[seg * (NT / 32) + (p.tid >> 5)] = make_float2(s.hi, s.lo);
        acc = FF{0.f, 0.f};
        ++seg;
      }
    }
    return !__syncthreads_or(!ok);   // a copy timed out: every thread stops
  };
  for (int k = k0; k <= k1; k += 3, phase ^= 1) {
    if (!step(std::integral_constant<int, 0>{}, k) ||
        (k + 1 <= k1 && !step(std::integral_constant<int, 1>{}, k + 1)) ||
        (k + 2 <= k1 && !step(std::integral_constant<int, 2>{}, k + 2))) {
      tma_abort(c, bar, kARing, k - k0, issued);   // (goes on to its arrival)
      break;
    }
  }
  double* slots = c.mslot + L.slot0 + (long long)b.y * L.nseg + zb / seglen;
  for (int s = threadIdx.x; s < seg; s += NT) {
    double t = 0.0;
    for (int q = 0; q < NT / 32; ++q) {
      const float2 f = segs[s * (NT / 32) + q];
      t += (double)f.x + (double)f.y;
    }
    slots[s] = t;
  }
  march_finish(c, rep, L.nblk, c.mslot + L.slot0, L.tx * L.ty * L.nseg, [&](double sigma) { alpha_of(c, rep, sigma); });
}

// Pass A on flat lattices (every lattice of the handle has one plane).  There
// is nothing to march over: a block of the marching form would hold one tile
// for two planes' steps, and its start, fence and arrival took 7 us a tile
// (4000 x 4000 x 1: 240 us a launch).  Here a block walks over a run of the
// same tiles, reads rows and their neighbours through the caches, without
// barriers, and arrives once for all of them: 85 us, bound by HBM (an oxygen
// solve with Jacobi 21.1 -> 11.7 ms, 11.8 with the row kernels before the
// marching form; with the V-cycle 8.2 -> 7.1).  Sites, patches, lanes and sums
// are those of the marching form, so the results are the same bits.
constexpr int kFlatTiles = 32;   // tiles whose sums a block holds
constexpr int flat_blocks(int nt) { return 768 / nt; }   // resident: registers for 24 warps

template <int NT, bool DEFER>
__global__ void __launch_bounds__(NT, flat_blocks(NT)) k_cg_a_flat(Ctx c, int which) {
  constexpr int NW = NT / 32;
  __shared__ float2 segs[kFlatTiles * NW];
  HCA_COUNT_KERNEL(c);
  const int par = c.sync->parity;
  const int e0 = (int)((long long)c.n_ablk * blockIdx.x / gridDim.x), e1 = (int)((long long)c.n_ablk * (blockIdx.x + 1) / gridDim.x);
  const float2 zero = make_float2(0.f, 0.f);
  for (int e = e0; e < e1;) {
    // a run of tiles of one replicate
    const int rep = c.ablk[e].x, first = c.ablk[e].y;
    const MGLevel& L = c.cg_lv[rep];
    const int n = min(min(e1 - e, L.nblk - first), kFlatTiles);
    e += n;
    const RepSolve sv = c.solve[rep];
    if (!sv.active) continue;
    const RepDesc& rd = c.reps[rep];
    const float cpl = rd.cpl32[which];
    const long long off = rd.off;
    const float* __restrict__ zz = (const float*)c.z + off;
    const float* __restrict__ dd = (const float*)c.d + off;
    const float* __restrict__ po = (const float*)(par ? c.p_alt : c.p) + off;
    float* __restrict__ pn = (float*)(par ? c.p : c.p_alt) + off;
    float* __restrict__ qq = (float*)c.q + off;
    float* __restrict__ xx = (float*)c.dx + off;
    const float2 beta = dup((float)sv.beta), alpha = dup((float)sv.alpha);
    const bool add = DEFER && sv.pend, use_p = sv.beta != 0.0 || add, use_x = add && sv.iters > 1;
    const float2 zs = dup((sv.iters == 0 && !c.mg) ? (float)sv.scale : 1.f);
    const int ny = L.ny;
    for (int t = 0; t < n; ++t) {
      const Patch p = patch_of<NT, 1>(L, make_int4(rep, first + t, 0, 1));
      const int col = p.tid % L.cols, pr = p.tid / L.cols;
      const bool gok = p.x0 >= 0 && p.x0 < p.nx && pr < L.pairs, cin = col >= 1 && col <= L.ox;
      // rows y0 - 1 .. y0 + 2 of z and p_old; the outer two where an interior row needs them
      float2 u[4][2], o[4][2];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int y = p.y0 - 1 + i;
        const bool ok = gok && y >= 0 && y < ny && (i == 0 ? p.in[0] : i == 3 ? p.in[1] : true);
        u[i][0] = u[i][1] = o[i][0] = o[i][1] = zero;
        const unsigned a = ok ? (unsigned)p.x0 + p.sy * (unsigned)y : 0u;
        if (ok) get_row(u[i], reinterpret_cast<const float4*>(zz + a));
        if (ok && use_p) get_row(o[i], reinterpret_cast<const float4*>(po + a));
      }
      // left and right neighbours that another warp holds
      float zl[2] = {0.f, 0.f}, pl[2] = {0.f, 0.f}, zr[2] = {0.f, 0.f}, pq[2] = {0.f, 0.f};
      float2 d[2][2], x[2][2];
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        d[a][0] = d[a][1] = x[a][0] = x[a][1] = zero;
        if (!p.in[a]) continue;
        const unsigned ea = p.e + a * p.sy;
        get_row(d[a], reinterpret_cast<const float4*>(dd + ea));
        if (use_x) get_row(x[a], reinterpret_cast<const float4*>(xx + ea));
        if (p.l0 && p.x0 > 0) {
          zl[a] = zz[ea - 1];
          if (use_p) pl[a] = po[ea - 1];
        }
        if (p.l31 && p.x0 + 4 < p.nx) {
          zr[a] = zz[ea + 4];
          if (use_p) pq[a] = po[ea + 4];
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          u[i][h] = __ffma2_rn(beta, o[i][h], __fmul2_rn(zs, u[i][h]));
          if (p.part) {   // padding sites count as zeros
            if (p.x0 + 2 * h >= p.nx) u[i][h].x = 0.f;
            if (p.x0 + 2 * h + 1 >= p.nx) u[i][h].y = 0.f;
          }
        }
      FF acc{0.f, 0.f};
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        const float2 u0 = u[a + 1][0], u1 = u[a + 1][1];
        float lft = __shfl_up_sync(0xffffffffu, u1.y, 1), rgt = __shfl_down_sync(0xffffffffu, u0.x, 1);
        if (!p.in[a]) continue;
        if (p.l0) lft = __fmaf_rn(beta.x, pl[a], __fmul_rn(zs.x, zl[a]));
        if (p.l31) rgt = __fmaf_rn(beta.x, pq[a], __fmul_rn(zs.x, zr[a]));
        const float2 xs[2] = {make_float2(lft + u0.y, u0.x + u1.x), make_float2(u0.y + u1.y, u1.x + rgt)};
        float2 q[2];
        float g_s = 0.f;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float2 S = __fadd2_rn(__fadd2_rn(__fadd2_rn(xs[h], __fadd2_rn(u[a][h], u[a + 2][h])), zero), zero);
          const float2 m = __fmul2_rn(dup(cpl), S);
          const float2 w = u[a + 1][h];
          q[h] = __ffma2_rn(d[a][h], w, make_float2(-m.x, -m.y));
          if (p.part) {
            if (p.x0 + 2 * h >= p.nx) q[h].x = 0.f;
            if (p.x0 + 2 * h + 1 >= p.nx) q[h].y = 0.f;
          }
          g_s = cg_madd(w.x, q[h].x, g_s);
          g_s = cg_madd(w.y, q[h].y, g_s);
        }
        const unsigned ea = p.e + a * p.sy;
        if (add) {
#pragma unroll
          for (int h = 0; h < 2; ++h) x[a][h] = __ffma2_rn(alpha, o[a + 1][h], x[a][h]);
          *reinterpret_cast<float4*>(xx + ea) = make_float4(x[a][0].x, x[a][0].y, x[a][1].x, x[a][1].y);
        }
        *reinterpret_cast<float4*>(pn + ea) = make_float4(u0.x, u0.y, u1.x, u1.y);
        *reinterpret_cast<float4*>(qq + ea) = make_float4(q[0].x, q[0].y, q[1].x, q[1].y);
        acc = ff_add(acc, g_s);
      }
      const FF s = row_reduce_ff(acc, 32);
      if (p.lane == 0) segs[t * NW + (p.tid >> 5)] = make_float2(s.hi, s.lo);
    }
    __syncthreads();
    double* slots = c.mslot + L.slot0 + first;
    for (int t = threadIdx.x; t < n; t += NT) {
      double v = 0.0;
      for (int w = 0; w < NW; ++w) {
        const float2 f = segs[t * NW + w];
        v += (double)f.x + (double)f.y;
      }
      slots[t] = v;
    }
    march_finish(c, rep, L.nblk, c.mslot + L.slot0, L.tx * L.ty, [&](double sigma) { alpha_of(c, rep, sigma); }, n);
  }
}

// ----------------------------------------------------------------- pass B --
constexpr int kBT = 256, kBRing = 3, kBMaxChunks = 64;
template <bool MG, bool DEFER>
constexpr int b_arrays() { return (MG ? 2 : 3) + (DEFER ? 0 : 2); }   // r|z, q (, d) (, p, x)
template <bool MG, bool DEFER>
constexpr size_t b_smem() { return (size_t)kBRing * b_arrays<MG, DEFER>() * kBT * 16 + (size_t)kBMaxChunks * (kBT / 32) * 16; }

template <bool MG, bool DEFER>
__global__ void __launch_bounds__(kBT, 4) k_cg_b(Ctx c, int which, float* __restrict__ xfield, CondArg cnd) {
  extern __shared__ __align__(16) float4 msm[];
  constexpr int NA = b_arrays<MG, DEFER>();
  const int4 b = c.bblk[blockIdx.x];
  const int rep = b.x;
  const int4 geo = c.bgeo[rep];   // groups, groups per chunk, chunks, first slot
  const long long off = c.reps[rep].off;
  HCA_COUNT_KERNEL(c);
  __shared__ int s_last;
  __shared__ double s_sum[2][kBT / 32];
  const RepSolve sv = c.solve[rep];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double* slot_rr = c.mslot + geo.w;
  double* slot_rho = slot_rr + geo.z;
  if (sv.active) {
    const int par = c.sync->parity;
    const float* __restrict__ qq = (const float*)c.q + off;
    const float* __restrict__ dd = (const float*)c.d + off;
    const float* __restrict__ pp = (const float*)(par ? c.p : c.p_alt) + off;
    float* __restrict__ zz = (float*)(MG ? c.r : c.z) + off;
    float* __restrict__ xx = xfield + off;
    const float2 alpha = dup((float)sv.alpha), malpha = dup(-(float)sv.alpha);
    const float2 zs = dup((sv.iters == 0 && (!MG || c.lazy_scale)) ? (float)sv.scale : 1.f);
    float4* ring = msm + threadIdx.x;   // [stage][array][thread]
    float4* cs = msm + kBRing * NA * kBT;   // [chunk][warp]: (|r|^2, rho) as float-float pairs
    const unsigned sring = smem_addr(ring);
    const int g0 = b.y * geo.y, g1 = min(geo.x, b.z * geo.y);   // this block's groups
    const int per = geo.y / kBT;          // groups of a thread per chunk
    const int n = (b.z - b.y) * per;
    auto fetch = [&](int i, int st) {
      const int g = g0 + i * kBT + threadIdx.x;
      const int m = i < n && g < g1 ? 16 : 0;
      const unsigned e = m ? 4u * (unsigned)g : 0u, sa = sring + (unsigned)st * (NA * kBT * 16);
      cp16(sa, zz + e, m);
      cp16(sa + kBT * 16, qq + e, m);
      if (!MG) cp16(sa + 2 * kBT * 16, dd + e, m);
      if (!DEFER) {
        cp16(sa + (NA - 2) * kBT * 16, pp + e, m);
        cp16(sa + (NA - 1) * kBT * 16, xx + e, m);
      }
    };
    fetch(0, 0);
    cp_commit();
    fetch(1, 1);
    cp_commit();
    FF rr{0.f, 0.f}, rho{0.f, 0.f};
    int st = 0, left = per, chunk = 0;
    for (int i = 0; i < n; ++i) {
      fetch(i + 2, st >= 1 ? st - 1 : kBRing - 1);
      cp_commit();
      cp_wait<2>();
      const int g = g0 + i * kBT + threadIdx.x;
      if (g < g1) {
        const float4* s = ring + st * NA * kBT;
        const unsigned e = 4u * (unsigned)g;
        float2 z[2], q[2];
        get_row(z, s);
        get_row(q, s + kBT);
        float g_rr = 0.f, g_rho = 0.f;
        if (MG) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            z[h] = __ffma2_rn(malpha, q[h], __fmul2_rn(zs, z[h]));
            g_rr = fmaf(z[h].x, z[h].x, g_rr);
            g_rr = fmaf(z[h].y, z[h].y, g_rr);
          }
        } else {
          float2 d[2];
          get_row(d, s + 2 * kBT);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const float2 w = make_float2(d[h].x != 0.f ? q[h].x / d[h].x : 0.f, d[h].y != 0.f ? q[h].y / d[h].y : 0.f);
            z[h] = __ffma2_rn(malpha, w, __fmul2_rn(zs, z[h]));
            const float2 r = __fmul2_rn(d[h], z[h]);
            g_rho = fmaf(r.x, z[h].x, g_rho);
            g_rho = fmaf(r.y, z[h].y, g_rho);
            g_rr = fmaf(r.x, r.x, g_rr);
            g_rr = fmaf(r.y, r.y, g_rr);
          }
        }
        *reinterpret_cast<float4*>(zz + e) = make_float4(z[0].x, z[0].y, z[1].x, z[1].y);
        if (!DEFER) {
          float2 p[2], x[2];
          get_row(p, s + (NA - 2) * kBT);
          get_row(x, s + (NA - 1) * kBT);
#pragma unroll
          for (int h = 0; h < 2; ++h) x[h] = __ffma2_rn(alpha, p[h], x[h]);
          *reinterpret_cast<float4*>(xx + e) = make_float4(x[0].x, x[0].y, x[1].x, x[1].y);
        }
        rr = ff_add(rr, g_rr);
        if (!MG) rho = ff_add(rho, g_rho);
      }
      st = st + 1 == kBRing ? 0 : st + 1;
      if (--left == 0) {   // a chunk done: the warp's sums (fixed lane order)
        const FF s0 = row_reduce_ff(rr, 32), s1 = MG ? FF{0.f, 0.f} : row_reduce_ff(rho, 32);
        if (lane == 0) cs[chunk * (kBT / 32) + warp] = make_float4(s0.hi, s0.lo, s1.hi, s1.lo);
        rr = rho = FF{0.f, 0.f};
        left = per;
        ++chunk;
      }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < b.z - b.y; k += kBT) {
      double t0 = 0.0, t1 = 0.0;
      for (int w = 0; w < kBT / 32; ++w) {
        const float4 f = cs[k * (kBT / 32) + w];
        t0 += (double)f.x + (double)f.y;
        if (!MG) t1 += (double)f.z + (double)f.w;
      }
      slot_rr[b.y + k] = t0;
      if (!MG) slot_rho[b.y + k] = t1;
    }
  }
  // the replicate's last block adds its chunks in a fixed order; the last
  // replicate sets the loop condition
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(&c.mcnt[rep], 1) == b.w - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (sv.active) {
    double t0 = 0.0, t1 = 0.0;
#pragma unroll 8
    for (int i = threadIdx.x; i < geo.z; i += kBT) {
      t0 += __ldcg(&slot_rr[i]);
      if (!MG) t1 += __ldcg(&slot_rho[i]);
    }
    for (int o = 16; o > 0; o >>= 1) {
      t0 += __shfl_xor_sync(0xffffffffu, t0, o);
      if (!MG) t1 += __shfl_xor_sync(0xffffffffu, t1, o);
    }
    if (lane == 0) {
      s_sum[0][warp] = t0;
      s_sum[1][warp] = t1;
    }
    __syncthreads();
  }
  if (threadIdx.x != 0) return;
  c.mcnt[rep] = 0;
  if (sv.active) {
    double t0 = 0.0, t1 = 0.0;
    for (int w = 0; w < kBT / 32; ++w) {
      t0 += s_sum[0][w];
      t1 += s_sum[1][w];
    }
    RepSolve& s = c.solve[rep];
    s.iters += 1;
    s.pend = DEFER;
    s.pbuf = c.sync->parity ? 0 : 1;
    if (!isfinite(t0) || !isfinite(t1)) {
      c.sync->error = 1;
      s.active = 0;
    } else {
      if (!MG) {   // the V-cycle form sets beta and rho after z = M r
        s.beta = t1 / s.rho;
        s.rho = t1;
      }
      s.rnorm2 = t0;
      const bool conv = sqrt(t0) <= s.rtol * sqrt(s.bnorm2);
      if (conv || s.iters >= s.maxit) s.active = 0;
    }
  }
  __threadfence();
  if (atomicAdd(&c.sync->ticket, 1u) != (unsigned)c.n_reps - 1u) return;
  __threadfence();
  c.sync->ticket = 0u;
  int n_active = 0;
  for (int r = 0; r < c.n_reps; ++r) n_active += *(volatile int*)&c.solve[r].active;
  c.sync->active_count = n_active;
  c.sync->parity ^= 1;
  const int g = ++c.sync->guard;
  bool go = n_active > 0 && *(volatile int*)&c.sync->error != SYNC_ERR_TIMEOUT;
  if (go && g >= c.sync->guard_limit) {
    // every replicate stops at maxit; this only guards the graph loop
    c.sync->error = 2;
    go = false;
  }
  set_cond(cnd, go);
}

template <int NT>
bool a_init() {
  return cudaFuncSetAttribute((const void*)k_cg_a<NT, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)a_smem(NT)) == cudaSuccess &&
         cudaFuncSetAttribute((const void*)k_cg_a<NT, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)a_smem(NT)) == cudaSuccess;
}
template <bool MG, bool DEFER>
bool b_init() {
  return cudaFuncSetAttribute((const void*)k_cg_b<MG, DEFER>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)b_smem<MG, DEFER>()) == cudaSuccess;
}
template <int NT>
void a_launch(const Ctx& c, int which, bool defer) {
  const dim3 t(NT);
  if (c.flat) {
    const dim3 gf(std::min(c.n_ablk, flat_blocks(NT) * c.sm_count));
    if (defer) launch_k(c.pdl != 0, k_cg_a_flat<NT, true>, gf, t, 0, c.stream, c, which);
    else launch_k(c.pdl != 0, k_cg_a_flat<NT, false>, gf, t, 0, c.stream, c, which);
    return;
  }
  const dim3 g(c.n_ablk);
  if (defer) launch_k(c.pdl != 0, k_cg_a<NT, true>, g, t, a_smem(NT), c.stream, c, which);
  else launch_k(c.pdl != 0, k_cg_a<NT, false>, g, t, a_smem(NT), c.stream, c, which);
}

}  // namespace

// Dynamic shared memory of the passes in the current context.
bool cg_init() {
  const bool ok = a_init<64>() && a_init<128>() && a_init<256>() && b_init<true, true>() && b_init<true, false>() &&
                  b_init<false, true>() && b_init<false, false>();
  if (!ok) (void)cudaGetLastError();
  return ok;
}

// Tilings and blocks of the passes over the lattices `reps` (host tables;
// sums per tile segment and per chunk, whose geometry depends on the lattice
// alone); returns the reduction slots needed.
long long cg_plan(const std::vector<RepDesc>& reps, int sm_count, std::vector<MGLevel>& lv, std::vector<int4>& ablk,
                  std::vector<int4>& bblk, std::vector<int4>& bgeo, int* a_nt) {
  std::vector<MGLevel*> set;
  std::vector<int> ids;
  long long slots = 0;
  lv.assign(reps.size(), MGLevel{});
  for (size_t i = 0; i < reps.size(); ++i) {
    MGLevel& L = lv[i];
    L.nx = reps[i].nx;
    L.ny = reps[i].ny;
    L.nz = reps[i].nz;
    L.pitch = reps[i].nxp;
    march_tile(L, 1);
    L.slot0 = (int)slots;
    slots += 3LL * L.tx * L.ty * L.nseg;   // (the residual sweep has three sums)
    set.push_back(&L);
    ids.push_back((int)i);
  }
  march_blocks(set, ids, sm_count, 4, ablk);
  *a_nt = march_threads(set);
  // pass B: chunks of at least 1024 groups, at most 4096 of them a lattice;
  // blocks for one wave at 4 per multiprocessor
  long long bslots = 0, chunks = 0;
  for (size_t i = 0; i < reps.size(); ++i) {
    const long long ng = (long long)reps[i].gpr * reps[i].ny * reps[i].nz;
    long long per = 4 * kBT;
    while ((ng + per - 1) / per > 4096) per *= 2;
    if (ng <= 64 * per) per = kBT;   // small lattices: a block per chunk
    const int nc = (int)((ng + per - 1) / per);
    bgeo.push_back(make_int4((int)ng, (int)per, nc, (int)bslots));
    bslots += 2LL * nc;
    chunks += nc;
  }
  const long long share = std::min<long long>(kBMaxChunks, std::max<long long>(1, (chunks + 4LL * sm_count - 1) / (4LL * sm_count)));
  for (size_t i = 0; i < reps.size(); ++i) {
    const int nc = bgeo[i].z, nb = (int)((nc + share - 1) / share);
    for (int k = 0; k < nb; ++k)
      bblk.push_back(make_int4((int)i, (int)((long long)nc * k / nb), (int)((long long)nc * (k + 1) / nb), nb));
  }
  return std::max(slots, bslots);
}

void launch_cg_a(const Ctx& c, int which, bool defer) {
  switch (c.a_nt) {
    case 64: a_launch<64>(c, which, defer); break;
    case 128: a_launch<128>(c, which, defer); break;
    default: a_launch<256>(c, which, defer); break;
  }
}

void launch_cg_b(const Ctx& c, int which, void* xfield, bool defer, CondArg cnd) {
  const dim3 g(c.n_bblk), t(kBT);
  float* x = (float*)xfield;
  const bool pdl = c.pdl != 0;
  if (c.mg && defer) launch_k(pdl, k_cg_b<true, true>, g, t, b_smem<true, true>(), c.stream, c, which, x, cnd);
  else if (c.mg) launch_k(pdl, k_cg_b<true, false>, g, t, b_smem<true, false>(), c.stream, c, which, x, cnd);
  else if (defer) launch_k(pdl, k_cg_b<false, true>, g, t, b_smem<false, true>(), c.stream, c, which, x, cnd);
  else launch_k(pdl, k_cg_b<false, false>, g, t, b_smem<false, false>(), c.stream, c, which, x, cnd);
}

}  // namespace hca
