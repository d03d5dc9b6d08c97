// Plane-marching multigrid sweeps for FP32 fields: everything a V-cycle does
// on one grid level (the lattice or a coarse grid level, single lattices and
// batches) in two kernels,
//
//   k_mg_down  both pre-sweeps, the residual, its restriction and the part of
//              the first post-sweep that does not need the coarse correction;
//   k_mg_up    the prolongation and both post-sweeps (on the lattice also
//              rho = r.z and beta).
//
// With w = 1 / d, c the level's coupling and W1, W2 the Chebyshev weights:
//   u  = W1 w r                                  first sweep (from zero)
//   v  = u + W2 w (r - A u) = K u + W2 c w S(u)   second sweep, d u = W1 r,
//                                                K = 1 + W2 (1 - W1) / W1
//   res = r + c S(v) - d v,  rhs of the next level = its sum over children
//   v' = v + W2 w res
//   y  = v' + (1 - W2) p + W2 c w S(p)            first post-sweep of v + p,
//                                                p = P x_coarse
//   x  = (1 - W1) y + W1 w (r + c S(y))           second post-sweep
// with S the sum over the in-box neighbours.  Algorithmic traffic per site:
// down reads r, d, writes v' and 1/8 of a coarse site (12.5 B); up reads v',
// r, d and 1/8 of a coarse site and writes x (16.5 B): 29 B a V-cycle.
//
// Form.  A block of kMT threads owns a tile of 4-site groups by row pairs (a
// thread holds a 4 x 2 patch) and walks up z through a slab of planes.  The
// tile includes the halo the fused sweeps need (one group in x, two rows in
// y; two planes in z), so every thread runs the same code and only interior
// threads write.  Each plane's inputs arrive by tensor copies (zeros outside
// the level) in a shared-memory ring, two planes ahead; z neighbours stay in
// registers (the loop body is unrolled by three, so nothing is rotated), y
// neighbours go through shared memory (one barrier per plane), x neighbours
// through lane shuffles.  Bound: shared-memory and shuffle traffic and the
// latency a barrier a plane exposes at 16 warps per multiprocessor.  Measured
// at 256^3 (FP32): down 64 us and up 66 us a launch (74 and 92 with a
// per-thread cp.async of each patch), against 110 us for the pre-sweep and
// restriction kernels and 118 us for the two post-sweep kernels they replaced
// (28.5 B a site each); on 16 uneven replicates (59 M sites, all levels'
// launches apart) 124 and 131 us, against 449 and 495 us.
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "march.cuh"

namespace hca {

namespace {

constexpr int kDownRing = 5;          // planes k - 2 .. k + 2 of r and d
constexpr int kUpRing = 3;            // planes k .. k + 2 of v' and d, k - 1 .. k + 1 of r
constexpr float kW1 = (float)MG_W1, kW2 = (float)MG_W2;
constexpr float kK = (float)(1.0 + MG_W2 * (1.0 - MG_W1) / MG_W1);
constexpr float k1W1 = (float)(1.0 - MG_W1), k1W2 = (float)(1.0 - MG_W2);
constexpr size_t down_smem(int nt) { return (size_t)(kDownRing * 4 + 2 * 2 + 2 * 2) * nt * 16 + 128; }
constexpr size_t up_smem(int nt) { return (size_t)(kUpRing * 6 + 2 * 2 + 2) * nt * 16 + (size_t)kMaxSeg * (nt / 32) * 8 + 128; }

// The coupling of level l of the operator: the lattice's FP32 coupling times
// the level's scale.
__device__ __forceinline__ float level_coupling(const Ctx& c, int rep, int which, const MGLevel& L) {
  return c.reps[rep].cpl32[which] * L.cscale32;
}

// On the first application of a rescaled inner solve the stored residual is
// still unscaled: the factor the lattice kernels apply to r as they read it.
__device__ __forceinline__ float r_scale(const RepSolve& sv) { return sv.iters == 0 ? (float)sv.scale : 1.f; }

// ------------------------------------------------------------------ down --
template <bool LAT, int NT>
__global__ void __launch_bounds__(NT, blocks_per_sm(NT)) k_mg_down(Ctx c, int which, int l, const int4* __restrict__ blocks) {
  extern __shared__ __align__(16) float4 msm[];
  const int4 b = blocks[blockIdx.x];
  const int rep = b.x;
  const MGLevel& L = ((const MGLevel*)c.mg_lv)[rep * MG_MAXLEV + l];
  const MGLevel& C = (&L)[1];
  const Patch p = patch_of<NT, 2>(L, b);
  const int zb = b.z, ze = b.w;
  const float cpl = level_coupling(c, rep, which, L);
  const float2 w2c = dup(kW2 * cpl);
  const CUtensorMap* maps = c.tmaps + L.map0;   // r, d, v'
  float* __restrict__ vv = (float*)L.t;
  float* __restrict__ rc = (float*)C.rhs;
  const uint32_t box = 32u * (uint32_t)(L.cols * L.pairs);
  __shared__ __align__(8) uint64_t bar[kDownRing];
  mbars_init(bar, kDownRing, maps, 2);
  const bool two = p.x0 / 2 + 1 < C.nx;
  const unsigned cel = (unsigned)(p.x0 / 2) + (unsigned)C.pitch * (unsigned)(p.y0 / 2), csz = (unsigned)C.pitch * (unsigned)C.ny;
  HCA_VC_ENTRY(c);
  float sc = 1.f;
  if (c.skip_idle && !c.solve[rep].active) return;   // this replicate's solve has ended
  if (LAT) sc = r_scale(c.solve[rep]);
  const float2 w1s = dup(LAT ? kW1 * sc : kW1);
  float4* ring = align128(msm);                // [plane mod kDownRing][r, d][row][group]
  float4* ub = ring + kDownRing * 4 * NT;      // [plane & 1][row of the pair][thread]
  float4* vb = ub + 4 * NT;
  auto fetch = [&](int k, int slot) {
    mbar_expect_tx(&bar[slot], 2 * box);
    tma_load_3d(ring + (slot * 4) * NT, &maps[0], p.tx0, p.ty0, k, &bar[slot]);
    tma_load_3d(ring + (slot * 4 + 2) * NT, &maps[1], p.tx0, p.ty0, k, &bar[slot]);
  };
  P8 u[3], v[3], w[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    zero_patch(u[i]);
    zero_patch(v[i]);
    zero_patch(w[i]);
  }
  float2 acc = make_float2(0.f, 0.f);
  const int k0 = zb - 2, k1 = ze + 1;   // planes whose u is formed
  int issued = 2;   // (thread 0)
  if (p.tid == 0) {
    fetch(k0, 0);
    fetch(k0 + 1, 1);
  }
  int slot = 0;
  uint32_t par = 0;
  // one plane: u of plane k, v of plane k - 1, the residual of plane k - 2;
  // false when a copy timed out (the same in every thread)
  auto step = [&](auto ph, int k) {
    constexpr int P0 = decltype(ph)::value, P1 = (P0 + 2) % 3, P2 = (P0 + 1) % 3;   // planes k, k - 1, k - 2
    if (p.tid == 0 && k + 2 <= k1) {
      fetch(k + 2, slot + 2 >= kDownRing ? slot + 2 - kDownRing : slot + 2);
      ++issued;
    }
    const bool ok = tc::mbar_wait(&bar[slot], par, kTmaWaitLimit);
    float4* U0 = ub + (k & 1) * 2 * NT;
    const float4* U1 = ub + ((k & 1) ^ 1) * 2 * NT;
    float4* V1 = vb + ((k & 1) ^ 1) * 2 * NT;
    const float4* V2 = vb + (k & 1) * 2 * NT;
    // every read of shared memory and every lane exchange first: they depend
    // on nothing formed in this step (the sums still lack the plane above)
    const float4* rs = ring + slot * 4 * NT;
    float2 r[2][2], d[2][2];
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      get_row(r[a], rs + (a ? p.r1 : p.r0));
      get_row(d[a], rs + 2 * NT + (a ? p.r1 : p.r0));
    }
    nb_patch<NT>(p, U1, u[P1], u[P2], u[P2]);
    nb_patch<NT>(p, V2, v[P2], v[P0], v[P0]);
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        w[P0].v[a][h] = inv_d(d[a][h]);
        u[P0].v[a][h] = __fmul2_rn(__fmul2_rn(w1s, w[P0].v[a][h]), r[a][h]);
      }
    put_patch<NT>(p, U0, u[P0]);
    {
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int h = 0; h < 2; ++h)
          v[P1].v[a][h] = __ffma2_rn(__fmul2_rn(w2c, w[P1].v[a][h]), __fadd2_rn(u[P2].v[a][h], u[P0].v[a][h]),
                                     __fmul2_rn(dup(kK), u[P1].v[a][h]));
      put_patch<NT>(p, V1, v[P1]);
      // the residual of plane k - 2
      if (k >= zb + 2) {
        const int z = k - 2;
        if (p.out) {
          const float4* rz = ring + (slot >= 2 ? slot - 2 : slot - 2 + kDownRing) * 4 * NT;
          const unsigned e = p.e + (unsigned)z * p.sz;
          float2 pl = make_float2(0.f, 0.f);
#pragma unroll
          for (int a = 0; a < 2; ++a) {
            float2 r[2], d[2], o[2], res[2];
            get_row(r, rz + (a ? p.r1 : p.r0));
            get_row(d, rz + 2 * NT + (a ? p.r1 : p.r0));
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const float2 vc = v[P2].v[a][h];
              const float2 rn = __ffma2_rn(dup(cpl), __fadd2_rn(v[P0].v[a][h], v[P1].v[a][h]),
                                           LAT ? __fmul2_rn(r[h], dup(sc)) : r[h]);
              res[h] = __ffma2_rn(make_float2(-d[h].x, -d[h].y), vc, rn);
              o[h] = __ffma2_rn(__fmul2_rn(dup(kW2), w[P2].v[a][h]), res[h], vc);
            }
            if (p.part) {   // padding sites are no children
              if (p.x0 + 1 >= p.nx) res[0].y = 0.f;
              if (p.x0 + 2 >= p.nx) res[1].x = 0.f;
              if (p.x0 + 3 >= p.nx) res[1].y = 0.f;
            }
            if (a == 0 || p.rok[1]) {
              const float2 pr = make_float2(res[0].x + res[0].y, res[1].x + res[1].y);
              pl = a == 0 ? pr : __fadd2_rn(pl, pr);
              *reinterpret_cast<float4*>(vv + e + a * p.sy) = make_float4(o[0].x, o[0].y, o[1].x, o[1].y);
            }
          }
          // the children's sum: rows, then planes
          if (z & 1) pl = __fadd2_rn(acc, pl);
          else acc = pl;
          if ((z & 1) || z == p.nz - 1) {
            float* q = rc + (cel + (unsigned)(z >> 1) * csz);
            q[0] = pl.x;
            if (two) q[1] = pl.y;
          }
        }
      }
    }
    slot = slot + 1 == kDownRing ? 0 : slot + 1;
    par ^= slot == 0;
    return !__syncthreads_or(!ok);
  };
  for (int k = k0; k <= k1; k += 3) {
    if (!step(std::integral_constant<int, 0>{}, k) ||
        (k + 1 <= k1 && !step(std::integral_constant<int, 1>{}, k + 1)) ||
        (k + 2 <= k1 && !step(std::integral_constant<int, 2>{}, k + 2))) {
      tma_abort(c, bar, kDownRing, k - k0, issued);
      return;
    }
  }
}

// -------------------------------------------------------------------- up --
template <bool LAT, int NT>
__global__ void __launch_bounds__(NT, blocks_per_sm(NT)) k_mg_up(Ctx c, int which, int l, const int4* __restrict__ blocks) {
  extern __shared__ __align__(16) float4 msm[];
  const int4 b = blocks[blockIdx.x];
  const int rep = b.x;
  const MGLevel& L = ((const MGLevel*)c.mg_lv)[rep * MG_MAXLEV + l];
  const MGLevel& C = (&L)[1];
  const Patch p = patch_of<NT, 2>(L, b);
  const int zb = b.z, ze = b.w;
  const float cpl = level_coupling(c, rep, which, L);
  const float2 w2c = dup(kW2 * cpl);
  const CUtensorMap* maps = c.tmaps + L.map0;   // r, d, v'
  const float* __restrict__ xc = (const float*)C.x;
  const uint32_t box = 32u * (uint32_t)(L.cols * L.pairs);
  __shared__ __align__(8) uint64_t bar[kUpRing];
  mbars_init(bar, kUpRing, maps, 3);
  float* __restrict__ xo = (float*)L.x;
  const int cnz = C.nz;
  const bool two = p.x0 / 2 + 1 < C.nx;
  const unsigned csz = (unsigned)C.pitch * (unsigned)C.ny;
  const unsigned cel = p.rok[0] ? (unsigned)(p.x0 / 2) + (unsigned)C.pitch * (unsigned)(p.y0 / 2) : 0u;
  HCA_VC_ENTRY(c);
  float sc = 1.f;
  if (c.skip_idle && !c.solve[rep].active) return;
  if (LAT) sc = r_scale(c.solve[rep]);
  float4* ring = align128(msm);             // [phase][v', d, r (of the plane before)][row][group]
  float4* yb = ring + kUpRing * 6 * NT;     // [plane & 1][row of the pair][thread]
  float2* cells = reinterpret_cast<float2*>(yb + 4 * NT);   // [coarse plane & 3][thread]: the patch's two coarse cells
  float2* segs = cells + 4 * NT;
  const unsigned scell = smem_addr(cells + p.tid);
  // v' and d of plane k, r of plane k - 1 (used one step later)
  auto fetch = [&](int k, int slot) {
    mbar_expect_tx(&bar[slot], 3 * box);
    tma_load_3d(ring + (slot * 6) * NT, &maps[2], p.tx0, p.ty0, k, &bar[slot]);
    tma_load_3d(ring + (slot * 6 + 2) * NT, &maps[1], p.tx0, p.ty0, k, &bar[slot]);
    tma_load_3d(ring + (slot * 6 + 4) * NT, &maps[0], p.tx0, p.ty0, k - 1, &bar[slot]);
  };
  auto fetch_cells = [&](int Z) {
    const bool ok = p.rok[0] && Z >= 0 && Z < cnz;
    const unsigned sa = scell + (unsigned)(Z & 3) * (NT * 8);
    const unsigned e = ok ? cel + (unsigned)Z * csz : 0u;
    cp4(sa, xc + e, ok ? 4 : 0);
    cp4(sa + 4, xc + (two && ok ? e + 1 : 0u), two && ok ? 4 : 0);
  };
  P8 y[3], w[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    zero_patch(y[i]);
    zero_patch(w[i]);
  }
  FF acc{0.f, 0.f};
  const int k0 = zb - 1, k1 = ze;   // planes whose y is formed (k0 odd: zb is even)
  // coarse planes k0 / 2 - 1 .. k0 / 2 + 1 before the first step (-1 below the level: zeros)
  const int Z0 = k0 >> 1;
  int issued = 2;   // (thread 0)
  if (p.tid == 0) {
    fetch(k0, 0);
    fetch(k0 + 1, 1);
  }
  fetch_cells(Z0);
  fetch_cells(Z0 + 1);
  cp_commit();
  fetch_cells(Z0 + 2);
  cp_commit();
  // cell slots of the neighbours (clamped for outermost halo patches)
  const int cm = p.im - NT, cp = p.ip, cl = p.tid > 0 ? p.tid - 1 : 0, cr = p.tid + 1 < NT ? p.tid + 1 : p.tid;
  const bool yin = p.rok[1];
  float2 cur = make_float2(0.f, 0.f), below = cur;   // the patch's cells of the current coarse plane and of the one below
  cp_wait<1>();
  __syncthreads();
  int seg = 0;
  const int seglen = L.seg;
  uint32_t par = 0;
  auto step = [&](auto ph, int k) {
    constexpr int P0 = decltype(ph)::value, P1 = (P0 + 2) % 3, P2 = (P0 + 1) % 3;
    const bool odd = k & 1;
    const int Z = k >> 1;
    if (k + 2 <= k1) {
      if (p.tid == 0) {
        fetch(k + 2, P1);
        ++issued;
      }
      if (!odd) fetch_cells(Z + 2);
    }
    cp_commit();
    cp_wait<2>();
    const bool ok = tc::mbar_wait(&bar[P0], par, kTmaWaitLimit);
    const float2* cz = cells + (Z & 3) * NT;
    if (!odd || k == k0) {
      below = cur;
      cur = cz[p.tid];
    }
    // y of plane k - 1: its neighbours but the plane above
    nb_patch<NT>(p, yb + ((k & 1) ^ 1) * 2 * NT, y[P1], y[P2], y[P2]);
    // the coarse cells around the patch: in x, in the coarse rows below and
    // above, and along z: in its own cells, or the coarse plane below (even
    // planes) or above (odd planes)
    const float xl = cz[cl].y, xr = cz[cr].x;
    const float2 co = odd ? cells[((Z + 1) & 3) * NT + p.tid] : below;
    const float2 zn = (odd || k + 1 < p.nz) ? __fadd2_rn(co, cur) : co;
    // the row's y neighbours: one coarse row outside the cells, one inside
    const float2 t[2] = {__fadd2_rn(yin ? __fadd2_rn(cz[cm], cur) : cz[cm], zn), __fadd2_rn(__fadd2_rn(cz[cp], cur), zn)};
    const float both = cur.x + cur.y;
    float2 xs[2] = {make_float2(xl + cur.x, both), make_float2(both, cur.y + xr)};
    if (p.part) {   // no neighbour to the right of the level's last site
      if (p.x0 + 1 == p.nx) xs[0].x = xl;
      if (p.x0 + 2 == p.nx) xs[0].y = cur.x;
      if (p.x0 + 3 == p.nx) xs[1].x = cur.x;
    }
    const float2 pw[2] = {__fmul2_rn(dup(k1W2), dup(cur.x)), __fmul2_rn(dup(k1W2), dup(cur.y))};
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      float2 vp[2], d[2];
      get_row(vp, ring + (P0 * 6) * NT + (a ? p.r1 : p.r0));
      get_row(d, ring + (P0 * 6 + 2) * NT + (a ? p.r1 : p.r0));
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float2 S = __fadd2_rn(xs[h], dup(h ? t[a].y : t[a].x));
        w[P0].v[a][h] = inv_d(d[h]);
        const float2 yv = __ffma2_rn(__fmul2_rn(w2c, w[P0].v[a][h]), S, __fadd2_rn(pw[h], vp[h]));
        y[P0].v[a][h] = make_float2(d[h].x > 0.f ? yv.x : 0.f, d[h].y > 0.f ? yv.y : 0.f);
      }
    }
    put_patch<NT>(p, yb + (k & 1) * 2 * NT, y[P0]);
    if (k > zb) {
      const int z = k - 1;
      if (p.out) {
        const unsigned e = p.e + (unsigned)z * p.sz;
#pragma unroll
        for (int a = 0; a < 2; ++a) {
          float2 r[2], o[2], rz = make_float2(0.f, 0.f);
          get_row(r, ring + (P0 * 6 + 4) * NT + (a ? p.r1 : p.r0));
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const float2 rs = LAT ? __fmul2_rn(r[h], dup(sc)) : r[h];
            const float2 rn = __ffma2_rn(dup(cpl), __fadd2_rn(y[P2].v[a][h], y[P0].v[a][h]), rs);
            o[h] = __ffma2_rn(__fmul2_rn(dup(kW1), w[P1].v[a][h]), rn, __fmul2_rn(dup(k1W1), y[P1].v[a][h]));
            if (LAT) rz = __ffma2_rn(rs, o[h], rz);
          }
          if (a == 0 || p.rok[1]) {
            *reinterpret_cast<float4*>(xo + e + a * p.sy) = make_float4(o[0].x, o[0].y, o[1].x, o[1].y);
            if (LAT) acc = ff_add(acc, rz.x + rz.y);
          }
        }
      }
      if (LAT && (((z + 1) % seglen) == 0 || z == ze - 1)) {
        // the segment's sum over this warp's patches (fixed lane order)
        const FF s = row_reduce_ff(acc, 32);
        if (p.lane == 0) segs[seg * (NT / 32) + (p.tid >> 5)] = make_float2(s.hi, s.lo);
        acc = FF{0.f, 0.f};
        ++seg;
      }
    }
    return !__syncthreads_or(!ok);
  };
  for (int k = k0; k <= k1; k += 3, par ^= 1) {
    if (!step(std::integral_constant<int, 0>{}, k) ||
        (k + 1 <= k1 && !step(std::integral_constant<int, 1>{}, k + 1)) ||
        (k + 2 <= k1 && !step(std::integral_constant<int, 2>{}, k + 2))) {
      tma_abort(c, bar, kUpRing, k - k0, issued);   // (goes on to its arrival)
      break;
    }
  }
  if (!LAT) return;
  // the block's segment sums to their slots (warps in order), then the
  // replicate's last block adds all slots in a fixed order
  double* slots = c.mslot + L.slot0 + (long long)b.y * L.nseg + zb / seglen;
  for (int s = threadIdx.x; s < seg; s += NT) {
    double t = 0.0;
    for (int q = 0; q < NT / 32; ++q) {
      const float2 f = segs[s * (NT / 32) + q];
      t += (double)f.x + (double)f.y;
    }
    slots[s] = t;
  }
  march_finish(c, rep, L.nblk, c.mslot + L.slot0, L.tx * L.ty * L.nseg, [&](double rz) {
    RepSolve& s = c.solve[rep];
    if (!s.active) return;
    if (!(rz > 0.0) || !isfinite(rz)) {
      if (!isfinite(rz)) c.sync->error = 1;
      s.active = 0;
      return;
    }
    s.beta = s.iters == 0 ? 0.0 : rz / s.rho;
    s.rho = rz;
  });
}

}  // namespace

// ---------------------------------------------------------- configuration --
int march_threads(const std::vector<MGLevel*>& lv);
// Segments below which a lattice's segments are cut shorter: near the number of
// multiprocessors, but the same on every chip, as segments shape the sums.
constexpr int kFewSegs = 128;

// Tiling of a level: the fewest tiles of kMT patches (every halo patch is
// redundant work).  It depends on the level's shape alone, as do the segment
// sums, so results do not depend on slabs, batches or launch forms.
void march_tile(MGLevel& L, int halo_rows) {
  const int gpr = (L.nx + 3) / 4;
  long long best = -1;
  for (int n = 1; n <= gpr; ++n) {
    const int ox = (gpr + n - 1) / n, cols = ox + 2, pairs = std::min(kMT / cols, 128);
    const int most = 2 * pairs - 2 * halo_rows;   // rows of the interior
    if (most < 2 || 4 * cols > 256) continue;   // (a tensor copy's box: at most 256 elements a side)
    int ty = (L.ny + most - 1) / most;
    const int oy = ((L.ny + ty - 1) / ty + 1) / 2 * 2;   // even shares
    const int tx = (gpr + ox - 1) / ox;
    ty = (L.ny + oy - 1) / oy;
    const long long cost = (long long)tx * ty;
    if (best < 0 || cost < best) {
      best = cost;
      L.cols = cols;
      L.pairs = oy / 2 + halo_rows;
      L.ox = ox;
      L.oy = oy;
      L.tx = tx;
      L.ty = ty;
    }
    if (cols <= 6) break;
  }
  // planes per reduction segment (even, so a slab starts on a coarse plane);
  // shorter on lattices of few tiles, whose slabs of whole segments would leave
  // multiprocessors idle (oxygen solve with Jacobi, 43 x 41 x 300: 1.46 ms, 2.06
  // with 16 planes a segment, 1.75 with the row kernels before)
  L.seg = L.nz > 256 ? 16 : L.nz > 128 ? 8 : L.nz > 64 ? 4 : 2;
  while (L.seg > 2 && (long long)L.tx * L.ty * ((L.nz + L.seg - 1) / L.seg) < kFewSegs) L.seg /= 2;
  L.nseg = (L.nz + L.seg - 1) / L.seg;
}

// The blocks (replicate, tile, slab) of one level's launches over the
// replicates that sweep it on the grid: slabs of whole segments, as thick as
// balances the planes of a slab's halo and start-up (extra) against idle
// multiprocessors.
void march_blocks(std::vector<MGLevel*>& lv, const std::vector<int>& reps, int sm_count, int extra,
                  std::vector<int4>& out) {
  const long long resident = (long long)blocks_per_sm(march_threads(lv)) * sm_count;
  // a block has slots for kMaxSeg segments (the last one may be partial)
  auto slab = [](const MGLevel& L, int zs) { return std::min(L.nz, std::min((zs + L.seg - 1) / L.seg, kMaxSeg) * L.seg); };
  int best_zs = 0;
  double best = -1;
  for (int zs = 2; zs <= 1024; zs = zs < 64 ? zs + 2 : zs + 8) {
    long long nb = 0;
    double work = 0, longest = 0;
    bool more = false;
    for (MGLevel* L : lv) {
      const int z = slab(*L, zs), ns = (L->nz + z - 1) / z;
      if (z < L->nz && z < kMaxSeg * L->seg) more = true;
      nb += (long long)ns * L->tx * L->ty;
      work += (double)ns * L->tx * L->ty * (z + extra);
      longest = std::max(longest, z + (double)extra);
    }
    // whole waves while there are few, an even share plus a tail beyond
    const double waves = (double)nb / resident;
    const double t = waves <= 4 ? std::max(1.0, std::ceil(waves)) * longest : work / resident + 0.5 * longest;
    if (best < 0 || t < best) {
      best = t;
      best_zs = zs;
    }
    if (!more) break;
  }
  for (size_t i = 0; i < lv.size(); ++i) {
    MGLevel& L = *lv[i];
    const int z = slab(L, best_zs);
    L.nblk = 0;
    for (int zb = 0; zb < L.nz; zb += z)
      for (int ty = 0; ty < L.ty; ++ty)
        for (int tx = 0; tx < L.tx; ++tx) {
          out.push_back(make_int4(reps[i], ty * L.tx + tx, zb, std::min(L.nz, zb + z)));
          ++L.nblk;
        }
  }
}

namespace {
template <int NT>
bool march_init_t() {
  const void* fn[4] = {(const void*)k_mg_down<true, NT>, (const void*)k_mg_down<false, NT>,
                       (const void*)k_mg_up<true, NT>, (const void*)k_mg_up<false, NT>};
  for (int i = 0; i < 4; ++i)
    if (cudaFuncSetAttribute(fn[i], cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(i < 2 ? down_smem(NT) : up_smem(NT))) != cudaSuccess) {
      (void)cudaGetLastError();
      return false;
    }
  return true;
}

template <int NT>
void launch_march_t(const Ctx& c, int which, const MGHost& H, int l, bool down) {
  const dim3 g(H.mb_n[l]), t(NT);
  const int4* bl = c.mblk + H.mb_off[l];
  const bool pdl = c.pdl != 0;
  if (down && l == 0) launch_k(pdl, k_mg_down<true, NT>, g, t, down_smem(NT), c.stream, c, which, l, bl);
  else if (down) launch_k(pdl, k_mg_down<false, NT>, g, t, down_smem(NT), c.stream, c, which, l, bl);
  else if (l == 0) launch_k(pdl, k_mg_up<true, NT>, g, t, up_smem(NT), c.stream, c, which, l, bl);
  else launch_k(pdl, k_mg_up<false, NT>, g, t, up_smem(NT), c.stream, c, which, l, bl);
}
}  // namespace

// A tensor map of one array of a level (x extent nx, rows `pitch` apart), box a
// tile's rows of one plane, zero fill outside.  False if the driver's entry
// point is missing or refuses the encoding.
bool march_map(CUtensorMap* m, const MGLevel& L, const void* base) {
  using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
      q != cudaDriverEntryPointSuccess || !fn) {
    (void)cudaGetLastError();
    return false;
  }
  const cuuint64_t dims[3] = {(cuuint64_t)L.nx, (cuuint64_t)L.ny, (cuuint64_t)L.nz};
  const cuuint64_t strides[2] = {(cuuint64_t)L.pitch * 4, (cuuint64_t)L.pitch * L.ny * 4};
  const cuuint32_t box[3] = {(cuuint32_t)(4 * L.cols), (cuuint32_t)(2 * L.pairs), 1};
  const cuuint32_t es[3] = {1, 1, 1};
  return ((Encode)fn)(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(base), dims, strides, box, es,
                      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Dynamic shared memory of the marching kernels in the current context.
bool march_init() { return march_init_t<64>() && march_init_t<128>() && march_init_t<256>(); }

// Threads per block for a set of tilings.
int march_threads(const std::vector<MGLevel*>& lv) {
  int n = 64;
  for (const MGLevel* L : lv)
    while (n < L->cols * L->pairs) n *= 2;
  return n;
}

// k_mg_down (down) or k_mg_up on grid level l.
void launch_march(const Ctx& c, int which, const MGHost& H, int l, bool down) {
  if (H.mb_n[l] == 0) return;
  switch (H.mb_nt[l]) {
    case 64: launch_march_t<64>(c, which, H, l, down); break;
    case 128: launch_march_t<128>(c, which, H, l, down); break;
    default: launch_march_t<256>(c, which, H, l, down); break;
  }
}

}  // namespace hca
