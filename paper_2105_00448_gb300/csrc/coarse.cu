// The coarse levels of a V-cycle (FP32 fields) in one launch of thread-block
// clusters: one cluster per replicate keeps the levels from `lc` on in the
// shared memory of its blocks, so a sweep costs a cluster barrier instead of
// a kernel launch.
//
// The levels of more than MG_SMALL_SITES sites are cut into slabs of whole
// planes over the cluster's blocks (aligned between levels, so restriction
// and prolongation stay inside a block); a block reads the planes next to its
// slab from its neighbours' shared memory.  The smaller levels run in block 0
// (block barriers only).  A thread takes 4-site groups of a row; per site the
// arithmetic, with its roundings and its order of sums, is that of the
// plane-marching sweeps (march.cu), so where a level runs does not change a
// bit.
//
// Planes lie along z (rows along y), or along y (rows along z) on lattices
// with few z planes.
//
// Bound: the latency of ~45 dependent phases (a phase is 600-1500 cycles, a
// cluster barrier ~600): 19 us for the levels 32^3, 16^3 and 8^3, where a
// launch per sweep of 32^3 and the single-block kernel of the others took
// 37 us.
#include <cooperative_groups.h>

#include <algorithm>
#include <vector>

#include "hca_internal.cuh"

namespace cg = cooperative_groups;

namespace hca {

namespace {

constexpr int kCT = 512;              // threads per block
constexpr int kCLev = 12;             // most levels a cluster holds
constexpr float kW1 = (float)MG_W1, kW2 = (float)MG_W2;
constexpr float kK = (float)(1.0 + MG_W2 * (1.0 - MG_W1) / MG_W1);
constexpr float k1W1 = (float)(1.0 - MG_W1), k1W2 = (float)(1.0 - MG_W2);
constexpr float kWC = (float)MG_OMEGA_COARSE;

__device__ __forceinline__ float2 dup(float a) { return make_float2(a, a); }
__device__ __forceinline__ float inv_d(float d) {
  float w;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(w) : "f"(d));
  return d > 0.f ? w : 0.f;
}

struct Q4 {
  float2 v[2];
};
__device__ __forceinline__ Q4 ldq(const float* p) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  return Q4{{make_float2(q.x, q.y), make_float2(q.z, q.w)}};
}
__device__ __forceinline__ void stq(float* p, const Q4& q) {
  *reinterpret_cast<float4*>(p) = make_float4(q.v[0].x, q.v[0].y, q.v[1].x, q.v[1].y);
}
__device__ __forceinline__ Q4 zeroq() { return Q4{{make_float2(0.f, 0.f), make_float2(0.f, 0.f)}}; }
__device__ __forceinline__ Q4 invq(const Q4& d) {
  return Q4{{make_float2(inv_d(d.v[0].x), inv_d(d.v[0].y)), make_float2(inv_d(d.v[1].x), inv_d(d.v[1].y))}};
}

__device__ __forceinline__ float keep(float v, bool ok) { return ok ? v : 0.f; }
__device__ __forceinline__ Q4 keep(const Q4& q, bool ok) {
  return Q4{{make_float2(keep(q.v[0].x, ok), keep(q.v[0].y, ok)), make_float2(keep(q.v[1].x, ok), keep(q.v[1].y, ok))}};
}

// One level as this block sees it: its slab of np planes of nr rows of gpr
// groups, first plane o0 of no; arrays in shared memory (or global memory,
// for the right-hand side and the diagonal of the first level).
struct Slab {
  int nx, nr, gpr, no, np, o0;
  float *a, *b;                 // [plane][row][pitch]
  const float *r, *d;
  int rrow, rplane, drow, dplane;   // strides of r and d
  const float *alo, *ahi, *blo, *bhi;   // the neighbouring blocks' adjacent planes of a and b (null: none)
  float c;
  unsigned mg, mr, mc;          // reciprocals of gpr, nr and the coarse level's nr
};

// S of group (q, g) of local plane lp over array `arr` (its neighbour planes
// lo, hi), own the group itself.  zp: planes lie along z.
__device__ __forceinline__ Q4 nb_group(const Slab& s, const float* arr, const float* lo, const float* hi, int lp, int q,
                                       int g, bool zp, const Q4& own) {
  const int pitch = 4 * s.gpr, ps = pitch * s.nr, e = lp * ps + q * pitch + 4 * g, ei = q * pitch + 4 * g;
  // every read unconditional (of the group itself where there is no
  // neighbour, then dropped): branches would serialise their latencies
  const bool gl = g > 0, gr = g + 1 < s.gpr, ql = q > 0, qr = q + 1 < s.nr;
  const bool pl = lp > 0 || lo, pr = lp + 1 < s.np || hi;
  const float lft = keep(arr[gl ? e - 1 : e], gl), rgt = keep(arr[gr ? e + 4 : e], gr);
  const Q4 rm = keep(ldq(arr + (ql ? e - pitch : e)), ql), rp = keep(ldq(arr + (qr ? e + pitch : e)), qr);
  const float* am = lp > 0 ? arr + (e - ps) : lo ? lo + ei : arr + e;
  const float* ap = lp + 1 < s.np ? arr + (e + ps) : hi ? hi + ei : arr + e;
  const Q4 pm = keep(ldq(am), pl), pp = keep(ldq(ap), pr);
  const Q4 &ym = zp ? rm : pm, &yp = zp ? rp : pp, &zm = zp ? pm : rm, &zq = zp ? pp : rp;
  const float2 x[2] = {make_float2(lft + own.v[0].y, own.v[0].x + own.v[1].x),
                       make_float2(own.v[0].y + own.v[1].y, own.v[1].x + rgt)};
  Q4 S;
#pragma unroll
  for (int h = 0; h < 2; ++h)
    S.v[h] = __fadd2_rn(__fadd2_rn(__fadd2_rn(x[h], __fadd2_rn(ym.v[h], yp.v[h])), zm.v[h]), zq.v[h]);
  return S;
}

// t / d for t <= 512 by a rounded-up reciprocal m = 2^20 / d + 1: the excess
// t / 2^20 stays below 1 / d for d <= 512, and for larger d the quotient is 0.
__device__ __forceinline__ int div_small(int t, unsigned m) { return (int)(((unsigned)t * m) >> 20); }

// Items (local plane, row, group) of a slab, strided over the block.
struct Walk3 {
  int lp, q, g, dp, dq, dg, gpr, nr;
  __device__ __forceinline__ Walk3(int t, int gpr_, int nr_, unsigned mg, unsigned mr) : gpr(gpr_), nr(nr_) {
    int k = div_small(t, mg);
    g = t - k * gpr;
    lp = div_small(k, mr);
    q = k - lp * nr;
    k = div_small(kCT, mg);
    dg = kCT - k * gpr;
    dp = div_small(k, mr);
    dq = k - dp * nr;
  }
  __device__ __forceinline__ void next() {
    g += dg;
    int cy = g >= gpr;
    if (cy) g -= gpr;
    q += dq + cy;
    cy = q >= nr;
    if (cy) q -= nr;
    lp += dp + cy;
  }
};
__device__ __forceinline__ Q4 u_of(const Q4& r, const Q4& w) {
  Q4 u;
#pragma unroll
  for (int h = 0; h < 2; ++h) u.v[h] = __fmul2_rn(__fmul2_rn(dup(kW1), w.v[h]), r.v[h]);
  return u;
}

// a = u (first sweep from zero); rs: where to keep the first level's
// right-hand side, read from global memory here (null: it stays there)
__device__ __forceinline__ void phase_u(const Slab& s, const float* r, int rrow, int rplane, float* rs) {
  const int pitch = 4 * s.gpr, ps = pitch * s.nr, n = s.np * s.nr * s.gpr;
  Walk3 w(threadIdx.x, s.gpr, s.nr, s.mg, s.mr);
  for (int t = threadIdx.x; t < n; t += kCT, w.next()) {
    const Q4 q = ldq(r + w.lp * rplane + w.q * rrow + 4 * w.g), d = ldq(s.d + w.lp * s.dplane + w.q * s.drow + 4 * w.g);
    const int e = w.lp * ps + w.q * pitch + 4 * w.g;
    if (rs) stq(rs + e, q);
    stq(s.a + e, u_of(q, invq(d)));
  }
}

// b = v (second sweep)
__device__ __forceinline__ void phase_v(const Slab& s, bool zp) {
  const int pitch = 4 * s.gpr, ps = pitch * s.nr, n = s.np * s.nr * s.gpr;
  const float2 w2c = dup(kW2 * s.c);
  Walk3 k(threadIdx.x, s.gpr, s.nr, s.mg, s.mr);
  for (int t = threadIdx.x; t < n; t += kCT, k.next()) {
    const int e = k.lp * ps + k.q * pitch + 4 * k.g;
    const Q4 u = ldq(s.a + e), w = invq(ldq(s.d + k.lp * s.dplane + k.q * s.drow + 4 * k.g));
    const Q4 S = nb_group(s, s.a, s.alo, s.ahi, k.lp, k.q, k.g, zp, u);
    Q4 v;
#pragma unroll
    for (int h = 0; h < 2; ++h)
      v.v[h] = __ffma2_rn(__fmul2_rn(w2c, w.v[h]), S.v[h], __fmul2_rn(dup(kK), u.v[h]));
    stq(s.b + e, v);
  }
}

// The residual of v (b), a = v', and the right-hand side of the next level
// (rc, its planes from this slab's first on): a pair of lanes takes the two
// by two rows under a coarse group pair, a lane one of the two planes.
__device__ __forceinline__ void phase_r(const Slab& s, float* rc, int cpitch, int cnr, int cnx, bool zp) {
  const int pitch = 4 * s.gpr, ps = pitch * s.nr;
  const int ncp = (s.np + 1) >> 1, n = ncp * cnr * s.gpr;
  const int dpl = threadIdx.x & 1;
  Walk3 k(threadIdx.x >> 1, s.gpr, cnr, s.mg, s.mc);
  k.dg = 0;   // half the block's items per round
  {
    const int h = div_small(kCT / 2, s.mg);
    k.dg = kCT / 2 - h * s.gpr;
    k.dp = div_small(h, s.mc);
    k.dq = h - k.dp * cnr;
  }
  for (int t = threadIdx.x >> 1; t < ((n + 15) & ~15); t += kCT / 2, k.next()) {   // whole warps: the lanes exchange
    float2 row[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    const int lp = 2 * k.lp + dpl;
    const bool live = t < n && lp < s.np;
#pragma unroll
    for (int dr = 0; dr < 2; ++dr) {
      const int q = 2 * k.q + dr;
      if (!live || q >= s.nr) continue;
      const int e = lp * ps + q * pitch + 4 * k.g;
      const Q4 v = ldq(s.b + e), r = ldq(s.r + lp * s.rplane + q * s.rrow + 4 * k.g),
               d = ldq(s.d + lp * s.dplane + q * s.drow + 4 * k.g);
      const Q4 S = nb_group(s, s.b, s.blo, s.bhi, lp, q, k.g, zp, v), w = invq(d);
      Q4 res, o;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float2 rn = __ffma2_rn(dup(s.c), S.v[h], r.v[h]);
        res.v[h] = __ffma2_rn(make_float2(-d.v[h].x, -d.v[h].y), v.v[h], rn);
        o.v[h] = __ffma2_rn(__fmul2_rn(dup(kW2), w.v[h]), res.v[h], v.v[h]);
      }
      const int x0 = 4 * k.g;
      if (x0 + 1 >= s.nx) res.v[0].y = 0.f;
      if (x0 + 2 >= s.nx) res.v[1].x = 0.f;
      if (x0 + 3 >= s.nx) res.v[1].y = 0.f;
      row[dr] = make_float2(res.v[0].x + res.v[0].y, res.v[1].x + res.v[1].y);
      stq(s.a + e, o);
    }
    // (dz 0: dy 0 + dy 1) + (dz 1: dy 0 + dy 1), whichever way the planes lie
    float2 other[2];
#pragma unroll
    for (int dr = 0; dr < 2; ++dr) {
      other[dr].x = __shfl_xor_sync(0xffffffffu, row[dr].x, 1);
      other[dr].y = __shfl_xor_sync(0xffffffffu, row[dr].y, 1);
    }
    if (t < n && dpl == 0) {
      const float2 acc = zp ? __fadd2_rn(__fadd2_rn(row[0], row[1]), __fadd2_rn(other[0], other[1]))
                            : __fadd2_rn(__fadd2_rn(row[0], other[0]), __fadd2_rn(row[1], other[1]));
      float* out = rc + k.lp * cpitch * cnr + k.q * cpitch + 2 * k.g;
      out[0] = acc.x;
      if (2 * k.g + 1 < cnx) out[1] = acc.y;
    }
  }
}

// b = y (first post-sweep).  The coarse correction's planes lo .. hi - 1 are
// at ca, the ones next to them at clo and chi.
__device__ __forceinline__ void phase_y(const Slab& s, const float* ca, const float* clo, const float* chi, int lo, int hi,
                                        int cpitch, int cnr, int cno, int cnx, bool zp) {
  const int cps = cpitch * cnr;
  auto plane = [&](int O) { return O < lo ? clo : O >= hi ? chi : ca + (O - lo) * cps; };
  const int pitch = 4 * s.gpr, ps = pitch * s.nr, n = s.np * s.nr * s.gpr;
  const float2 w2c = dup(kW2 * s.c);
  Walk3 k(threadIdx.x, s.gpr, s.nr, s.mg, s.mr);
  for (int t = threadIdx.x; t < n; t += kCT, k.next()) {
    const int e = k.lp * ps + k.q * pitch + 4 * k.g, X = 2 * k.g;
    const int o = s.o0 + k.lp, O = o >> 1, Q = k.q >> 1;
    const int Oo = (o & 1) ? O + 1 : O - 1, Qo = (k.q & 1) ? Q + 1 : Q - 1;
    const bool two = X + 1 < cnx;
    const float* c0 = plane(O);
    const float* cp = Oo >= 0 && Oo < cno ? plane(Oo) : nullptr;
    const int ce = Q * cpitch + X, co = Qo * cpitch + X;
    auto pair = [&](const float* p, int i) { return p ? make_float2(p[i], two ? p[i + 1] : 0.f) : make_float2(0.f, 0.f); };
    const float2 cur = pair(c0, ce);
    const float2 pl = pair(cp, ce), rw = Qo >= 0 && Qo < cnr ? pair(c0, co) : make_float2(0.f, 0.f);
    const float xl = X > 0 ? c0[ce - 1] : 0.f, xr = X + 2 < cnx ? c0[ce + 2] : 0.f;
    const bool pin = (o & 1) || o + 1 < s.no, rin = (k.q & 1) || k.q + 1 < s.nr;
    const float2 fp = pin ? __fadd2_rn(pl, cur) : pl, fr = rin ? __fadd2_rn(rw, cur) : rw;
    const float2 tt = zp ? __fadd2_rn(fr, fp) : __fadd2_rn(fp, fr);
    const float both = cur.x + cur.y;
    float2 xs[2] = {make_float2(xl + cur.x, both), make_float2(both, cur.y + xr)};
    const int x0 = 4 * k.g;
    if (x0 + 1 == s.nx) xs[0].x = xl;
    if (x0 + 2 == s.nx) xs[0].y = cur.x;
    if (x0 + 3 == s.nx) xs[1].x = cur.x;
    const Q4 vp = ldq(s.a + e), d = ldq(s.d + k.lp * s.dplane + k.q * s.drow + 4 * k.g), w = invq(d);
    Q4 y;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float2 S = __fadd2_rn(xs[h], dup(h ? tt.y : tt.x));
      const float2 pw = __fmul2_rn(dup(k1W2), dup(h ? cur.y : cur.x));
      const float2 yv = __ffma2_rn(__fmul2_rn(w2c, w.v[h]), S, __fadd2_rn(pw, vp.v[h]));
      y.v[h] = make_float2(d.v[h].x > 0.f ? yv.x : 0.f, d.v[h].y > 0.f ? yv.y : 0.f);
    }
    stq(s.b + e, y);
  }
}

// The second post-sweep: x into a, or into global memory (gx with strides)
// on the first level.
__device__ __forceinline__ void phase_x(const Slab& s, float* gx, int grow, int gplane, bool zp) {
  const int pitch = 4 * s.gpr, ps = pitch * s.nr, n = s.np * s.nr * s.gpr;
  Walk3 k(threadIdx.x, s.gpr, s.nr, s.mg, s.mr);
  for (int t = threadIdx.x; t < n; t += kCT, k.next()) {
    const int e = k.lp * ps + k.q * pitch + 4 * k.g;
    const Q4 y = ldq(s.b + e), w = invq(ldq(s.d + k.lp * s.dplane + k.q * s.drow + 4 * k.g)),
             r = ldq(s.r + k.lp * s.rplane + k.q * s.rrow + 4 * k.g);
    const Q4 S = nb_group(s, s.b, s.blo, s.bhi, k.lp, k.q, k.g, zp, y);
    Q4 x;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float2 rn = __ffma2_rn(dup(s.c), S.v[h], r.v[h]);
      x.v[h] = __ffma2_rn(__fmul2_rn(dup(kW1), w.v[h]), rn, __fmul2_rn(dup(k1W1), y.v[h]));
    }
    if (gx) stq(gx + k.lp * (long long)gplane + k.q * grow + 4 * k.g, x);
    else stq(s.a + e, x);
  }
}

// The coarsest level: MG_NU_COARSE sweeps of weight MG_OMEGA_COARSE; the
// result ends in a.  At most MG_MIN_SITES sites are at most one group a
// thread, whose right-hand side and diagonal stay in registers; a hierarchy
// that ran out of levels (a chain of millions of sites) has more.
static_assert(MG_MIN_SITES <= kCT, "a thread holds at most one group of the coarsest level");
__device__ __noinline__ void coarsest_large(const Slab& s, bool zp) {
  const int pitch = 4 * s.gpr, ps = pitch * s.nr, n = s.np * s.nr * s.gpr;
  for (int it = 0; it < MG_NU_COARSE; ++it) {
    float* dst = ((MG_NU_COARSE - 1 - it) & 1) ? s.b : s.a;
    const float* src = dst == s.a ? s.b : s.a;
    Walk3 k(threadIdx.x, s.gpr, s.nr, s.mg, s.mr);
    for (int t = threadIdx.x; t < n; t += kCT, k.next()) {
      const int e = k.lp * ps + k.q * pitch + 4 * k.g;
      const Q4 d = ldq(s.d + k.lp * s.dplane + k.q * s.drow + 4 * k.g), w = invq(d),
               r = ldq(s.r + k.lp * s.rplane + k.q * s.rrow + 4 * k.g);
      Q4 o, S = zeroq(), x = zeroq();
      if (it > 0) {
        x = ldq(src + e);
        S = nb_group(s, src, nullptr, nullptr, k.lp, k.q, k.g, zp, x);
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float2 res = __ffma2_rn(make_float2(-d.v[h].x, -d.v[h].y), x.v[h], __ffma2_rn(dup(s.c), S.v[h], r.v[h]));
        o.v[h] = __ffma2_rn(__fmul2_rn(dup(kWC), w.v[h]), res, x.v[h]);
      }
      stq(dst + e, o);
    }
    __syncthreads();
  }
}
__device__ __forceinline__ void coarsest(const Slab& s, bool zp) {
  const int pitch = 4 * s.gpr, ps = pitch * s.nr, n = s.np * s.nr * s.gpr;
  if (n > kCT) {
    coarsest_large(s, zp);
    return;
  }
  const bool live = (int)threadIdx.x < n;
  Walk3 k(live ? threadIdx.x : 0, s.gpr, s.nr, s.mg, s.mr);
  const int e = k.lp * ps + k.q * pitch + 4 * k.g;
  Q4 d = zeroq(), r = zeroq(), x;
  if (live) {
    d = ldq(s.d + k.lp * s.dplane + k.q * s.drow + 4 * k.g);
    r = ldq(s.r + k.lp * s.rplane + k.q * s.rrow + 4 * k.g);
  }
  Q4 w = invq(d);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    w.v[h] = __fmul2_rn(dup(kWC), w.v[h]);
    x.v[h] = __fmul2_rn(w.v[h], r.v[h]);
  }
  for (int it = 0;; ++it) {
    float* dst = ((MG_NU_COARSE - 1 - it) & 1) ? s.b : s.a;
    if (live) stq(dst + e, x);
    __syncthreads();
    if (it == MG_NU_COARSE - 1) break;
    if (live) {
      const Q4 S = nb_group(s, dst, nullptr, nullptr, k.lp, k.q, k.g, zp, x);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float2 rn = __ffma2_rn(dup(s.c), S.v[h], r.v[h]);
        const float2 res = __ffma2_rn(make_float2(-d.v[h].x, -d.v[h].y), x.v[h], rn);
        x.v[h] = __ffma2_rn(w.v[h], res, x.v[h]);
      }
    }
  }
}

__device__ __forceinline__ void cp16a(float* sdst, const float* gsrc) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gsrc) : "memory");
}

__global__ void __launch_bounds__(kCT, 1) k_mg_cluster(Ctx c, int which) {
  extern __shared__ __align__(16) float csm[];
  __shared__ MGClusterLevel T[kCLev];
  cg::cluster_group cl = cg::this_cluster();
  const int cs = (int)cl.num_blocks(), rank = (int)cl.block_rank(), rep = blockIdx.x / cs;
  const MGCluster& R = c.mgc[rep];
  const int nl = R.nl, ndist = R.ndist;   // levels held, the first ndist of them distributed
  const bool zp = R.zp != 0;
  {
    const int* src = reinterpret_cast<const int*>(R.lev);
    int* dst = reinterpret_cast<int*>(T);
    for (int i = threadIdx.x; i < nl * (int)(sizeof(MGClusterLevel) / 4); i += kCT) dst[i] = src[i];
  }
  const float c0 = c.reps[rep].cpl32[which];
  __syncthreads();
  // this block's slab of level i (single-block levels: whole, block 0 only)
  auto slab = [&](int i) {
    const MGClusterLevel& L = T[i];
    Slab s;
    s.nx = L.nx;
    s.nr = L.nr;
    s.gpr = L.gpr;
    s.no = L.no;
    const bool dist = i < ndist;
    s.o0 = dist ? L.p0[rank] : 0;
    s.np = dist ? L.p0[rank + 1] - s.o0 : (rank == 0 ? L.no : 0);
    s.a = csm + L.oa;
    s.b = csm + L.ob;
    const int pitch = 4 * L.gpr, ps = pitch * L.nr;
    s.r = L.orr >= 0 ? csm + L.orr : L.grhs + (long long)s.o0 * L.gplane;
    s.rrow = L.orr >= 0 ? pitch : L.grow;
    s.rplane = L.orr >= 0 ? ps : L.gplane;
    s.d = L.od >= 0 ? csm + L.od : L.gd + (long long)s.o0 * L.gplane;
    s.drow = L.od >= 0 ? pitch : L.grow;
    s.dplane = L.od >= 0 ? ps : L.gplane;
    s.c = c0 * L.cscale;
    s.mg = L.mg;
    s.mr = L.mr;
    s.mc = i + 1 < nl ? T[i + 1].mr : 0u;
    s.alo = s.ahi = s.blo = s.bhi = nullptr;
    if (dist && s.np > 0) {
      if (s.o0 > 0) {
        int k = rank - 1;
        while (L.p0[k + 1] == L.p0[k]) --k;   // blocks without a plane (levels of fewer planes than blocks)
        const int off = (L.p0[k + 1] - L.p0[k] - 1) * ps;
        s.alo = cl.map_shared_rank(s.a, k) + off;
        s.blo = cl.map_shared_rank(s.b, k) + off;
      }
      if (s.o0 + s.np < L.no) {
        int k = rank + 1;
        while (L.p0[k + 1] == L.p0[k]) ++k;
        s.ahi = cl.map_shared_rank(s.a, k);
        s.bhi = cl.map_shared_rank(s.b, k);
      }
    }
    return s;
  };
  // the diagonals that live in shared memory move in before the predecessor
  // has finished (they were written at the start of the solve), and the
  // right-hand sides' padding becomes zero
  for (int i = 0; i < nl; ++i) {
    const MGClusterLevel& L = T[i];
    const Slab s = slab(i);
    const int pitch = 4 * L.gpr, n = s.np * L.nr * L.gpr;
    if (L.orr >= 0 && L.nx < pitch)
      for (int t = threadIdx.x; t < s.np * L.nr; t += kCT)
        for (int x = L.nx; x < pitch; ++x) csm[L.orr + t * pitch + x] = 0.f;
    if (L.od < 0) continue;
    Walk3 k(threadIdx.x, L.gpr, L.nr, L.mg, L.mr);
    for (int t = threadIdx.x; t < n; t += kCT, k.next())
      cp16a(csm + L.od + (k.lp * L.nr + k.q) * pitch + 4 * k.g,
            L.gd + (long long)(s.o0 + k.lp) * L.gplane + k.q * L.grow + 4 * k.g);
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  HCA_VC_ENTRY(c);
  if (c.skip_idle && !c.solve[rep].active) return;   // the same for the whole cluster
  // down: the distributed levels in every block, then the single-block levels in block 0
  for (int i = 0; i < nl - 1; ++i) {
    const bool dist = i < ndist;
    if (!dist && rank != 0) break;
    const Slab s = slab(i);
    const MGClusterLevel &L = T[i], &C = T[i + 1];
    if (i == 0) phase_u(s, L.grhs + (long long)s.o0 * L.gplane, L.grow, L.gplane, L.orr >= 0 ? csm + L.orr : nullptr);
    else phase_u(s, s.r, s.rrow, s.rplane, nullptr);
    if (dist) cl.sync();
    else __syncthreads();
    phase_v(s, zp);
    if (dist) cl.sync();
    else __syncthreads();
    float* rc = csm + C.orr;
    if (i + 1 == ndist) rc = cl.map_shared_rank(rc, 0) + (s.o0 >> 1) * (4 * C.gpr * C.nr);
    phase_r(s, rc, 4 * C.gpr, C.nr, C.nx, zp);
    if (i + 1 == ndist) cl.sync();
    else __syncthreads();
  }
  if (rank == 0) {
    const Slab s = slab(nl - 1);
    const MGClusterLevel& L = T[nl - 1];
    const int pitch = 4 * L.gpr, n = L.no * L.nr * L.gpr;
    if (nl == 1) {   // the first level is the coarsest
      Walk3 k(threadIdx.x, L.gpr, L.nr, L.mg, L.mr);
      for (int t = threadIdx.x; t < n; t += kCT, k.next())
        stq(csm + L.orr + (k.lp * L.nr + k.q) * pitch + 4 * k.g,
            ldq(L.grhs + (long long)k.lp * L.gplane + k.q * L.grow + 4 * k.g));
    }
    coarsest(s, zp);
    if (nl == 1) {
      Walk3 k(threadIdx.x, L.gpr, L.nr, L.mg, L.mr);
      for (int t = threadIdx.x; t < n; t += kCT, k.next())
        stq(L.gx + (long long)k.lp * L.gplane + k.q * L.grow + 4 * k.g, ldq(s.a + (k.lp * L.nr + k.q) * pitch + 4 * k.g));
    }
  }
  // up: the single-block levels in block 0, then the distributed levels
  for (int i = nl - 2; i >= 0; --i) {
    const bool dist = i < ndist;
    if (!dist && rank != 0) continue;
    const Slab s = slab(i);
    const MGClusterLevel &L = T[i], &C = T[i + 1];
    const int cps = 4 * C.gpr * C.nr;
    const float *ca = csm + C.oa, *clo = nullptr, *chi = nullptr;
    int lo = 0, hi = C.no;
    if (i + 1 == ndist) {
      // the planes of block 0's level under this slab and next to it, into
      // this block's own (unused) copy of that level
      cl.sync();
      const int f = max(0, (s.o0 >> 1) - 1), t1 = min(C.no, ((s.o0 + s.np + 1) >> 1) + 1);
      if (rank != 0 && s.np > 0) {
        const float4* src = reinterpret_cast<const float4*>(cl.map_shared_rank(csm + C.oa, 0));
        float4* dst = reinterpret_cast<float4*>(csm + C.oa);
        for (int t = f * (cps >> 2) + threadIdx.x; t < t1 * (cps >> 2); t += kCT) dst[t] = src[t];
      }
      __syncthreads();
    } else if (dist) {
      const Slab q = slab(i + 1);
      ca = q.a;
      clo = q.alo;
      chi = q.ahi;
      lo = q.o0;
      hi = q.o0 + q.np;
    }
    phase_y(s, ca, clo, chi, lo, hi, 4 * C.gpr, C.nr, C.no, C.nx, zp);
    if (dist) cl.sync();
    else __syncthreads();
    phase_x(s, i == 0 ? L.gx + (long long)s.o0 * L.gplane : nullptr, L.grow, L.gplane, zp);
    // x before the finer level reads it; before a block's exit, its neighbours' reads
    if (dist) cl.sync();
    else __syncthreads();
  }
}

}  // namespace

// First level a cluster of cs blocks can hold for the hierarchy lv[1 ..
// nl - 1] (at least `from`) within `smem` bytes a block, and its layout in
// *R; 0 when not even the single-block levels fit.
int cluster_plan(const MGLevel* lv, int nl, int from, int cs, long long smem, MGCluster* R) {
  int single = nl - 1;
  while (single > 1 && lv[single - 1].n <= MG_SMALL_SITES) --single;
  for (int lc = std::min(from, single); lc < nl; ++lc) {
    if (nl - lc > kCLev) continue;
    MGCluster P{};
    P.lc = lc;
    P.nl = nl - lc;
    P.ndist = std::max(0, single - lc);
    P.zp = lv[lc].nz >= 8 || lv[lc].nz >= lv[lc].ny;
    long long o = 0;
    // pass 1: the first distributed level's right-hand side and diagonal stay
    // in global memory; pass 2: the single-block levels' diagonals too
    for (int pass = 0; pass < 3; ++pass) {
      o = 0;
      for (int i = 0; i < P.nl; ++i) {
        const MGLevel& L = lv[lc + i];
        MGClusterLevel& Q = P.lev[i];
        Q.nx = L.nx;
        Q.nr = P.zp ? L.ny : L.nz;
        Q.no = P.zp ? L.nz : L.ny;
        Q.gpr = (L.nx + 3) / 4;
        Q.cscale = L.cscale32;
        Q.grhs = (const float*)L.rhs;
        Q.gd = (const float*)L.d;
        Q.gx = (float*)L.x;
        const int srow = L.pitch, splane = L.pitch * L.ny;
        Q.grow = P.zp ? srow : splane;
        Q.gplane = P.zp ? splane : srow;
        long long planes = Q.no;
        if (i < P.ndist) {
          // whole planes of the first single-block level per block
          const int shift = P.ndist - i;
          const MGLevel& S = lv[lc + P.ndist];
          const int ns = P.zp ? S.nz : S.ny;
          planes = 0;
          for (int k = 0; k <= cs; ++k) {
            const long long p = ((long long)ns * k / cs) << shift;
            Q.p0[k] = (int)std::min<long long>(p, Q.no);
            if (k) planes = std::max<long long>(planes, Q.p0[k] - Q.p0[k - 1]);
          }
        }
        const long long n = planes * Q.nr * Q.gpr * 4;
        Q.oa = (int)o;
        Q.ob = (int)(o + n);
        o += 2 * n;
        const bool out = i == 0 && P.ndist > 0 && pass > 0;
        Q.orr = out ? -1 : (int)o;
        if (!out) o += n;
        Q.od = out || (pass == 2 && i >= P.ndist) ? -1 : (int)o;
        if (Q.od >= 0) o += n;
        Q.mg = (1u << 20) / (unsigned)Q.gpr + 1u;
        Q.mr = (1u << 20) / (unsigned)Q.nr + 1u;
      }
      if (o * 4 <= smem) break;
    }
    if (o * 4 > smem) continue;
    P.smem = (int)(o * 4);
    *R = P;
    return lc;
  }
  return 0;
}

static bool cluster_launch_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* at, const MGHost& H, int reps,
                                  cudaStream_t s, bool pdl) {
  cfg = {};
  cfg.gridDim = dim3(reps * H.cl_size);
  cfg.blockDim = dim3(kCT);
  cfg.dynamicSmemBytes = (size_t)H.cl_smem;
  cfg.stream = s;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = H.cl_size;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 2 : 1;
  return true;
}

// Whether clusters of H.cl_size blocks with H.cl_smem bytes can run.
bool cluster_init(const MGHost& H) {
  const void* fn = (const void*)k_mg_cluster;
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024 - 4096) != cudaSuccess ||
      cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
    (void)cudaGetLastError();
    return false;
  }
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[2];
  cluster_launch_config(cfg, at, H, 1, nullptr, false);
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();
    return false;
  }
  return n >= 1;
}

void launch_mg_cluster(const Ctx& c, int which, const MGHost& H) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[2];
  cluster_launch_config(cfg, at, H, c.n_reps, c.stream, c.pdl != 0);
  (void)cudaLaunchKernelEx(&cfg, k_mg_cluster, c, which);
}

}  // namespace hca
