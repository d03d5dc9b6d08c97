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
// Bound: the latency of ~45 dependent phases on one or two groups a thread
// (block barriers ~250 cycles, cluster barriers 1200 and more) and of code that
// runs once.  A thread keeps its groups' places and values in registers
// through a level, slabs are worked out once, and the coarsest sweeps run on
// the warps that have groups.  The levels 32^3, 16^3 and 8^3: 14 us (19 us
// with each phase on its own; 37 us with a launch per sweep of 32^3 and a
// single-block kernel for the others); a step at 64^3 2.46 -> 2.30 ms.
#include <cooperative_groups.h>

#include <algorithm>
#include <vector>

#include "hca_internal.cuh"

namespace cg = cooperative_groups;

namespace hca {

namespace {

constexpr int kCT = 512;              // threads per block
constexpr int kCLev = 12;             // most levels a cluster holds
constexpr int kPush = 256;            // most planes of a level whose planes are pushed
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
  unsigned calo, cahi;          // alo, ahi as cluster shared addresses
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

// ---- levels of at most kGT groups a thread (all but odd shapes) ----
// A thread keeps its groups through the phases of a level: places, neighbour
// offsets and its own values stay in registers, which is what the phases'
// instructions mostly went into.  Same operations, same order of sums.
constexpr int kGT = 2;

struct Place {
  bool live;
  int e, lp, q, g;                       // element in a and b
  // shared addresses of the group and its neighbour rows and planes in a (b is
  // at the same distance everywhere; planes may be a neighbouring block's),
  // and whether they are inside: predicated loads, no branches
  unsigned c, rm, rp, pm, pp;
  int gl, gr, irm, irp, ipm, ipp;
};
__device__ __forceinline__ unsigned sm_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ Q4 lds_if(unsigned a, int ok) {
  Q4 q;
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.s32 p, %5, 0;\nmov.f32 %0, 0f00000000;\nmov.f32 %1, 0f00000000;\n"
      "mov.f32 %2, 0f00000000;\nmov.f32 %3, 0f00000000;\n@p ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];\n}"
      : "=&f"(q.v[0].x), "=&f"(q.v[0].y), "=&f"(q.v[1].x), "=&f"(q.v[1].y)
      : "r"(a), "r"(ok)
      : "memory");
  return q;
}
__device__ __forceinline__ Q4 ldc_if(unsigned a, int ok) {   // any block's shared memory
  Q4 q;
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.s32 p, %5, 0;\nmov.f32 %0, 0f00000000;\nmov.f32 %1, 0f00000000;\n"
      "mov.f32 %2, 0f00000000;\nmov.f32 %3, 0f00000000;\n@p ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];\n}"
      : "=&f"(q.v[0].x), "=&f"(q.v[0].y), "=&f"(q.v[1].x), "=&f"(q.v[1].y)
      : "r"(a), "r"(ok)
      : "memory");
  return q;
}
__device__ __forceinline__ float lds1_if(unsigned a, int ok) {
  float v;
  asm volatile("{\n.reg .pred p;\nsetp.ne.s32 p, %2, 0;\nmov.f32 %0, 0f00000000;\n@p ld.shared.f32 %0, [%1];\n}"
               : "=&f"(v)
               : "r"(a), "r"(ok)
               : "memory");
  return v;
}
template <int N>
__device__ __forceinline__ void places(const Slab& s, Place (&P)[N]) {
  const int pitch = 4 * s.gpr, ps = pitch * s.nr, n = s.np * s.nr * s.gpr;
  const unsigned a = sm_u32(s.a);
  Walk3 w(threadIdx.x, s.gpr, s.nr, s.mg, s.mr);
#pragma unroll
  for (int j = 0; j < N; ++j, w.next()) {
    Place& p = P[j];
    p.live = (int)threadIdx.x + j * kCT < n;
    p.lp = w.lp;
    p.q = w.q;
    p.g = w.g;
    p.e = p.live ? w.lp * ps + w.q * pitch + 4 * w.g : 0;
    const unsigned ei = 4u * (unsigned)(w.q * pitch + 4 * w.g);
    p.c = a + 4u * (unsigned)p.e;
    p.rm = p.c - 4u * (unsigned)pitch;
    p.rp = p.c + 4u * (unsigned)pitch;
    p.pm = w.lp > 0 ? p.c - 4u * (unsigned)ps : s.calo + ei;
    p.pp = w.lp + 1 < s.np ? p.c + 4u * (unsigned)ps : s.cahi + ei;
    p.gl = p.live && w.g > 0;
    p.gr = p.live && w.g + 1 < s.gpr;
    p.irm = p.live && w.q > 0;
    p.irp = p.live && w.q + 1 < s.nr;
    p.ipm = p.live && (w.lp > 0 || s.alo);
    p.ipp = p.live && (w.lp + 1 < s.np || s.ahi);
  }
}
// S of a group over a (d = 0) or b (d = their distance in bytes), own the group itself.
__device__ __forceinline__ Q4 nb_place(const Place& p, unsigned d, bool zp, const Q4& own) {
  const Q4 rm = lds_if(p.rm + d, p.irm), rp = lds_if(p.rp + d, p.irp);
  const Q4 pm = ldc_if(p.pm + d, p.ipm), pp = ldc_if(p.pp + d, p.ipp);
  const float lft = lds1_if(p.c + d - 4u, p.gl), rgt = lds1_if(p.c + d + 16u, p.gr);
  const float2 x[2] = {make_float2(lft + own.v[0].y, own.v[0].x + own.v[1].x),
                       make_float2(own.v[0].y + own.v[1].y, own.v[1].x + rgt)};
  const Q4 &ym = zp ? rm : pm, &yp = zp ? rp : pp, &zm = zp ? pm : rm, &zq = zp ? pp : rp;
  Q4 S;
#pragma unroll
  for (int h = 0; h < 2; ++h)
    S.v[h] = __fadd2_rn(__fadd2_rn(__fadd2_rn(x[h], __fadd2_rn(ym.v[h], yp.v[h])), zm.v[h]), zq.v[h]);
  return S;
}

// Down a level: both pre-sweeps, the residual's restriction into rc (see
// phase_r) and a = v'.  sync: the level's barrier; rs: see phase_u; scratch:
// kGT kCT row sums.
template <class Sync>
__device__ __forceinline__ void level_down(const Slab& s, const float* gr, int rrow, int rplane, float* rs, float* rc,
                                           int cpitch, int cnr, bool zp, float2* scratch, Sync sync) {
  Place P[kGT];
  places(s, P);
  const unsigned d = sm_u32(s.b) - sm_u32(s.a);
  Q4 r[kGT], dg[kGT], w[kGT], u[kGT], v[kGT];
#pragma unroll
  for (int j = 0; j < kGT; ++j) {
    r[j] = dg[j] = zeroq();
    if (P[j].live) {
      r[j] = ldq(gr + P[j].lp * rplane + P[j].q * rrow + 4 * P[j].g);
      dg[j] = ldq(s.d + P[j].lp * s.dplane + P[j].q * s.drow + 4 * P[j].g);
    }
  }
#pragma unroll
  for (int j = 0; j < kGT; ++j) {
    w[j] = invq(dg[j]);
    u[j] = u_of(r[j], w[j]);
    if (!P[j].live) continue;
    if (rs) stq(rs + P[j].e, r[j]);
    stq(s.a + P[j].e, u[j]);
  }
  sync();
  const float2 w2c = dup(kW2 * s.c);
#pragma unroll
  for (int j = 0; j < kGT; ++j) {
    if (!P[j].live) continue;
    const Q4 S = nb_place(P[j], 0, zp, u[j]);
#pragma unroll
    for (int h = 0; h < 2; ++h)
      v[j].v[h] = __ffma2_rn(__fmul2_rn(w2c, w[j].v[h]), S.v[h], __fmul2_rn(dup(kK), u[j].v[h]));
    stq(s.b + P[j].e, v[j]);
  }
  sync();
#pragma unroll
  for (int j = 0; j < kGT; ++j) {
    if (!P[j].live) continue;
    const Q4 S = nb_place(P[j], d, zp, v[j]);
    Q4 res, o;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float2 rn = __ffma2_rn(dup(s.c), S.v[h], r[j].v[h]);
      res.v[h] = __ffma2_rn(make_float2(-dg[j].v[h].x, -dg[j].v[h].y), v[j].v[h], rn);
      o.v[h] = __ffma2_rn(__fmul2_rn(dup(kW2), w[j].v[h]), res.v[h], v[j].v[h]);
    }
    const int x0 = 4 * P[j].g;
    if (x0 + 1 >= s.nx) res.v[0].y = 0.f;
    if (x0 + 2 >= s.nx) res.v[1].x = 0.f;
    if (x0 + 3 >= s.nx) res.v[1].y = 0.f;
    scratch[threadIdx.x + j * kCT] = make_float2(res.v[0].x + res.v[0].y, res.v[1].x + res.v[1].y);
    stq(s.a + P[j].e, o);
  }
  __syncthreads();
  // (dz 0: dy 0 + dy 1) + (dz 1: dy 0 + dy 1), whichever way the planes lie
  const int ncp = (s.np + 1) >> 1, n = ncp * cnr * s.gpr, gps = s.nr * s.gpr;
  Walk3 k(threadIdx.x, s.gpr, cnr, s.mg, s.mc);
  for (int t = threadIdx.x; t < n; t += kCT, k.next()) {
    const int f = 2 * k.lp * gps + 2 * k.q * s.gpr + k.g;
    const bool q1 = 2 * k.q + 1 < s.nr, p1 = 2 * k.lp + 1 < s.np;
    const float2 zero = make_float2(0.f, 0.f);
    const float2 a00 = scratch[f], a01 = q1 ? scratch[f + s.gpr] : zero;
    const float2 a10 = p1 ? scratch[f + gps] : zero, a11 = p1 && q1 ? scratch[f + gps + s.gpr] : zero;
    const float2 acc = zp ? __fadd2_rn(__fadd2_rn(a00, a01), __fadd2_rn(a10, a11))
                          : __fadd2_rn(__fadd2_rn(a00, a10), __fadd2_rn(a01, a11));
    // (a pair's second cell may be padding: its sum is zero)
    *reinterpret_cast<float2*>(rc + k.lp * cpitch * cnr + k.q * cpitch + 2 * k.g) = acc;
  }
}

// Up a level: both post-sweeps (see phase_y, phase_x); the coarse correction's
// padding is zero.  push: block 0's level below the distributed ones; each
// plane of x also goes to the blocks (first, last) whose slabs lie over or next
// to it, so that they need not fetch it after the barrier.
template <class Sync>
__device__ __forceinline__ void level_up(const Slab& s, const float* ca, const float* clo, const float* chi, int lo, int hi,
                                         int cpitch, int cnr, int cno, int cnx, float* gx, int grow, int gplane, bool zp,
                                         const uchar2* push, Sync sync) {
  Place P[kGT];
  places(s, P);
  const int cps = cpitch * cnr;
  const unsigned d = sm_u32(s.b) - sm_u32(s.a);
  const float2 w2c = dup(kW2 * s.c);
  Q4 r[kGT], w[kGT], y[kGT];
#pragma unroll
  for (int j = 0; j < kGT; ++j) {
    const Place& p = P[j];
    if (!p.live) continue;
    const int X = 2 * p.g, o = s.o0 + p.lp, O = o >> 1, Q = p.q >> 1;
    const int Oo = (o & 1) ? O + 1 : O - 1, Qo = (p.q & 1) ? Q + 1 : Q - 1;
    const int ce = Q * cpitch + X;
    const float* c0 = (O < lo ? clo : O >= hi ? chi : ca + (O - lo) * cps) + ce;
    const float* cp = (Oo < lo ? clo : Oo >= hi ? chi : ca + (Oo - lo) * cps) + ce;
    auto pair = [](const float* f) { return *reinterpret_cast<const float2*>(f); };
    const float2 zero = make_float2(0.f, 0.f);
    float2 pl = zero, rw = zero;
    float xl = 0.f, xr = 0.f;
    const float2 cur = pair(c0);
    if (Oo >= 0 && Oo < cno) pl = pair(cp);
    if (Qo >= 0 && Qo < cnr) rw = pair(c0 + (Qo - Q) * cpitch);
    if (X > 0) xl = c0[-1];
    if (X + 2 < cnx) xr = c0[2];
    const Q4 vp = ldq(s.a + p.e), dg = ldq(s.d + p.lp * s.dplane + p.q * s.drow + 4 * p.g);
    r[j] = ldq(s.r + p.lp * s.rplane + p.q * s.rrow + 4 * p.g);
    w[j] = invq(dg);
    const bool pin = (o & 1) || o + 1 < s.no, rin = (p.q & 1) || p.q + 1 < s.nr;
    const float2 fp = pin ? __fadd2_rn(pl, cur) : pl, fr = rin ? __fadd2_rn(rw, cur) : rw;
    const float2 tt = zp ? __fadd2_rn(fr, fp) : __fadd2_rn(fp, fr);
    const float both = cur.x + cur.y;
    float2 xs[2] = {make_float2(xl + cur.x, both), make_float2(both, cur.y + xr)};
    const int x0 = 4 * p.g;
    if (x0 + 1 == s.nx) xs[0].x = xl;
    if (x0 + 2 == s.nx) xs[0].y = cur.x;
    if (x0 + 3 == s.nx) xs[1].x = cur.x;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float2 S = __fadd2_rn(xs[h], dup(h ? tt.y : tt.x));
      const float2 pw = __fmul2_rn(dup(k1W2), dup(h ? cur.y : cur.x));
      const float2 yv = __ffma2_rn(__fmul2_rn(w2c, w[j].v[h]), S, __fadd2_rn(pw, vp.v[h]));
      y[j].v[h] = make_float2(dg.v[h].x > 0.f ? yv.x : 0.f, dg.v[h].y > 0.f ? yv.y : 0.f);
    }
    stq(s.b + p.e, y[j]);
  }
  sync();
#pragma unroll
  for (int j = 0; j < kGT; ++j) {
    const Place& p = P[j];
    if (!p.live) continue;
    const Q4 S = nb_place(p, d, zp, y[j]);
    Q4 x;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float2 rn = __ffma2_rn(dup(s.c), S.v[h], r[j].v[h]);
      x.v[h] = __ffma2_rn(__fmul2_rn(dup(kW1), w[j].v[h]), rn, __fmul2_rn(dup(k1W1), y[j].v[h]));
    }
    if (gx) stq(gx + p.lp * (long long)gplane + p.q * grow + 4 * p.g, x);
    else stq(s.a + p.e, x);
    if (push) {
      const uchar2 to = push[p.lp];
      for (int k = max(1, (int)to.x); k <= (int)to.y; ++k)
        asm volatile(
            "{\n.reg .u32 a;\nmapa.shared::cluster.u32 a, %0, %1;\nst.shared::cluster.v4.f32 [a], {%2, %3, %4, %5};\n}" ::"r"(p.c),
            "r"(k), "f"(x.v[0].x), "f"(x.v[0].y), "f"(x.v[1].x), "f"(x.v[1].y)
            : "memory");
    }
  }
}

// The coarsest level: MG_NU_COARSE sweeps of weight MG_OMEGA_COARSE; the
// result ends in a.  At most MG_MIN_SITES sites (the hierarchies end there:
// MG_MAXLEV) are at most one group a thread, whose right-hand side and diagonal
// stay in registers.
static_assert(MG_MIN_SITES <= kCT, "a thread holds at most one group of the coarsest level");
// zero: 16 bytes of zeros in shared memory.
__device__ __forceinline__ void coarsest(const Slab& shared_s, bool zp, const float4* zero) {
  const int n = shared_s.np * shared_s.nr * shared_s.gpr;
  const Slab s = shared_s;
  const int nt = (n + 31) & ~31;   // the warps with groups
  if ((int)threadIdx.x < nt) {
    Place P[1];
    places(s, P);
    const Place& p = P[0];
    const unsigned d = sm_u32(s.b) - sm_u32(s.a), z = sm_u32(zero);
    // addresses of the neighbours in a and in b; zeros where there is none
    unsigned at[2][6];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const unsigned o = k ? d : 0u;
      at[k][0] = p.irm ? p.rm + o : z;
      at[k][1] = p.irp ? p.rp + o : z;
      at[k][2] = p.ipm ? p.pm + o : z;
      at[k][3] = p.ipp ? p.pp + o : z;
      at[k][4] = p.gl ? p.c + o - 4u : z;
      at[k][5] = p.gr ? p.c + o + 16u : z;
    }
    Q4 dg = zeroq(), r = zeroq(), x;
    if (p.live) {
      dg = ldq(s.d + p.lp * s.dplane + p.q * s.drow + 4 * p.g);
      r = ldq(s.r + p.lp * s.rplane + p.q * s.rrow + 4 * p.g);
    }
    Q4 w = invq(dg);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      w.v[h] = __fmul2_rn(dup(kWC), w.v[h]);
      x.v[h] = __fmul2_rn(w.v[h], r.v[h]);
      dg.v[h] = make_float2(-dg.v[h].x, -dg.v[h].y);
    }
    auto lds4 = [](unsigned a) {
      Q4 q;
      asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                   : "=f"(q.v[0].x), "=f"(q.v[0].y), "=f"(q.v[1].x), "=f"(q.v[1].y)
                   : "r"(a)
                   : "memory");
      return q;
    };
    auto lds1 = [](unsigned a) {
      float f;
      asm volatile("ld.shared.f32 %0, [%1];" : "=f"(f) : "r"(a) : "memory");
      return f;
    };
    auto put = [&](int k) {
      if (p.live)
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(p.c + (k ? d : 0u)), "f"(x.v[0].x), "f"(x.v[0].y),
                     "f"(x.v[1].x), "f"(x.v[1].y)
                     : "memory");
    };
    auto sweep = [&](int k) {   // x stored in buffer k by every thread
      asm volatile("bar.sync 1, %0;" ::"r"(nt) : "memory");
      const Q4 rm = lds4(at[k][0]), rp = lds4(at[k][1]), pm = lds4(at[k][2]), pp = lds4(at[k][3]);
      const float lft = lds1(at[k][4]), rgt = lds1(at[k][5]);
      const float2 xs[2] = {make_float2(lft + x.v[0].y, x.v[0].x + x.v[1].x),
                            make_float2(x.v[0].y + x.v[1].y, x.v[1].x + rgt)};
      const Q4 &ym = zp ? rm : pm, &yp = zp ? rp : pp, &zm = zp ? pm : rm, &zq = zp ? pp : rp;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float2 S = __fadd2_rn(__fadd2_rn(__fadd2_rn(xs[h], __fadd2_rn(ym.v[h], yp.v[h])), zm.v[h]), zq.v[h]);
        const float2 rn = __ffma2_rn(dup(s.c), S, r.v[h]);
        const float2 res = __ffma2_rn(dg.v[h], x.v[h], rn);
        x.v[h] = __ffma2_rn(w.v[h], res, x.v[h]);
      }
    };
    // the result ends in a
    static_assert(MG_NU_COARSE % 2 == 0, "sweeps in pairs");
    put(1);
#pragma unroll 1
    for (int it = 0; it < MG_NU_COARSE / 2 - 1; ++it) {
      sweep(1);
      put(0);
      sweep(0);
      put(1);
    }
    sweep(1);
    put(0);
  }
  __syncthreads();
}

__device__ __forceinline__ void cp16a(float* sdst, const float* gsrc) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gsrc) : "memory");
}

__global__ void __launch_bounds__(kCT, 1) k_mg_cluster(Ctx c, int which) {
  extern __shared__ __align__(16) float csm[];
  __shared__ MGClusterLevel T[kCLev];
  __shared__ float2 scratch[kGT * kCT];
  __shared__ Slab SL[kCLev];   // this block's slabs
  __shared__ float4 s_zero;
  __shared__ uchar2 s_push[kPush];   // per plane of the first single-block level: the blocks that need it
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
  auto make_slab = [&](int i) {
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
    s.calo = s.cahi = 0u;
    auto mapa = [](const float* p, int k) {
      unsigned r;
      asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(sm_u32(p)), "r"(k));
      return r;
    };
    if (dist && s.np > 0) {
      if (s.o0 > 0) {
        int k = rank - 1;
        while (L.p0[k + 1] == L.p0[k]) --k;   // blocks without a plane (levels of fewer planes than blocks)
        const int off = (L.p0[k + 1] - L.p0[k] - 1) * ps;
        s.alo = cl.map_shared_rank(s.a, k) + off;
        s.calo = mapa(s.a, k) + 4u * (unsigned)off;
        s.blo = cl.map_shared_rank(s.b, k) + off;
      }
      if (s.o0 + s.np < L.no) {
        int k = rank + 1;
        while (L.p0[k + 1] == L.p0[k]) ++k;
        s.ahi = cl.map_shared_rank(s.a, k);
        s.cahi = mapa(s.a, k);
        s.bhi = cl.map_shared_rank(s.b, k);
      }
    }
    return s;
  };
  const bool pushes = ndist > 0 && ndist < nl - 1 && T[ndist].no <= kPush && T[ndist].few;
  if (threadIdx.x == 511) s_zero = make_float4(0.f, 0.f, 0.f, 0.f);
  if ((int)threadIdx.x < nl) SL[threadIdx.x] = make_slab((int)threadIdx.x);
  else if (pushes && threadIdx.x >= 32 && (int)threadIdx.x - 32 < T[ndist].no) {
    const MGClusterLevel& L = T[ndist - 1];
    const int O = threadIdx.x - 32, f0 = max(0, 2 * O - 1), f1 = min(L.no - 1, 2 * O + 2);
    int k0 = 0, k1 = cs - 1;
    while (L.p0[k0 + 1] <= f0) ++k0;
    while (L.p0[k1] > f1) --k1;
    s_push[O] = make_uchar2((unsigned char)k0, (unsigned char)k1);
  }
  __syncthreads();
  auto slab = [&](int i) { return SL[i]; };
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
    float* rc = csm + C.orr;
    if (i + 1 == ndist) rc = cl.map_shared_rank(rc, 0) + (s.o0 >> 1) * (4 * C.gpr * C.nr);
    auto sync = [&] {
      if (dist) cl.sync();
      else __syncthreads();
    };
    const float* r0 = i == 0 ? L.grhs + (long long)s.o0 * L.gplane : s.r;
    const int rrow = i == 0 ? L.grow : s.rrow, rplane = i == 0 ? L.gplane : s.rplane;
    float* rs = i == 0 && L.orr >= 0 ? csm + L.orr : nullptr;
    if (L.few) {   // (the same in every block)
      level_down(s, r0, rrow, rplane, rs, rc, 4 * C.gpr, C.nr, zp, scratch, sync);
    } else {
      phase_u(s, r0, rrow, rplane, rs);
      sync();
      phase_v(s, zp);
      sync();
      phase_r(s, rc, 4 * C.gpr, C.nr, C.nx, zp);
    }
    if (i + 1 == ndist) cl.sync();
    else __syncthreads();
  }
  if (rank == 0) {
    const Slab& s = SL[nl - 1];
    const MGClusterLevel& L = T[nl - 1];
    const int pitch = 4 * L.gpr, n = L.no * L.nr * L.gpr;
    if (nl == 1) {   // the first level is the coarsest
      Walk3 k(threadIdx.x, L.gpr, L.nr, L.mg, L.mr);
      for (int t = threadIdx.x; t < n; t += kCT, k.next())
        stq(csm + L.orr + (k.lp * L.nr + k.q) * pitch + 4 * k.g,
            ldq(L.grhs + (long long)k.lp * L.gplane + k.q * L.grow + 4 * k.g));
    }
    coarsest(s, zp, &s_zero);
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
      // the planes of block 0's level under this slab and next to it, in this
      // block's own (otherwise unused) copy of that level: pushed by block 0
      // as it formed them, or fetched here
      cl.sync();
      if (!pushes) {
        const int f = max(0, (s.o0 >> 1) - 1), t1 = min(C.no, ((s.o0 + s.np + 1) >> 1) + 1);
        if (rank != 0 && s.np > 0) {
          const float4* src = reinterpret_cast<const float4*>(cl.map_shared_rank(csm + C.oa, 0));
          float4* dst = reinterpret_cast<float4*>(csm + C.oa);
          for (int t = f * (cps >> 2) + threadIdx.x; t < t1 * (cps >> 2); t += kCT) dst[t] = src[t];
        }
        __syncthreads();
      }
    } else if (dist) {
      const Slab q = slab(i + 1);
      ca = q.a;
      clo = q.alo;
      chi = q.ahi;
      lo = q.o0;
      hi = q.o0 + q.np;
    }
    auto sync = [&] {
      if (dist) cl.sync();
      else __syncthreads();
    };
    float* gx = i == 0 ? L.gx + (long long)s.o0 * L.gplane : nullptr;
    if (L.few) {
      level_up(s, ca, clo, chi, lo, hi, 4 * C.gpr, C.nr, C.no, C.nx, gx, L.grow, L.gplane, zp,
               i == ndist && pushes ? s_push : nullptr, sync);
    } else {
      phase_y(s, ca, clo, chi, lo, hi, 4 * C.gpr, C.nr, C.no, C.nx, zp);
      sync();
      phase_x(s, gx, L.grow, L.gplane, zp);
    }
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
        Q.few = n <= 4 * kGT * kCT;
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
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kClusterSmem) != cudaSuccess ||
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
