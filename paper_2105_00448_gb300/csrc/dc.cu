// The residual sweep of the FP32 defect correction.
//
// The solution is kept as two FP32 words, x = x_hi + x_lo.  Each sweep
// evaluates the residual r = b - A x to about 48 bits (float-float arithmetic)
// from the two-word solution, with the diagonal rebuilt exactly as c n + a from
// the stored FP32 reaction coefficient a (storing d = c n + a itself in FP32
// would round away most digits of the small reaction part: 1/dt + psi ~ 0.03
// next to c n ~ 600 for a drug).  It stops the solve when |r| <= rtol |b| (FP64
// norms) and otherwise starts an FP32 inner CG on the correction, A32 dx =
// fl32(r), dx0 = 0, to the inner tolerance, where A32 uses the FP32 diagonal.
// The first sweep of a solve (FIRST) also builds and stores a, d (and b).
// With the multigrid preconditioner (MG) the kernel stores r for the V-cycle,
// which forms z itself; otherwise it stores the Jacobi z = r / d and sums r.z.
//
// Form.  Marches up z with pass A's tiles and blocks (cg.cu): x_hi and x_lo of
// a plane arrive by tensor copies (four planes in the ring, so every neighbour
// row and plane is read where it landed: holding them in registers spilled), a
// and b (first sweep: the perfusion, V or the linearisation field) in a second
// ring, x neighbours by lane shuffles; the float-float arithmetic runs on two
// sites an instruction.  Traffic per site: a later sweep reads 16 B and writes
// 4, the first reads 9 to 17 B and writes 16.  Bound: instruction issue and the
// float-float chains' latency at 16 warps per multiprocessor (ncu at 256^3:
// 51 % of issue slots, 3 TB/s).  Measured, an average of first and later
// sweeps (FP32, V-cycle form): 137 us at 256^3 against 170 us of the row kernel
// it replaced, 384 against 859 us on 16 uneven replicates (59 M sites).
#include <algorithm>
#include <type_traits>
#include <vector>

#include "march.cuh"
#include "reaction.cuh"

namespace hca {

namespace {

constexpr int kXRing = 4;    // planes k - 1 .. k + 2 of x_hi and x_lo
constexpr int kSRing = 2;   // planes k, k + 1 of the two per-site arrays
constexpr size_t dc_smem(int nt) {
  return (size_t)(kXRing * 4 + kSRing * 4) * nt * 16 + (size_t)kMaxSeg * 3 * (nt / 32) * 8 + 128;
}

// Two sites of a float-float value; the same operations as FF's, on both.
struct FF2 {
  float2 hi, lo;
};
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }   // exact product
__device__ __forceinline__ FF2 ff_add(FF2 a, float2 b) {
  const float2 s = __fadd2_rn(a.hi, b), bb = sub2(s, a.hi);
  const float2 err = __fadd2_rn(sub2(a.hi, sub2(s, bb)), sub2(b, bb));
  return FF2{s, __fadd2_rn(a.lo, err)};
}
__device__ __forceinline__ FF2 ff_add(FF2 a, FF2 b) {
  FF2 r = ff_add(a, b.hi);
  r.lo = __fadd2_rn(r.lo, b.lo);
  return r;
}
__device__ __forceinline__ float2 neg2(float2 a) { return __fmul2_rn(a, make_float2(-1.f, -1.f)); }
__device__ __forceinline__ FF2 ff_two_prod(float2 a, float2 b) {
  const float2 p = __fmul2_rn(a, b);
  return FF2{p, __ffma2_rn(a, b, neg2(p))};
}
__device__ __forceinline__ FF2 ff_mul(FF2 x, float2 b) {
  FF2 p = ff_two_prod(x.hi, b);
  p.lo = __ffma2_rn(x.lo, b, p.lo);
  return p;
}
__device__ __forceinline__ FF2 ff_mul(FF2 x, FF2 y) {
  FF2 p = ff_two_prod(x.hi, y.hi);
  p.lo = __ffma2_rn(x.hi, y.lo, __ffma2_rn(x.lo, y.hi, p.lo));
  return p;
}

// The scale of a running sum of squares: the exponent field of the largest
// magnitude so far (a decayed field's residual, ~1e-22, would underflow when
// squared unscaled).  Terms 2^63 below the largest drop out.
struct RunScale {
  unsigned e = 1u << 23;
  float inv = 0x1p126f;   // 1 / 2^(exponent)
  // takes magnitude m in; returns the factor 2^(old - new exponent)
  __device__ __forceinline__ float take(float m) {
    const unsigned b = __float_as_uint(m) & 0x7f800000u;
    if (b <= e) return 1.f;
    const unsigned d = (b - e) >> 23;
    e = b;
    inv = b < 254u << 23 ? __uint_as_float((254u << 23) - b) : b == 254u << 23 ? __uint_as_float(1u << 22) : 0.f;
    return d < 126u ? __uint_as_float((127u - d) << 23) : 0.f;
  }
  // the factor to the warp's largest scale, which becomes this one's
  __device__ __forceinline__ float join() {
    const unsigned m = __reduce_max_sync(0xffffffffu, e), d = (m - e) >> 23;
    e = m;
    return d < 126u ? __uint_as_float((127u - d) << 23) : 0.f;
  }
  __device__ __forceinline__ double value() const { return __longlong_as_double((long long)((e >> 23) + 896u) << 52); }
};
__device__ __forceinline__ FF scaled(FF s, float f) { return FF{s.hi * f, s.lo * f}; }   // f a power of two

// One thread: the end of a sweep of replicate rep, s3 = |r|^2, |b|^2 (first
// sweep), r.z (Jacobi form).
template <bool FIRST, bool MG>
__device__ void dc_finish(const Ctx& c, int rep, int which, const double* s3) {
  const RepDesc& rr = c.reps[rep];
  RepSolve& s = c.solve[rep];
  DevStats& st = c.stats[rep];
  if (FIRST) {
    s.outer = 0;
    s.zero_b = 0;
    s.dc_apply = 0;
    s.active = 0;
    s.iters = 0;
    s.pend = 0;
    if (c.frozen[rep]) return;
  } else if (!s.dc_apply) {
    return;   // this replicate finished in an earlier sweep
  }
  st.iters[which] += s.iters;
  st.sweeps[which] += 1;
  s.pend = 0;
  // |b|^2 is summed on the first sweep only (b does not change)
  if (FIRST) s.bb_outer = s3[1];
  const double bb = s.bb_outer;
  if (!isfinite(s3[0]) || !isfinite(bb) || !isfinite(s3[2])) {
    c.sync->error = 1;
    st.nonfinite = 1;
    s.active = 0;
    s.dc_apply = 0;
    return;
  }
  const double tol = which == 0 ? rr.rtol_o2 : rr.rtol_drug;
  if (bb == 0.0) {
    s.zero_b = 1;
    s.rel_true = 0.0;
    st.rel[which] = 0.0;
    s.active = 0;
    s.dc_apply = 0;
    return;
  }
  const double rel = sqrt(s3[0] / bb);
  s.rel_true = rel;
  st.rel[which] = rel;
  if (rel <= tol || s.outer >= rr.max_outer) {
    if (rel > tol) st.not_converged |= 1 << which;
    s.active = 0;
    s.dc_apply = 0;
    return;
  }
  // start the inner FP32 solve A dx = fl32(r), rescaled by a
  // power of two so that its values are O(1) per site (the
  // residual of a decayed field can be ~1e-22, whose FP32
  // squares underflow); the update divides the scale out
  s.outer += 1;
  const double n_sites = (double)rr.nx * rr.ny * rr.nz;
  const double rms = sqrt(s3[0] / n_sites);
  int e = rms > 0.0 ? -ilogb(rms) : 0;
  e = e < -120 ? -120 : (e > 120 ? 120 : e);
  const double sc = ldexp(1.0, e);
  s.scale = sc;
  s.rho = s3[2] * sc * sc;
  s.rnorm2 = s3[0] * sc * sc;
  s.bnorm2 = s3[0] * sc * sc;
  // inner tolerance: rtol_inner relative to this sweep's
  // defect, or, when the outer target is within a factor 8
  // of that (or looser), the reduction that reaches half the
  // outer target, so the last sweep neither over-solves nor
  // falls just short and costs another sweep
  const double q = 0.5 * tol / rel;
  s.rtol = q >= 0.125 * rr.rtol_inner ? q : rr.rtol_inner;
  s.maxit = rr.maxit;
  s.iters = 0;
  s.alpha = 0.0;
  s.beta = 0.0;
  s.dc_apply = 1;
  // the multigrid form leaves rho to the V-cycle (s3[2] = 0)
  s.active = (MG ? s3[0] > 0.0 : s3[2] > 0.0) ? 1 : 0;
}

template <int KIND, bool FIRST, bool MG, int NT>
__global__ void __launch_bounds__(NT, blocks_per_sm(NT)) k_dc_residual(Ctx c, int which, int field_map, CondArg outer,
                                                                        CondArg inner) {
  extern __shared__ __align__(16) float4 msm[];
  constexpr int NW = NT / 32, NS = 3;
  const int4 b = c.ablk[blockIdx.x];
  const int rep = b.x;
  const MGLevel& L = c.cg_lv[rep];
  const RepDesc& rd = c.reps[rep];
  const Patch p = patch_of<NT, 1>(L, b);
  const int zb = b.z, ze = b.w, ny = L.ny;
  const long long off = rd.off;
  const CUtensorMap* map_x = c.tmaps + L.map0 + field_map;   // x_hi, x_lo
  const CUtensorMap* map_s = c.tmaps + L.map0 + kMapReac;    // a, b, perfusion, V, K_prev
  __shared__ __align__(8) uint64_t bar[kXRing + kSRing];
  __shared__ double s_G0;
  __shared__ int s_last;
  __shared__ double s_sum[NS][NW];
  if (p.tid == 0) maps_acquire(map_x, 2);
  mbars_init(bar, kXRing + kSRing, map_s, 5);
  uint64_t* bar_s = bar + kXRing;
  HCA_COUNT_KERNEL(c);
  const RepSolve sv = c.solve[rep];
  const bool live = FIRST || sv.active || sv.dc_apply;
  double* slots = c.mslot + L.slot0;
  const int nslot = L.tx * L.ty * L.nseg;
  if (live) {
    if (KIND == 1 && FIRST) {
      if (p.tid == 0) s_G0 = substep_plasma(rd, which, *c.step, c.sub);
      __syncthreads();
    }
    const bool vegf = KIND == 1 && which == WHICH_VEGF;
    const bool lagged = KIND == 0 && FIRST && c.lag != nullptr;
    // the per-site inputs: a and b; in the first sweep the linearisation
    // field, or the perfusion and V
    const bool use0 = !FIRST || KIND == 1 || lagged, use1 = !FIRST || vegf;
    const CUtensorMap* map0 = !FIRST ? map_s : map_s + (KIND == 0 ? 4 : 2);
    const CUtensorMap* map1 = !FIRST ? map_s + 1 : map_s + 3;
    float* __restrict__ dd = (float*)c.d + off;
    float* __restrict__ aa = (float*)c.reac + off;
    float* __restrict__ ro = (float*)(MG ? c.r : c.z) + off;
    float* __restrict__ bb = (float*)c.b + off;
    const uint8_t* __restrict__ state = c.state + off;
    const Coef<float> q = coef<float, KIND>(rd, which);
    const float cpl32 = q.cpl;
    const float G0 = KIND == 1 && FIRST ? (float)s_G0 : 0.f;
    const bool bax = rd.bax[which] != 0;
    const bool o2t = KIND == 0 && rd.bx[0] != 0.0;
    const double bx = rd.bx[which];
    // bx as an unevaluated float pair (b = bx x0 + ... is formed to ~48 bits)
    const float bx_hi = (float)bx, bx_lo = (float)(bx - (double)bx_hi);
    const float bvessel = (float)(bax ? 2.0 * rd.r_K * rd.K0 : rd.r_K * rd.K0);
    const float av = (float)(bax ? 2.0 * rd.a_vegf : rd.a_vegf);
    float4* ring = align128(msm);                  // [plane & 3][x_hi, x_lo][row][group]
    float4* sring = ring + kXRing * 4 * NT;        // [plane & 1][two arrays][row][group]
    double* segs = reinterpret_cast<double*>(sring + kSRing * 4 * NT);   // [segment][sum][warp]
    const uint32_t box = 32u * (uint32_t)(L.cols * L.pairs);
    const int k0 = zb - 1;   // first plane of x
    int issued = 3, issued_s = 0;     // (thread 0)
    auto fetch = [&](int k) {
      const int s = (k - k0) & 3;
      mbar_expect_tx(&bar[s], 2 * box);
      tma_load_3d(ring + s * 4 * NT, &map_x[0], p.tx0, p.ty0, k, &bar[s]);
      tma_load_3d(ring + (s * 4 + 2) * NT, &map_x[1], p.tx0, p.ty0, k, &bar[s]);
    };
    auto fetch_s = [&](int k) {
      const int s = (k - zb) & 1;
      mbar_expect_tx(&bar_s[s], ((uint32_t)use0 + (uint32_t)use1) * box);
      if (use0) tma_load_3d(sring + s * 4 * NT, map0, p.tx0, p.ty0, k, &bar_s[s]);
      if (use1) tma_load_3d(sring + (s * 4 + 2) * NT, map1, p.tx0, p.ty0, k, &bar_s[s]);
    };
    if (p.tid == 0) {
      for (int k = k0; k < k0 + 3; ++k) fetch(k);
      if (use0 || use1) {
        fetch_s(zb);
        ++issued_s;
      }
    }
    // neighbours in x and y of the patch's sites
    float2 nxc[2];
    nxc[0] = make_float2((float)((p.x0 > 0) + (p.x0 < p.nx - 1)), (float)(1 + (p.x0 + 1 < p.nx - 1)));
    nxc[1] = make_float2((float)(1 + (p.x0 + 2 < p.nx - 1)), (float)(1 + (p.x0 + 3 < p.nx - 1)));
    int nyc[2];
#pragma unroll
    for (int a = 0; a < 2; ++a) nyc[a] = (p.y0 + a > 0) + (p.y0 + a < ny - 1);
    const int cols = L.cols;
    const int rm = p.r0 >= cols ? p.r0 - cols : p.r0;                       // the row below the patch
    const int rp = p.r1 + cols < 2 * cols * L.pairs ? p.r1 + cols : p.r1;   // the row above
    const bool l0 = p.l0 && p.r0 > 0;
    RunScale er, eb, ez;
    FF srr{0.f, 0.f}, sbb{0.f, 0.f}, srz{0.f, 0.f};
    int seg = 0;
    const int seglen = L.seg;
    uchar4 st[2] = {make_uchar4(0, 0, 0, 0), make_uchar4(0, 0, 0, 0)};
    if (FIRST) {
#pragma unroll
      for (int a = 0; a < 2; ++a)
        if (p.in[a]) st[a] = ld_state4(state + (p.e + (unsigned)zb * p.sz + a * p.sy));
    }
    bool ok = tc::mbar_wait(&bar[0], 0u, kTmaWaitLimit);
    ok &= tc::mbar_wait(&bar[1], 0u, kTmaWaitLimit);
    for (int z1 = zb; z1 < ze; ++z1) {
      const int n = z1 - zb;
      if (p.tid == 0) {
        if (z1 + 2 <= ze) {
          fetch(z1 + 2);
          ++issued;
        }
        if ((use0 || use1) && z1 + 1 < ze) {
          fetch_s(z1 + 1);
          ++issued_s;
        }
      }
      uchar4 stn[2] = {make_uchar4(0, 0, 0, 0), make_uchar4(0, 0, 0, 0)};   // the states of the next plane
      if (FIRST && z1 + 1 < ze) {
#pragma unroll
        for (int a = 0; a < 2; ++a)
          if (p.in[a]) stn[a] = ld_state4(state + (p.e + (unsigned)(z1 + 1) * p.sz + a * p.sy));
      }
      ok &= tc::mbar_wait(&bar[(n + 2) & 3], (uint32_t)((n + 2) >> 2) & 1u, kTmaWaitLimit);
      if (use0 || use1) ok &= tc::mbar_wait(&bar_s[n & 1], (uint32_t)(n >> 1) & 1u, kTmaWaitLimit);
      const float4* rc = ring + ((n + 1) & 3) * 4 * NT;   // the plane, the ones below and above
      const float4* rb = ring + (n & 3) * 4 * NT;
      const float4* rt = ring + ((n + 2) & 3) * 4 * NT;
      const float4* ss = sring + (n & 1) * 4 * NT;
      P8 xh, xl;
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        get_row(xh.v[a], rc + (a ? p.r1 : p.r0));
        get_row(xl.v[a], rc + 2 * NT + (a ? p.r1 : p.r0));
      }
      const unsigned e1 = p.e + (unsigned)z1 * p.sz;
      const int nz = (z1 > 0) + (z1 < p.nz - 1);
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        const int row = a ? p.r1 : p.r0;
        float lh = __shfl_up_sync(0xffffffffu, xh.v[a][1].y, 1), rh = __shfl_down_sync(0xffffffffu, xh.v[a][0].x, 1);
        float ll = __shfl_up_sync(0xffffffffu, xl.v[a][1].y, 1), rl = __shfl_down_sync(0xffffffffu, xl.v[a][0].x, 1);
        if (!p.in[a]) continue;
        if (l0) {
          lh = reinterpret_cast<const float*>(rc + row)[-1];
          ll = reinterpret_cast<const float*>(rc + 2 * NT + row)[-1];
        }
        if (p.l31) {
          rh = reinterpret_cast<const float*>(rc + row)[4];
          rl = reinterpret_cast<const float*>(rc + 2 * NT + row)[4];
        }
        float2 AR[2], B[2], D[2], R[2], Z[2], SRC;
        auto half = [&](const float4* f, int h) { return reinterpret_cast<const float2*>(f)[h]; };
        const unsigned e = e1 + a * p.sy;
        const float2 nyz = dup((float)(nyc[a] + nz));
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const FF2 xv{xh.v[a][h], xl.v[a][h]};
          if (!FIRST) {
            AR[h] = half(ss + row, h);
            B[h] = half(ss + 2 * NT + row, h);
          } else {
            const float2 pf = use0 ? half(ss + row, h) : make_float2(0.f, 0.f);
            const float2 vc = use1 ? half(ss + 2 * NT + row, h) : make_float2(0.f, 0.f);
            // x0 bx to ~48 bits, rounded once; x0 rounded to FP32
            const FF2 xbx = ff_mul(xv, FF2{dup(bx_hi), dup(bx_lo)});
            const float2 xb = __fadd2_rn(xbx.hi, xbx.lo), x32 = __fadd2_rn(xv.hi, xv.lo);
            float* ar = &AR[h].x;
            float* bv = &B[h].x;
            float* sr = &SRC.x;
#pragma unroll
            for (int w = 0; w < 2; ++w) {
              const int j = 2 * h + w;
              const uint8_t s = st_at(st[a], j);
              const float p0 = w ? pf.y : pf.x, v0 = w ? vc.y : vc.x, xb32 = w ? xb.y : xb.x;
              // the operator is linearised about K_prev: the start field, or c.lag when the solve starts from another guess
              const float lag = lagged ? p0 : (w ? x32.y : x32.x);
              const bool pad = p.part && p.x0 + j >= p.nx;
              float S, Bv;
              const float A = reaction_site<float, KIND>(q, s, lag, p0);
              if (KIND == 0) {
                S = is_vessel(s) ? bvessel : 0.f;
                Bv = S + (o2t ? xb32 : 0.f);
              } else {
                if (vegf) S = is_consumer(s) ? av * v0 : 0.f;
                else S = is_vessel(s) ? __fmul_rn(__fmul_rn(q.kappa, p0), G0) : 0.f;
                Bv = __fadd_rn(xb32, S);
              }
              ar[w] = pad ? 0.f : A;
              sr[w] = pad ? 0.f : S;
              bv[w] = pad ? 0.f : Bv;
            }
          }
          // r = b - (d x - c sum_nb x) in float-float (~48 bits): the
          // operator's terms cancel to the small defect; -d = -c n - a is
          // formed exactly from the stored reaction a
          const float2 n = __fadd2_rn(nxc[h], nyz);
          const float2 xh0 = xh.v[a][0], xh1 = xh.v[a][1], xl0 = xl.v[a][0], xl1 = xl.v[a][1];
          const FF2 xm = h ? FF2{make_float2(xh0.y, xh1.x), make_float2(xl0.y, xl1.x)}
                           : FF2{make_float2(lh, xh0.x), make_float2(ll, xl0.x)};
          const FF2 xp = h ? FF2{make_float2(xh1.y, rh), make_float2(xl1.y, rl)}
                           : FF2{make_float2(xh0.y, xh1.x), make_float2(xl0.y, xl1.x)};
          const FF2 yo{xh.v[1 - a][h], xl.v[1 - a][h]}, yn{half(rc + (a ? rp : rm), h), half(rc + 2 * NT + (a ? rp : rm), h)};
          const FF2 nb = ff_add(ff_add(ff_add(xm, xp), a ? ff_add(yo, yn) : ff_add(yn, yo)),
                                ff_add(FF2{half(rb + row, h), half(rb + 2 * NT + row, h)}, FF2{half(rt + row, h), half(rt + 2 * NT + row, h)}));
          const FF2 md = ff_add(ff_two_prod(dup(-cpl32), n), neg2(AR[h]));
          const FF2 mt = ff_add(ff_mul(md, xv), ff_mul(nb, dup(cpl32)));
          if (FIRST || !MG) D[h] = __ffma2_rn(dup(cpl32), n, AR[h]);
          // Crank-Nicolson: b = (4/h) x0 - A x0 + source, formed once from the start field
          if (FIRST && bax) {
            const FF2 bf = ff_add(ff_add(ff_mul(xv, FF2{dup(bx_hi), dup(bx_lo)}), SRC), mt);
            B[h] = __fadd2_rn(bf.hi, bf.lo);
          }
          const FF2 rf = ff_add(mt, B[h]);
          R[h] = __fadd2_rn(rf.hi, rf.lo);
          if (p.part) {   // padding sites hold 0
            if (p.x0 + 2 * h >= p.nx) D[h].x = B[h].x = R[h].x = 0.f;
            if (p.x0 + 2 * h + 1 >= p.nx) D[h].y = B[h].y = R[h].y = 0.f;
          }
          if (!MG) Z[h] = make_float2(D[h].x != 0.f ? R[h].x / D[h].x : 0.f, D[h].y != 0.f ? R[h].y / D[h].y : 0.f);
        }
        if (FIRST) {
          *reinterpret_cast<float4*>(dd + e) = make_float4(D[0].x, D[0].y, D[1].x, D[1].y);
          *reinterpret_cast<float4*>(aa + e) = make_float4(AR[0].x, AR[0].y, AR[1].x, AR[1].y);
          *reinterpret_cast<float4*>(bb + e) = make_float4(B[0].x, B[0].y, B[1].x, B[1].y);
          if (MG && c.mg_w)   // 1/d for the sweeps of a lattice without coarse levels (0 where d = 0), as k_mg_w0 forms it
            *reinterpret_cast<float4*>((float*)c.mg_w + off + e) =
                make_float4(D[0].x != 0.f ? 1.f / D[0].x : 0.f, D[0].y != 0.f ? 1.f / D[0].y : 0.f,
                            D[1].x != 0.f ? 1.f / D[1].x : 0.f, D[1].y != 0.f ? 1.f / D[1].y : 0.f);
        }
        const float2* o = MG ? R : Z;
        *reinterpret_cast<float4*>(ro + e) = make_float4(o[0].x, o[0].y, o[1].x, o[1].y);
        // |r|^2 (, |b|^2, r.z) in FP32 at the running scale, summed as a float-float pair
        auto big = [](const float2* v) { return fmaxf(fmaxf(fabsf(v[0].x), fabsf(v[0].y)), fmaxf(fabsf(v[1].x), fabsf(v[1].y))); };
        auto dot = [](const float2* u, const float2* v, float iu, float iv) {
          float2 t = __fmul2_rn(__fmul2_rn(u[0], dup(iu)), __fmul2_rn(v[0], dup(iv)));
          t = __ffma2_rn(__fmul2_rn(u[1], dup(iu)), __fmul2_rn(v[1], dup(iv)), t);
          return t.x + t.y;
        };
        const float fr = er.take(big(R));
        if (fr != 1.f) srr = scaled(scaled(srr, fr), fr);
        srr = ff_add(srr, dot(R, R, er.inv, er.inv));
        if (FIRST) {
          const float fb = eb.take(big(B));
          if (fb != 1.f) sbb = scaled(scaled(sbb, fb), fb);
          sbb = ff_add(sbb, dot(B, B, eb.inv, eb.inv));
        }
        if (!MG) {   // |z| may be far from |r|: each has its own scale
          const float fz = ez.take(big(Z));
          if (fr != 1.f || fz != 1.f) srz = scaled(scaled(srz, fr), fz);
          srz = ff_add(srz, dot(R, Z, er.inv, ez.inv));
        }
      }
      if (((z1 + 1) % seglen) == 0 || z1 == ze - 1) {   // the warp's sums of a segment
        const float fr = er.join(), fb = FIRST ? eb.join() : 1.f, fz = MG ? 1.f : ez.join();
        const FF s0 = row_reduce_ff(scaled(scaled(srr, fr), fr), 32);
        FF s1{0.f, 0.f}, s2{0.f, 0.f};
        if (FIRST) s1 = row_reduce_ff(scaled(scaled(sbb, fb), fb), 32);
        if (!MG) s2 = row_reduce_ff(scaled(scaled(srz, fr), fz), 32);
        if (p.lane == 0) {
          double* t = segs + seg * NS * NW + (p.tid >> 5);
          const double vr = er.value();
          t[0] = ((double)s0.hi + (double)s0.lo) * vr * vr;
          if (FIRST) t[NW] = ((double)s1.hi + (double)s1.lo) * eb.value() * eb.value();
          if (!MG) t[2 * NW] = ((double)s2.hi + (double)s2.lo) * vr * ez.value();
        }
        srr = sbb = srz = FF{0.f, 0.f};
        er = eb = ez = RunScale{};
        ++seg;
      }
      if (FIRST) {
        st[0] = stn[0];
        st[1] = stn[1];
      }
      if (__syncthreads_or(!ok)) {   // a copy timed out: every thread goes on to the arrivals, where the error ends the loops
        tma_abort(c, bar, kXRing, n + 2, issued);
        tma_abort(c, bar_s, kSRing, n, issued_s);
        break;
      }
    }
    for (int i = p.tid; i < seg * NS; i += NT) {
      const int s = i / NS, d = i - s * NS;
      if ((d == 1 && !FIRST) || (d == 2 && MG)) continue;
      double t = 0.0;
      for (int w = 0; w < NW; ++w) t += segs[i * NW + w];
      slots[(long long)d * nslot + (long long)b.y * L.nseg + zb / seglen + s] = t;
    }
  }
  // the replicate's last block adds the segments in a fixed order; the last
  // replicate sets the loop conditions
  __threadfence();
  __syncthreads();
  if (p.tid == 0) s_last = atomicAdd(&c.mcnt[rep], 1) == L.nblk - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (live) {
#pragma unroll
    for (int d = 0; d < NS; ++d) {
      if ((d == 1 && !FIRST) || (d == 2 && MG)) continue;
      double t = 0.0;
#pragma unroll 8
      for (int i = p.tid; i < nslot; i += NT) t += __ldcg(&slots[(long long)d * nslot + i]);
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (p.lane == 0) s_sum[d][p.tid >> 5] = t;
    }
    __syncthreads();
  }
  if (p.tid != 0) return;
  c.mcnt[rep] = 0;
  if (live) {
    double s3[NS] = {0.0, 0.0, 0.0};
    for (int d = 0; d < NS; ++d)
      if (!(d == 1 && !FIRST) && !(d == 2 && MG))
        for (int w = 0; w < NW; ++w) s3[d] += s_sum[d][w];
    dc_finish<FIRST, MG>(c, rep, which, s3);
  }
  __threadfence();
  if (atomicAdd(&c.sync->ticket, 1u) != (unsigned)c.n_reps - 1u) return;
  __threadfence();
  c.sync->ticket = 0u;
  int n_active = 0;
  for (int r = 0; r < c.n_reps; ++r) n_active += *(volatile int*)&c.solve[r].active;
  c.sync->active_count = n_active;
  c.sync->parity = 0;
  c.sync->guard = 0;
  const int g = FIRST ? (c.sync->guard_outer = 0) : ++c.sync->guard_outer;
  bool go = n_active > 0 && *(volatile int*)&c.sync->error != SYNC_ERR_TIMEOUT;
  if (go && g >= c.sync->guard_outer_limit) {
    c.sync->error = 2;
    go = false;
  }
  set_cond(outer, go);
  set_cond(inner, go);
}

template <int KIND, bool FIRST, bool MG, int NT>
bool dc_init_t() {
  return cudaFuncSetAttribute((const void*)k_dc_residual<KIND, FIRST, MG, NT>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dc_smem(NT)) == cudaSuccess;
}
template <int NT>
bool dc_init_nt() {
  return dc_init_t<0, true, true, NT>() && dc_init_t<1, true, true, NT>() && dc_init_t<0, false, true, NT>() &&
         dc_init_t<0, true, false, NT>() && dc_init_t<1, true, false, NT>() && dc_init_t<0, false, false, NT>();
}
template <bool MG, int NT>
void dc_launch(const Ctx& c, int which, bool first, CondArg outer, CondArg inner) {
  const dim3 g(c.n_ablk), t(NT);
  const int fm = kMapFields + 2 * which;
  const bool pdl = c.pdl != 0;
  if (first && which == 0)
    launch_k(pdl, k_dc_residual<0, true, MG, NT>, g, t, dc_smem(NT), c.stream, c, which, fm, outer, inner);
  else if (first)
    launch_k(pdl, k_dc_residual<1, true, MG, NT>, g, t, dc_smem(NT), c.stream, c, which, fm, outer, inner);
  else   // a later sweep only reads a and b: one kernel for every operator
    launch_k(pdl, k_dc_residual<0, false, MG, NT>, g, t, dc_smem(NT), c.stream, c, which, fm, outer, inner);
}

}  // namespace

// Dynamic shared memory of the residual sweep in the current context.
bool dc_init() {
  const bool ok = dc_init_nt<64>() && dc_init_nt<128>() && dc_init_nt<256>();
  if (!ok) (void)cudaGetLastError();
  return ok;
}

void launch_dc_residual(const Ctx& c, int which, bool first, CondArg outer, CondArg inner) {
  switch (c.a_nt) {
    case 64:
      if (c.mg) dc_launch<true, 64>(c, which, first, outer, inner);
      else dc_launch<false, 64>(c, which, first, outer, inner);
      break;
    case 128:
      if (c.mg) dc_launch<true, 128>(c, which, first, outer, inner);
      else dc_launch<false, 128>(c, which, first, outer, inner);
      break;
    default:
      if (c.mg) dc_launch<true, 256>(c, which, first, outer, inner);
      else dc_launch<false, 256>(c, which, first, outer, inner);
  }
}

}  // namespace hca
