// Matrix-free 7-point operators and the Jacobi-preconditioned CG passes for
// the oxygen (Eq. oxygen, s_K = 0, consumption linearised about the previous
// K as in Section 2.4.1) and drug (Eq. chemo, one implicit-Euler step) solves.
//
// Operator at site i (Neumann boundaries: out-of-box neighbours are omitted):
//     (A u)_i = d_i u_i - c * sum_{j in box, |i-j| = 1} u_j,
//     d_i = c * n_i + a_i,      c = D / dx^2,  n_i = in-box neighbour count,
//     oxygen: a_i = phi_K / (K1 + K_prev,i) [consumer] + r_K [vessel],  b_i = r_K K0 [vessel]
//     drug:   a_i = 1/dt + psi + kappa perf_i [vessel] + uptake [cancer],
//             b_i = G^n_i / dt + kappa perf_i G_0(t^{n+1}) [vessel].
//
// CG is carried in the preconditioned residual z = r / d instead of r, so
// the direction update p = z + beta p needs no division at neighbour sites:
//   pass A: p = z + beta p;  q = A p, stored;  sigma = p.q
//   pass B: x += alpha p;  z -= alpha q / d;  rho = r.z = sum d z^2,
//           |r|^2 = sum (d z)^2  (multigrid form: r -= alpha q, |r|^2; the
//           V-cycle then forms z = M r and rho)
// The row kernels here are the FP64 passes (FP32: cg.cu), the set-up, the
// residual of a finished solve, and what FP32's defect correction does
// besides its residual sweep (dc.cu).  Pass A rebuilds the new direction at
// neighbour sites from the old one, so the old and new directions live in two
// buffers that swap roles every iteration (an in-place update would let one
// block read a neighbour row another block has already overwritten); a parity
// bit in device memory, flipped by pass B, names the current buffer, so the
// same two kernels form the body of a graph loop.
#include <vector>

#include <cstdlib>

#include "hca_internal.cuh"
#include "reaction.cuh"
#include "row_ops.cuh"

namespace hca {
namespace {

// ------------------------------------------------------------------ setup --
// r = b - A x0 with x0 the current field; writes d, z = r/d (and b for drugs
// and the time-dependent oxygen form); reduces rho = r.z, |r|^2, |b|^2.
template <typename T, int KIND>
__global__ void __launch_bounds__(512) k_setup(Ctx c, int which, CondArg cnd) {
  HCA_COUNT_KERNEL(c);
  __shared__ double s_G0;
  const int2 ch = c.chunks[blockIdx.x];
  const RepDesc& rd = c.reps[ch.x];
  const int nrows = min(rd.chunk_rows, rd.ny * rd.nz - ch.y);
  const T* __restrict__ x = KIND == 0 ? (const T*)c.K : (const T*)c.G[which - 1];
  const T* __restrict__ perf = (const T*)c.perf;
  T* __restrict__ dd = (T*)c.d;
  T* __restrict__ zz = (T*)c.z;
  T* __restrict__ bb = (T*)c.b;
  if (KIND == 1) {
    if (threadIdx.x == 0) s_G0 = substep_plasma(rd, which, *c.step, c.sub);
    __syncthreads();
  }
  const T G0 = KIND == 1 ? (T)s_G0 : T(0);
  const Coef<T> q = coef<T, KIND>(rd, which);
  const T cpl = q.cpl;
  const T bx = (T)rd.bx[which];
  const bool bax = rd.bax[which] != 0;
  const bool o2t = KIND == 0 && rd.bx[0] != 0.0;   // time-dependent oxygen: b depends on x0
  const T bvessel = (T)(bax ? 2.0 * rd.r_K * rd.K0 : rd.r_K * rd.K0);
  const T av = (T)(bax ? 2.0 * rd.a_vegf : rd.a_vegf);
  const RowIter it = row_iter(rd);
  for (int rbase = it.warp * it.rpw; rbase < rd.chunk_rows; rbase += it.nw * it.rpw) {
    const int rl = rbase + it.sub;
    const bool row_ok = rl < nrows;
    const RowGeo geo = row_geo(rd, ch.y + (row_ok ? rl : 0));
    double acc[NDOT] = {0.0, 0.0, 0.0};
    T carry = T(0);
    for (int itn = 0; itn < it.niter; ++itn) {
      const int g = itn * it.lpr + it.sl;
      const bool gok = row_ok && g < rd.gpr;
      const long long e = geo.base + 4LL * g;
      const V4<T> X = ld4_if(x + e, gok);
      const V4<T> ym = ld4_if(x + e - geo.sy, gok && geo.ym);
      const V4<T> yp = ld4_if(x + e + geo.sy, gok && geo.yp);
      const V4<T> zm = ld4_if(x + e - geo.sz, gok && geo.zm);
      const V4<T> zp = ld4_if(x + e + geo.sz, gok && geo.zp);
      T left, right;
      x_neighbours(X, g, rd.gpr, it.sl, it.lpr, gok, carry, left, right, [&] { return x[e + 4]; });
      if (gok) {
        const uchar4 st = ld_state4(c.state + e);
        V4<T> PF = zero4<T>();
        if (KIND == 1) PF = ld4(perf + e);
        // the VEGF field's source is the cells' release a_V Vc (doubled under Crank-Nicolson)
        const bool vegf = KIND == 1 && which == WHICH_VEGF;
        const V4<T> VC = vegf ? ld4((const T*)c.Vc + e) : zero4<T>();
        const V4<T> LG = (KIND == 0 && c.lag) ? ld4((const T*)c.lag + e) : X;
        V4<T> D, Z, B, RR = zero4<T>();
        T g_rho = 0, g_rr = 0, g_bb = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int xk = 4 * g + k;
          const uint8_t s = st_at(st, k);
          T dk = T(0), zk = T(0), bk = T(0);
          if (xk < rd.nx) {
            dk = diag_site<T, KIND>(q, neighbour_count(rd, geo, xk), s, LG.a[k], PF.a[k]);
            if (KIND == 0) bk = (is_vessel(s) ? bvessel : T(0)) + (o2t ? X.a[k] * bx : T(0));
            else if (vegf) bk = X.a[k] * bx + (is_consumer(s) ? av * VC.a[k] : T(0));
            else bk = X.a[k] * bx + (is_vessel(s) ? q.kappa * PF.a[k] * G0 : T(0));
            const T ax = dk * X.a[k] - cpl * nb_sum(X, k, left, right, ym, yp, zm, zp);
            if (bax) bk -= ax;   // Crank-Nicolson: b = (4/h) x0 - A x0 + f^{k-1} + f^k
            const T r = bk - ax;
            RR.a[k] = r;
            zk = dk != T(0) ? r / dk : T(0);   // d = 0 only for an isolated, empty 1-site box
            g_rho += r * zk;
            g_rr += r * r;
            g_bb += bk * bk;
          }
          D.a[k] = dk;
          Z.a[k] = zk;
          B.a[k] = bk;
        }
        st4(dd + e, D);
        st4(zz + e, Z);
        if (c.mg) st4((T*)c.r + e, RR);
        if (KIND == 1 || o2t) st4(bb + e, B);
        acc[0] += (double)g_rho;
        acc[1] += (double)g_rr;
        acc[2] += (double)g_bb;
      }
    }
    store_row(c, blockIdx.x, rl, row_ok, it.sl, it.lpr, acc, 3);
  }
  const double rtol = KIND == 0 ? rd.rtol_o2 : rd.rtol_drug;
  (void)rtol;
  warp_epilogue(c, 3, blockIdx.x,
                 [&](int r, const double* s3) -> int {
                   const RepDesc& rr = c.reps[r];
                   RepSolve& sv = c.solve[r];
                   const double tol = which == 0 ? rr.rtol_o2 : rr.rtol_drug;
                   if (c.frozen[r]) {
                     sv.active = 0;
                     sv.zero_b = 0;
                     sv.iters = 0;
                     sv.rnorm2 = 0.0;
                     sv.bnorm2 = 1.0;
                     sv.scale = 1.0;
                     return 0;
                   }
                   sv.rho = s3[0];
                   sv.rnorm2 = s3[1];
                   sv.bnorm2 = s3[2];
                   sv.alpha = 0.0;
                   sv.beta = 0.0;
                   sv.scale = 1.0;
                   sv.iters = 0;
                   sv.pend = 0;
                   sv.rtol = tol;
                   sv.maxit = rr.maxit;
                   sv.zero_b = s3[2] == 0.0;
                   const bool fin = isfinite(s3[0]) && isfinite(s3[1]) && isfinite(s3[2]);
                   if (!fin) c.sync->error = 1;
                   sv.active = fin && !sv.zero_b && sqrt(s3[1]) > tol * sqrt(s3[2]) && rr.maxit > 0;
                   return sv.active;
                 },
                 [&](int n_active) {
                   c.sync->parity = 0;
                   c.sync->guard = 0;
                   set_cond(cnd, n_active > 0);
                 });
}

// ----------------------------------------------------------------- pass A --
// FP64 fields (FP32: cg.cu).  All loads of a group (own site and the four
// neighbour rows) are issued before any value is used, so a group costs one
// memory round trip; one block per chunk.
template <typename T>
__global__ void __maxnreg__(128) k_pass_a(Ctx c, int which) {
  HCA_COUNT_KERNEL(c);
  const int2 ch = c.chunks[blockIdx.x];
  const RepDesc& rd = c.reps[ch.x];
  const RepSolve sv = c.solve[ch.x];
  if (sv.active) {
    const int nrows = min(rd.chunk_rows, rd.ny * rd.nz - ch.y);
    const int gpr = rd.gpr;
    const int par = c.sync->parity;
    const T* __restrict__ pp = (const T*)(par ? c.p_alt : c.p);
    T* __restrict__ p_new = (T*)(par ? c.p : c.p_alt);
    const T* __restrict__ zz = (const T*)c.z;
    const T* __restrict__ dd = (const T*)c.d;
    T* __restrict__ qq = (T*)c.q;
    const T beta = (T)sv.beta;
    const bool use_p = sv.beta != 0.0;
    // the first iteration of a rescaled inner solve starts from scale * z
    // (the V-cycle scales r itself before it forms z)
    const T zs = (sv.iters == 0 && !c.mg) ? (T)sv.scale : T(1);
    const T cpl = op_coupling_t<T>(rd, which);
    const RowIter it = row_iter(rd);
    // one row j (chunk slot rl of `chunk`; row_ok false: a padding slot of the last chunk)
    auto row = [&](int chunk, int rl, bool row_ok, int j) {
      const RowGeo geo = row_geo(rd, j);
      LaneAcc<T> acc[1];
      T carry = T(0);
      for (int itn = 0; itn < it.niter; ++itn) {
        const int g = itn * it.lpr + it.sl;
        const bool gok = row_ok && g < gpr;
        const long long e = geo.base + 4LL * g;
        const bool last_lane = it.sl == it.lpr - 1 && gok && g + 1 < gpr;
        // issue every load of this group
        const V4<T> z0 = ld4_if(zz + e, gok);
        const V4<T> zym = ld4_if(zz + e - geo.sy, gok && geo.ym);
        const V4<T> zyp = ld4_if(zz + e + geo.sy, gok && geo.yp);
        const V4<T> zzm = ld4_if(zz + e - geo.sz, gok && geo.zm);
        const V4<T> zzp = ld4_if(zz + e + geo.sz, gok && geo.zp);
        const V4<T> D = ld4_if(dd + e, gok);
        const T zr = last_lane ? zz[e + 4] : T(0);
        V4<T> p0 = zero4<T>(), pym = zero4<T>(), pyp = zero4<T>(), pzm = zero4<T>(), pzp = zero4<T>();
        T pr = T(0);
        if (use_p) {
          p0 = ld4_if(pp + e, gok);
          pym = ld4_if(pp + e - geo.sy, gok && geo.ym);
          pyp = ld4_if(pp + e + geo.sy, gok && geo.yp);
          pzm = ld4_if(pp + e - geo.sz, gok && geo.zm);
          pzp = ld4_if(pp + e + geo.sz, gok && geo.zp);
          pr = last_lane ? pp[e + 4] : T(0);
        }
        // new direction at the site and at its neighbours: p = z + beta p_old
        V4<T> PN, ym, yp, zm, zp;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          PN.a[k] = cg_dir(zs, z0.a[k], beta, p0.a[k]);
          ym.a[k] = cg_dir(zs, zym.a[k], beta, pym.a[k]);
          yp.a[k] = cg_dir(zs, zyp.a[k], beta, pyp.a[k]);
          zm.a[k] = cg_dir(zs, zzm.a[k], beta, pzm.a[k]);
          zp.a[k] = cg_dir(zs, zzp.a[k], beta, pzp.a[k]);
        }
        const T right_next = cg_dir(zs, zr, beta, pr);
        T left, right;
        x_neighbours(PN, g, gpr, it.sl, it.lpr, gok, carry, left, right, [&] { return right_next; });
        if (gok) {
          T g_s = 0;
          V4<T> Q;
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            Q.a[k] = cg_apply(D.a[k], PN.a[k], cpl, nb_sum(PN, k, left, right, ym, yp, zm, zp));
            g_s = cg_madd(PN.a[k], Q.a[k], g_s);
          }
          st4(p_new + e, PN);
          st4(qq + e, Q);   // pass B reads A p instead of re-forming it from p's neighbours
          acc[0].add(g_s);
        }
      }
      store_rows_acc(c, chunk, rl, row_ok, it.sl, it.lpr, acc, 1);
    };
    for (int rbase = it.warp * it.rpw; rbase < rd.chunk_rows; rbase += it.nw * it.rpw) {
      const int rl = rbase + it.sub;
      const bool row_ok = rl < nrows;
      row(blockIdx.x, rl, row_ok, ch.y + (row_ok ? rl : 0));
    }
  }
  auto fin = [&](int r, const double* s1) -> int {
    RepSolve& s = c.solve[r];
    if (!s.active) return 0;
    if (!(s1[0] > 0.0) || !isfinite(s1[0])) {
      if (!isfinite(s1[0])) c.sync->error = 1;
      s.active = 0;
      return 0;
    }
    s.alpha = s.rho / s1[0];
    return 1;
  };
  warp_epilogue(c, 1, blockIdx.x, fin);
}

// ----------------------------------------------------------------- pass B --
template <typename T>
__global__ void __maxnreg__(128) k_pass_b(Ctx c, int which, void* xfield, CondArg cnd) {
  HCA_COUNT_KERNEL(c);
  const int2 ch = c.chunks[blockIdx.x];
  const RepDesc& rd = c.reps[ch.x];
  const RepSolve sv = c.solve[ch.x];
  if (sv.active) {
    const int nrows = min(rd.chunk_rows, rd.ny * rd.nz - ch.y);
    const int gpr = rd.gpr, nx = rd.nx;
    // Jacobi form: z = r / d is carried; V-cycle form: r itself (already scaled)
    const bool mg = c.mg != 0;
    T* __restrict__ zz = (T*)(mg ? c.r : c.z);
    const T* __restrict__ pp = (const T*)(c.sync->parity ? c.p : c.p_alt);
    const T* __restrict__ dd = (const T*)c.d;
    const T* __restrict__ qq = (const T*)c.q;
    T* __restrict__ xx = (T*)xfield;
    const T alpha = (T)sv.alpha;
    const T zs = (sv.iters == 0 && !mg) ? (T)sv.scale : T(1);
    const RowIter it = row_iter(rd);
    auto row = [&](int chunk, int rl, bool row_ok, int j) {
      const RowGeo geo = row_geo(rd, j);
      LaneAcc<T> acc[2];
      for (int itn = 0; itn < it.niter; ++itn) {
        const int g = itn * it.lpr + it.sl;
        const bool gok = row_ok && g < gpr;
        const long long e = geo.base + 4LL * g;
        // issue every load of this group (A p comes from pass A)
        const V4<T> P = ld4_if(pp + e, gok);
        const V4<T> Q = ld4_if(qq + e, gok);
        const V4<T> D = mg ? zero4<T>() : ld4_if(dd + e, gok);
        V4<T> X = ld4_if(xx + e, gok);
        V4<T> Z = ld4_if(zz + e, gok);
        if (gok) {
          T g_rho = 0, g_rr = 0;
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            if (4 * g + k < nx) {
              const T q = Q.a[k];
              X.a[k] += alpha * P.a[k];
              if (mg) {
                Z.a[k] -= alpha * q;
                g_rr += Z.a[k] * Z.a[k];
              } else {
                Z.a[k] = zs * Z.a[k] - alpha * (q / D.a[k]);
                const T r = D.a[k] * Z.a[k];
                g_rho += r * Z.a[k];
                g_rr += r * r;
              }
            }
          }
          st4(xx + e, X);
          st4(zz + e, Z);
          acc[0].add(g_rho);
          acc[1].add(g_rr);
        }
      }
      store_rows_acc(c, chunk, rl, row_ok, it.sl, it.lpr, acc, 2);
    };
    for (int rbase = it.warp * it.rpw; rbase < rd.chunk_rows; rbase += it.nw * it.rpw) {
      const int rl = rbase + it.sub;
      const bool row_ok = rl < nrows;
      row(blockIdx.x, rl, row_ok, ch.y + (row_ok ? rl : 0));
    }
  }
  auto fin = [&](int r, const double* s2) -> int {
    RepSolve& s = c.solve[r];
    if (!s.active) return 0;
    s.iters += 1;
    if (!isfinite(s2[0]) || !isfinite(s2[1])) {
      c.sync->error = 1;
      s.active = 0;
      return 0;
    }
    if (!c.mg) {   // the V-cycle form sets beta and rho after z = M r
      s.beta = s2[0] / s.rho;
      s.rho = s2[0];
    }
    s.rnorm2 = s2[1];
    const bool conv = sqrt(s2[1]) <= s.rtol * sqrt(s.bnorm2);
    if (conv || s.iters >= s.maxit) s.active = 0;
    return s.active;
  };
  auto post = [&](int n_active) {
    c.sync->parity ^= 1;
    const int g = ++c.sync->guard;
    bool go = n_active > 0;
    if (go && g >= c.sync->guard_limit) {
      // every replicate stops at maxit; this only guards the graph loop
      c.sync->error = 2;
      go = false;
    }
    set_cond(cnd, go);
  };
  warp_epilogue(c, 2, blockIdx.x, fin, post);
}

// ----------------------------------------------------------- true residual --
// rr = |b - A x|^2 with b rebuilt from the state (oxygen) or read back (drug);
// zeroes x where b = 0.  Records iterations and the relative residual in the
// statistics slot `which`.
template <typename T, int KIND>
__global__ void __launch_bounds__(512) k_true_residual(Ctx c, int which, void* xfield) {
  HCA_COUNT_KERNEL(c);
  const int2 ch = c.chunks[blockIdx.x];
  const RepDesc& rd = c.reps[ch.x];
  const RepSolve sv = c.solve[ch.x];
  const int nrows = min(rd.chunk_rows, rd.ny * rd.nz - ch.y);
  T* __restrict__ xx = (T*)xfield;
  const T* __restrict__ dd = (const T*)c.d;
  const T* __restrict__ bb = (const T*)c.b;
  const T cpl = op_coupling_t<T>(rd, which);
  const T bvessel = (T)(rd.r_K * rd.K0);
  const RowIter it = row_iter(rd);
  for (int rbase = it.warp * it.rpw; rbase < rd.chunk_rows; rbase += it.nw * it.rpw) {
    const int rl = rbase + it.sub;
    const bool row_ok = rl < nrows;
    const RowGeo geo = row_geo(rd, ch.y + (row_ok ? rl : 0));
    double acc[NDOT] = {0.0, 0.0, 0.0};
    T carry = T(0);
    for (int itn = 0; itn < it.niter; ++itn) {
      const int g = itn * it.lpr + it.sl;
      const bool gok = row_ok && g < rd.gpr;
      const long long e = geo.base + 4LL * g;
      const V4<T> X = ld4_if(xx + e, gok);
      const V4<T> ym = ld4_if(xx + e - geo.sy, gok && geo.ym);
      const V4<T> yp = ld4_if(xx + e + geo.sy, gok && geo.yp);
      const V4<T> zm = ld4_if(xx + e - geo.sz, gok && geo.zm);
      const V4<T> zp = ld4_if(xx + e + geo.sz, gok && geo.zp);
      T left, right;
      x_neighbours(X, g, rd.gpr, it.sl, it.lpr, gok, carry, left, right, [&] { return xx[e + 4]; });
      if (gok) {
        const V4<T> D = ld4(dd + e);
        V4<T> B;
        if (KIND == 0 && rd.bx[0] != 0.0) {
          B = ld4(bb + e);
        } else if (KIND == 0) {
          const uchar4 st = ld_state4(c.state + e);
#pragma unroll
          for (int k = 0; k < 4; ++k) B.a[k] = is_vessel(st_at(st, k)) ? bvessel : T(0);
        } else {
          B = ld4(bb + e);
        }
        T g_rr = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (4 * g + k < rd.nx) {
            const T r = B.a[k] - (D.a[k] * X.a[k] - cpl * nb_sum(X, k, left, right, ym, yp, zm, zp));
            g_rr += r * r;
          }
        }
        acc[0] += (double)g_rr;
      }
    }
    store_row(c, blockIdx.x, rl, row_ok, it.sl, it.lpr, acc, 1);
  }
  warp_epilogue(c, 1, blockIdx.x,
                 [&](int r, const double* s1) -> int {
                   RepSolve& s = c.solve[r];
                   DevStats& st = c.stats[r];
                   s.rel_true = s.zero_b ? 0.0 : sqrt(s1[0] / s.bnorm2);
                   st.iters[which] += s.iters;
                   st.rel[which] = s.rel_true;
                   if (!s.zero_b && !(sqrt(s.rnorm2) <= s.rtol * sqrt(s.bnorm2))) st.not_converged |= 1 << which;
                   if (!isfinite(s1[0])) {
                     c.sync->error = 1;
                     st.nonfinite = 1;
                   }
                   return 0;
                 });
  (void)sv;
}

// x = 0 for replicates whose right-hand side vanished.
template <typename T>
__global__ void k_zero_if_b_zero(Ctx c, void* xfield) {
  HCA_COUNT_KERNEL(c);
  const int2 ch = c.chunks[blockIdx.x];
  if (!c.solve[ch.x].zero_b) return;
  const RepDesc& rd = c.reps[ch.x];
  const int nrows = min(rd.chunk_rows, rd.ny * rd.nz - ch.y);
  T* xx = (T*)xfield;
  const long long base = rd.off + (long long)ch.y * rd.nxp;
  const long long n = (long long)nrows * rd.nxp;
  for (long long i = threadIdx.x; i < n; i += blockDim.x) xx[base + i] = T(0);
}

// ---------------------------------------------------------- apply operator --
// out = A u for one replicate (operator `which`, diagonal rebuilt from the
// state, the current K and the perfusion map).  Used to expose the stencil.
template <typename T, int KIND>
__global__ void __launch_bounds__(512) k_apply(Ctx c, int which, int rep, const T* __restrict__ u,
                                               T* __restrict__ out) {
  HCA_COUNT_KERNEL(c);
  const int2 ch = c.chunks[blockIdx.x];
  if (ch.x != rep) return;
  const RepDesc& rd = c.reps[ch.x];
  const int nrows = min(rd.chunk_rows, rd.ny * rd.nz - ch.y);
  const T* __restrict__ K = (const T*)c.K;
  const T* __restrict__ perf = (const T*)c.perf;
  const Coef<T> q = coef<T, KIND>(rd, which);
  const T cpl = q.cpl;
  const RowIter it = row_iter(rd);
  for (int rbase = it.warp * it.rpw; rbase < rd.chunk_rows; rbase += it.nw * it.rpw) {
    const int rl = rbase + it.sub;
    const bool row_ok = rl < nrows;
    const RowGeo geo = row_geo(rd, ch.y + (row_ok ? rl : 0));
    T carry = T(0);
    for (int itn = 0; itn < it.niter; ++itn) {
      const int g = itn * it.lpr + it.sl;
      const bool gok = row_ok && g < rd.gpr;
      const long long e = geo.base + 4LL * g;
      const V4<T> U = ld4_if(u + e, gok);
      const V4<T> ym = ld4_if(u + e - geo.sy, gok && geo.ym);
      const V4<T> yp = ld4_if(u + e + geo.sy, gok && geo.yp);
      const V4<T> zm = ld4_if(u + e - geo.sz, gok && geo.zm);
      const V4<T> zp = ld4_if(u + e + geo.sz, gok && geo.zp);
      T left, right;
      x_neighbours(U, g, rd.gpr, it.sl, it.lpr, gok, carry, left, right, [&] { return u[e + 4]; });
      if (gok) {
        const uchar4 st = ld_state4(c.state + e);
        const V4<T> KK = ld4(K + e);
        const V4<T> PF = ld4(perf + e);
        V4<T> O;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int xk = 4 * g + k;
          O.a[k] = T(0);
          if (xk < rd.nx) {
            const T dk = diag_site<T, KIND>(q, neighbour_count(rd, geo, xk), st_at(st, k), KK.a[k], PF.a[k]);
            O.a[k] = dk * U.a[k] - cpl * nb_sum(U, k, left, right, ym, yp, zm, zp);
          }
        }
        st4(out + e, O);
      }
    }
  }
}

// |a - b|^2 and |a|^2 per replicate (into solve[rep].rnorm2 / bnorm2); used
// by the fixed-point iteration of the initial oxygen field.
template <typename T>
__global__ void __launch_bounds__(512) k_diff_norms(Ctx c, const T* __restrict__ a, const T* __restrict__ b) {
  HCA_COUNT_KERNEL(c);
  const int2 ch = c.chunks[blockIdx.x];
  const RepDesc& rd = c.reps[ch.x];
  const int nrows = min(rd.chunk_rows, rd.ny * rd.nz - ch.y);
  const RowIter it = row_iter(rd);
  for (int rbase = it.warp * it.rpw; rbase < rd.chunk_rows; rbase += it.nw * it.rpw) {
    const int rl = rbase + it.sub;
    const bool row_ok = rl < nrows;
    const RowGeo geo = row_geo(rd, ch.y + (row_ok ? rl : 0));
    double acc[NDOT] = {0.0, 0.0, 0.0};
    for (int itn = 0; itn < it.niter; ++itn) {
      const int g = itn * it.lpr + it.sl;
      if (row_ok && g < rd.gpr) {
        const long long e = geo.base + 4LL * g;
        const V4<T> A = ld4(a + e), B = ld4(b + e);
        T s0 = 0, s1 = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const T df = A.a[k] - B.a[k];
          s0 += df * df;
          s1 += A.a[k] * A.a[k];
        }
        acc[0] += (double)s0;
        acc[1] += (double)s1;
      }
    }
    store_row(c, blockIdx.x, rl, row_ok, it.sl, it.lpr, acc, 2);
  }
  warp_epilogue(c, 2, blockIdx.x,
                 [&](int r, const double* s2) -> int {
                   c.solve[r].rnorm2 = s2[0];
                   c.solve[r].bnorm2 = s2[1];
                   return 0;
                 });
}

// x_hi + x_lo += dx (two-word sum), or x = 0 for a vanishing right-hand side.
// dx is what pass A of the later iterations accumulated plus the last
// iteration's step alpha p (0 + alpha p after a single iteration).
__global__ void __launch_bounds__(512) k_dc_update(Ctx c, float* __restrict__ x_hi, float* __restrict__ x_lo) {
  HCA_COUNT_KERNEL(c);
  const int2 ch = c.chunks[blockIdx.x];
  const RepSolve sv = c.solve[ch.x];
  if (!sv.dc_apply && !sv.zero_b) return;
  const RepDesc& rd = c.reps[ch.x];
  const int nrows = min(rd.chunk_rows, rd.ny * rd.nz - ch.y);
  const long long base0 = rd.off + (long long)ch.y * rd.nxp;
  const int ngroups = nrows * rd.gpr;
  const bool has_x = sv.iters - sv.pend > 0;
  const float* __restrict__ dxv = (const float*)c.dx;
  const float* __restrict__ pv = (const float*)(sv.pbuf ? c.p_alt : c.p);
  const float alpha = (float)sv.alpha;
  const float inv_s = (float)(1.0 / sv.scale);   // a power of two: exact
  for (int gi = threadIdx.x; gi < ngroups; gi += blockDim.x) {
    const long long e = base0 + 4LL * gi;   // rows follow each other
    if (sv.zero_b) {
      st4(x_hi + e, zero4<float>());
      st4(x_lo + e, zero4<float>());
      continue;
    }
    V4<float> H = ld4(x_hi + e), L = ld4(x_lo + e);
    V4<float> D = ld4_if(dxv + e, has_x);
    if (sv.pend) {
      const V4<float> P = ld4(pv + e);
#pragma unroll
      for (int k = 0; k < 4; ++k) D.a[k] = __fmaf_rn(alpha, P.a[k], D.a[k]);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) D.a[k] = __fmul_rn(D.a[k], inv_s);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      // two-sum of hi and dx, then renormalise with the low word
      const float s = __fadd_rn(H.a[k], D.a[k]);
      const float bv = __fsub_rn(s, H.a[k]);
      const float err = __fadd_rn(__fsub_rn(H.a[k], __fsub_rn(s, bv)), __fsub_rn(D.a[k], bv));
      const float lo = __fadd_rn(L.a[k], err);
      const float hi = __fadd_rn(s, lo);
      L.a[k] = __fsub_rn(lo, __fsub_rn(hi, s));
      H.a[k] = hi;
    }
    st4(x_hi + e, H);
    st4(x_lo + e, L);
  }
}

}  // namespace

// ------------------------------------------------------------- launchers --
void launch_dc_update(const Ctx& c, void* x_hi, void* x_lo) {
  launch_k(c.pdl != 0, k_dc_update, dim3(c.n_chunks), dim3(c.threads), 0, c.stream, c, (float*)x_hi, (float*)x_lo);
}

void launch_diff_norms(const Ctx& c, const void* a, const void* b, bool fp64) {
  if (fp64) k_diff_norms<double><<<c.n_chunks, c.threads, 0, c.stream>>>(c, (const double*)a, (const double*)b);
  else k_diff_norms<float><<<c.n_chunks, c.threads, 0, c.stream>>>(c, (const float*)a, (const float*)b);
}

template <typename T>
static void launch_setup_t(const Ctx& c, int which, CondArg cnd) {
  if (which == 0) k_setup<T, 0><<<c.n_chunks, c.threads, 0, c.stream>>>(c, which, cnd);
  else k_setup<T, 1><<<c.n_chunks, c.threads, 0, c.stream>>>(c, which, cnd);
}

void launch_setup(const Ctx& c, int which, bool fp64, CondArg cnd) {
  if (fp64) launch_setup_t<double>(c, which, cnd);
  else launch_setup_t<float>(c, which, cnd);
}

void launch_cg_a(const Ctx& c, int which, bool defer);
void launch_cg_b(const Ctx& c, int which, void* xfield, bool defer, CondArg cnd);

// FP32 fields: the marching pass A and streaming pass B (cg.cu); defer: the
// solve is a defect correction's inner one, whose x += alpha p pass A carries.
void launch_pass_a(const Ctx& c, int which, bool fp64, bool defer) {
  if (fp64) k_pass_a<double><<<c.n_chunks, c.threads, 0, c.stream>>>(c, which);
  else launch_cg_a(c, which, defer);
}

void launch_pass_b(const Ctx& c, int which, void* xfield, bool fp64, bool defer, CondArg cnd) {
  if (fp64) k_pass_b<double><<<c.n_chunks, c.threads, 0, c.stream>>>(c, which, xfield, cnd);
  else launch_cg_b(c, which, xfield, defer, cnd);
}

void launch_true_residual(const Ctx& c, int which, void* xfield, bool fp64) {
  if (fp64) {
    if (which == 0) k_true_residual<double, 0><<<c.n_chunks, c.threads, 0, c.stream>>>(c, which, xfield);
    else k_true_residual<double, 1><<<c.n_chunks, c.threads, 0, c.stream>>>(c, which, xfield);
    k_zero_if_b_zero<double><<<c.n_chunks, c.threads, 0, c.stream>>>(c, xfield);
  } else {
    if (which == 0) k_true_residual<float, 0><<<c.n_chunks, c.threads, 0, c.stream>>>(c, which, xfield);
    else k_true_residual<float, 1><<<c.n_chunks, c.threads, 0, c.stream>>>(c, which, xfield);
    k_zero_if_b_zero<float><<<c.n_chunks, c.threads, 0, c.stream>>>(c, xfield);
  }
}

void launch_apply(const Ctx& c, int which, int rep, const void* u, void* out, bool fp64) {
  if (fp64) {
    if (which == 0) k_apply<double, 0><<<c.n_chunks, c.threads, 0, c.stream>>>(c, which, rep, (const double*)u, (double*)out);
    else k_apply<double, 1><<<c.n_chunks, c.threads, 0, c.stream>>>(c, which, rep, (const double*)u, (double*)out);
  } else {
    if (which == 0) k_apply<float, 0><<<c.n_chunks, c.threads, 0, c.stream>>>(c, which, rep, (const float*)u, (float*)out);
    else k_apply<float, 1><<<c.n_chunks, c.threads, 0, c.stream>>>(c, which, rep, (const float*)u, (float*)out);
  }
}

}  // namespace hca
