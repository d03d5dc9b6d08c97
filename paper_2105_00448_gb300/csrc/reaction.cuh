// The operator's reaction part, shared by the solver kernels.
#pragma once

#include "hca_internal.cuh"

namespace hca {

// a + k p for the drug reaction: in FP32 rounded after the product and after
// the sum (no fused multiply-add), so the stored FP32 coefficients of the
// system are the plain IEEE result of these operations.
__device__ __forceinline__ float add_prod(float a, float k, float p) { return __fadd_rn(a, __fmul_rn(k, p)); }
__device__ __forceinline__ double add_prod(double a, double k, double p) { return a + k * p; }

// The coefficients of operator `which` in the field precision, converted
// from the handle's FP64 parameters once per thread: the conversions run on
// the FP64 pipe (a small fraction of the FP32 rate on this GPU), and the
// parameters sit in global memory, where the compiler cannot keep them in
// registers across the kernel's own stores.
template <typename T>
struct Coef {
  T cpl, phi_K, K1, r_K, o2_mass, base, kappa, uptake;
};
template <typename T, int KIND>
__device__ __forceinline__ Coef<T> coef(const RepDesc& rd, int which) {
  Coef<T> q;
  q.cpl = op_coupling_t<T>(rd, which);
  q.phi_K = q.K1 = q.r_K = q.o2_mass = q.base = q.kappa = q.uptake = T(0);
  if (KIND == 0) {
    q.phi_K = (T)rd.phi_K;
    q.K1 = (T)rd.K1;
    q.r_K = (T)rd.r_K;
    q.o2_mass = (T)rd.o2_mass;
  } else {
    const int dd = which - 1;
    q.base = (T)rd.base_drug[dd];
    q.kappa = (T)rd.kappa[dd];
    q.uptake = (T)rd.uptake[dd];
  }
  return q;
}

// Reaction coefficient a of the operator at one site (d = c n + a).
template <typename T, int KIND>
__device__ __forceinline__ T reaction_site(const Coef<T>& q, uint8_t s, T K_prev, T pf) {
  T a;
  if (KIND == 0) {
    a = is_consumer(s) ? q.phi_K / (q.K1 + K_prev) : T(0);
    if (is_vessel(s)) a += q.r_K;
    a += q.o2_mass;   // 0 for the quasi-steady form
  } else {
    a = q.base;
    if (is_vessel(s)) a = add_prod(a, q.kappa, pf);
    if (is_cancer(s)) a += q.uptake;
  }
  return a;
}

// Diagonal of the operator at one site.
template <typename T, int KIND>
__device__ __forceinline__ T diag_site(const Coef<T>& q, int n_nb, uint8_t s, T K_prev, T pf) {
  return q.cpl * (T)n_nb + reaction_site<T, KIND>(q, s, K_prev, pf);
}

}  // namespace hca
