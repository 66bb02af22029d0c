// pnp_lane.cuh -- the VMS PNP residual and its Jacobian action at one lane (element, corner),
// whose Gauss point is the one next to the corner (Def. 3 of arXiv 2301.05985 with the fine
// scales c^f = -tau_c R_c of Sec. 3.1; the same statement as element_kernels.cu).
#pragma once

#include "kernels.h"
#include "lane_ops.cuh"

namespace {

// physical parameters in the kernel's arithmetic type
template <typename T>
struct LaneParams {
  T kappa;   // beta0 / dt
  T tau_t;   // 4 / dt^2
  T cid;     // C_I d
  T e2;      // 2 Lambda^2
};
template <typename C>
LaneParams<C> lane_params(const PhysParams& P, int dim) {
  return LaneParams<C>{C(P.kappa), C(P.tau_t), C(P.C_I * dim), C(P.eps2x2)};
}

// Nodal values of the lane's corner (u: c+, c-, phi; h: history; v: advection; d: direction,
// JV only) -> the element vector's entries of the corner, without the factor
// lane_weight_c(D) 2^lane_weight_e(D, lev).  Scaled quantities (lane_ops.cuh; c~ = c / a^D,
// g~ = reflected gradient h / a^(D-1)):
//   V = (a^(D-1) / h) v~ reflected,  beta = a^(D-2) / h^2,  delta = a^2 h^2,  alpha = a^D
//   S~ = kappa c~ + h~ + V . g~c,   R~ = S~ - z beta g~phi . g~c          (times alpha)
//   Phi~ = g~c + z alpha (c~ - tau R~) g~phi + tau delta R~ V             (times a^(D-1) / h)
// and the element vector is (h/2)^D a^D beta times the test transpose of (delta S~, Phi~).
// ADV false: the advection is zero and not read.
constexpr double lane_weight_c(int D) { return ipow(kVal, 2 * D - 2); }
__device__ __forceinline__ int lane_weight_e(int D, int lev) { return 2 * lev - D * (lev + 1); }

template <typename C, int D, bool JV, bool ADV>
__device__ __forceinline__ void lane_pnp(const C (&un)[3], const C (&hn)[2], const C (&vn)[3], const C (&dn)[3], int c,
                                         int lev, const LaneParams<C>& K, pair_t<C>& rs, C& rp) {
  const C rho = C(kRho);
  const C beta = const_pow2(ipow(kVal, D - 2), 2 * lev, C(0));
  const C delta = const_pow2(kVal * kVal, -2 * lev, C(0));
  const C kappa = K.kappa, e2 = K.e2;
  // state at this lane's Gauss point; the species, (v_0, v_1) and (phi, v_2) or (phi, dphi)
  // run as pairs
  using C2 = pair_t<C>;
  const C2 rho2 = both<C>(rho);
  C V[D], vd[D], gp[3], dgp[3];
  if constexpr (ADV) {
    const C2 v01 = lane_v<C2, D>(pair(vn[0], vn[1]), rho2);
    vd[0] = first(v01);
    vd[1] = second(v01);
    if constexpr (JV && D == 3) vd[2] = lane_v<C, D>(vn[2], rho);
  }
  if constexpr (JV || (ADV && D == 3)) {
    C2 val, g[3];
    lane_vg<C2, D, !JV>(pair(un[2], JV ? dn[2] : vn[2]), rho2, val, g);
#pragma unroll
    for (int k = 0; k < D; ++k) {
      gp[k] = first(g[k]);
      if (JV) dgp[k] = second(g[k]);
    }
    if constexpr (!JV) vd[2] = second(val);
  } else {
    C unused;
    lane_vg<C, D, false>(un[2], rho, unused, gp);
  }
  // 4/dt^2 + C_I d (2/h)^4 + (2/h)^2 |v|^2
  C arg = times_pow2(K.cid, 4 * lev + 4) + K.tau_t;
  if constexpr (ADV) {
    C vv;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      vv = k == 0 ? vd[k] * vd[k] : fma_q(vd[k], vd[k], vv);
      V[k] = reflect(times_const(vd[k], ipow(kVal, D - 1), lev), reflect_mask(c, k));
    }
    arg = fma_q(const_pow2(ipow(kVal, 2 * D), 2 * lev + 2, C(0)), vv, arg);
  }
  const C tau = inv_sqrt(arg);
  const C2 taud = both<C>(tau * delta), tau2 = both<C>(tau);
  const C2 zb = pair(-beta, beta), kap2 = both<C>(kappa);
  constexpr double alpha = ipow(kVal, D);
  C2 cv, gc[3];
  lane_vg<C2, D, true>(pair(un[0], un[1]), rho2, cv, gc);
  C2 sv = fma_q(kap2, cv, lane_v<C2, D>(pair(hn[0], hn[1]), rho2));
  C2 gg = both<C>(gp[0]) * gc[0];
#pragma unroll
  for (int k = 1; k < D; ++k) gg = fma_q(both<C>(gp[k]), gc[k], gg);
  if constexpr (ADV)
#pragma unroll
    for (int k = 0; k < D; ++k) sv = fma_q(both<C>(V[k]), gc[k], sv);
  const C2 R = fma_q(zb, gg, sv);
  C2 S, Phi[3];
  C Sp, Pp[3];
  if constexpr (!JV) {
    const C2 q = times_pm(cv - tau2 * R, alpha), p = taud * R;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      Phi[k] = fma_q(q, both<C>(gp[k]), gc[k]);
      if constexpr (ADV) Phi[k] = fma_q(p, both<C>(V[k]), Phi[k]);
    }
    S = times_const2(sv, kVal * kVal, -2 * lev);
    Sp = times_const(fma_q(tau, first(R) - second(R), second(cv) - first(cv)), kVal * kVal, -2 * lev);
#pragma unroll
    for (int k = 0; k < D; ++k) Pp[k] = e2 * gp[k];
  } else {
    C2 dcv, dgc[3];
    lane_vg<C2, D, true>(pair(dn[0], dn[1]), rho2, dcv, dgc);
    C2 dsv = kap2 * dcv, dgg = both<C>(gp[0]) * dgc[0];
#pragma unroll
    for (int k = 1; k < D; ++k) dgg = fma_q(both<C>(gp[k]), dgc[k], dgg);
#pragma unroll
    for (int k = 0; k < D; ++k) {
      dgg = fma_q(both<C>(dgp[k]), gc[k], dgg);
      if constexpr (ADV) dsv = fma_q(both<C>(V[k]), dgc[k], dsv);
    }
    const C2 dR = fma_q(zb, dgg, dsv);
    const C2 q1 = times_pm(cv - tau2 * R, alpha), q2 = times_pm(dcv - tau2 * dR, alpha), p = taud * dR;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      Phi[k] = fma_q(q2, both<C>(gp[k]), fma_q(q1, both<C>(dgp[k]), dgc[k]));
      if constexpr (ADV) Phi[k] = fma_q(p, both<C>(V[k]), Phi[k]);
    }
    S = times_const2(dsv, kVal * kVal, -2 * lev);
    Sp = times_const(fma_q(tau, first(dR) - second(dR), second(dcv) - first(dcv)), kVal * kVal, -2 * lev);
#pragma unroll
    for (int k = 0; k < D; ++k) Pp[k] = e2 * dgp[k];
  }

  rs = lane_test<C2, D>(S, Phi, rho2);
  rp = lane_test<C, D>(Sp, Pp, rho);
}

}  // namespace
