// Pointwise physics of the CNP discontinuous Galerkin operator (Eq. NPDG and Eq.
// chargeDG, Sec. 3.3): velocity, exchange current, volume fluxes, and the
// numerical fluxes on interior and boundary faces with their adjoints, for any
// scalar type (FP64, FP32, double-float, forward tangents).
#pragma once
#include "enp_common.cuh"

namespace enp {

// ----------------------------------------------------------------- physics
// Component i (0..2) of a 3-vector held in registers, selected rather than
// indexed, so that a run-time i keeps the vector out of local memory.
template <class R>
__device__ __forceinline__ R pick3(const R* v, int i) {
  return i == 0 ? v[0] : (i == 1 ? v[1] : v[2]);
}

template <class R>
__device__ __forceinline__ void velocity(const PhysT<R>& p, const R* x, R* uv) {
  if (p.vel_kind == 0) {
    uv[0] = p.vp[0]; uv[1] = p.vp[1]; uv[2] = p.vp[2];
  } else {  // plate flow u_A = 6 u_avg s (H - s) / H^2 (Sec. 5.2)
    const int A = p.velA;
    const R s = pick3(x, p.velN) - p.vp[2], H = p.vp[3];
    const R ua = p.vel_coef * s * (H - s);
    uv[0] = A == 0 ? ua : R(0);
    uv[1] = A == 1 ? ua : R(0);
    uv[2] = A == 2 ? ua : R(0);
  }
}

// J_0 = 3/5 Jbar [2 - ((t - w/2)/(w/2))^2] (Sec. 5.2), or constant.
template <class C, class R>
__device__ __forceinline__ C exchange_current(const PhysT<C>& p, const R* x) {
  if (p.J0axis < 0) return p.J0;
  const C r = (pick3(x, p.J0axis) - p.J0lo - p.J0half) * p.J0inv_half;
  return R(0.6) * p.J0 * (R(2) - r * r);
}

// Volume flux at one point (Eq. NPDG and Eq. chargeDG volume terms): the
// coefficient Sf of phi_i and the vector Gf multiplying grad phi_i.
template <int NF, int DIM, class S, class R, class C = R>
__device__ __forceinline__ void volume_flux(const PhysT<C>& p, const S* c, const S (*g)[3],
                                            const R* uv, S* Sf, S (*Gf)[3]) {
  S kap = S(R(0));
#pragma unroll
  for (int k = 0; k < NF - 1; ++k) kap += p.kcoef[k] * c[k + 1];
#pragma unroll
  for (int d = 0; d < DIM; ++d) {
    S acc = kap * g[0][d];
#pragma unroll
    for (int k = 0; k < NF - 1; ++k) acc += p.acoef[k] * g[k + 1][d];
    Gf[0][d] = acc;
  }
#pragma unroll
  for (int k = 0; k < NF - 1; ++k)
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
      const S qk = uv[d] - p.mig[k] * g[0][d];
      Gf[k + 1][d] = p.D[k] * g[k + 1][d] - c[k + 1] * qk;
    }
#pragma unroll
  for (int f = 0; f < NF; ++f) Sf[f] = S(R(0));
}

// Own-row flux on an interior face (Eq. NPDG / Eq. chargeDG face integrals over
// Gamma_I, tested with this element's basis: [[v]] = phi_i n, {grad v} = grad phi_i / 2).
// cm, dm: values and normal derivatives (along n = this element's outward
// normal) on this side; cp, dp on the other side. Returns the coefficient Sf
// of phi_i and Tf of grad phi_i . n. Upwind reading: {c q}.n + |{q}.n|/2 [[c]].
template <int NF, class S, class R, class C = R>
__device__ __forceinline__ void face_interior_flux(const PhysT<C>& p, const S* cm, const S* dm,
                                                   const S* cp, const S* dp, R un, R delta,
                                                   S* Sf, S* Tf) {
  S kapm = S(R(0)), kapp = S(R(0));
  S T0 = S(R(0)), S0 = S(R(0));
#pragma unroll
  for (int k = 0; k < NF - 1; ++k) {
    const int f = k + 1;
    const C Dk = p.D[k], mg = p.mig[k], ak = p.acoef[k];
    const S jc = cm[f] - cp[f];
    const S qnm = un - mg * dm[0];
    const S qnp = un - mg * dp[0];
    const S qa = R(0.5) * (qnm + qnp);
    Tf[f] = R(-0.5) * Dk * jc;
    Sf[f] = R(-0.5) * Dk * (dm[f] + dp[f]) + (Dk * delta) * jc +
            R(0.5) * (cm[f] * qnm + cp[f] * qnp) + R(0.5) * absv(qa) * jc;
    kapm += p.kcoef[k] * cm[f];
    kapp += p.kcoef[k] * cp[f];
    T0 += R(-0.5) * ak * jc;
    S0 += R(-0.5) * ak * (dm[f] + dp[f]);
  }
  const S jphi = cm[0] - cp[0];
  Tf[0] = T0 + R(-0.5) * kapm * jphi;
  Sf[0] = S0 + R(-0.5) * (kapm * dm[0] + kapp * dp[0]) + (R(0.5) * delta) * (kapm + kapp) * jphi;
}

// Concentration of the Butler-Volmer oxidant (Eq. substitution if it is c_m).
template <int NF, class S, class R, class C = R>
__device__ __forceinline__ S oxidant_conc(const PhysT<C>& p, const S* c) {
  if (p.bv_ox < NF - 1) {  // selected, not indexed: c stays in registers
    S o = c[1];
#pragma unroll
    for (int k = 1; k < NF - 1; ++k)
      if (k == p.bv_ox) o = c[k + 1];
    return o;
  }
  S s = S(R(0));
#pragma unroll
  for (int k = 0; k < NF - 1; ++k) s += p.z[k] * c[k + 1];
  return p.neg_inv_zm * s;
}

// Own-row flux on a boundary face (the boundary integrals of Eq. NPDG and
// Eq. chargeDG; DIRICHLET is the Nitsche form of the interior terms with the
// exterior state g, used for manufactured solutions).
template <int NF, class S, class R, class C = R>
__device__ __forceinline__ void face_boundary_flux(const PhysT<C>& p, int tag, const S* cm,
                                                   const S* dm, const R* g, R un, R delta,
                                                   const R* x, C phiapp, S* Sf, S* Tf) {
#pragma unroll
  for (int f = 0; f < NF; ++f) { Sf[f] = S(R(0)); Tf[f] = S(R(0)); }
  if (tag == kInlet) {
#pragma unroll
    for (int k = 0; k < NF - 1; ++k) Sf[k + 1] = S(un * p.cin[k]);
  } else if (tag == kOutlet) {
#pragma unroll
    for (int k = 0; k < NF - 1; ++k) Sf[k + 1] = (un - p.mig[k] * dm[0]) * cm[k + 1];
  } else if (tag >= kElectrode0) {
    if (p.bv_ox < 0) return;
    const S co = oxidant_conc<NF, S, R, C>(p, cm);
    const S eta = phiapp - cm[0];
    S r = p.inv_cref * co;
    if (valof(p.gam) != R(1)) r = powv(r, valof(p.gam));
    const S Jn = exchange_current(p, x) * (expv(p.e1 * eta) - r * expv((-p.e2) * eta));
#pragma unroll
    for (int k = 0; k < NF - 1; ++k)
      if (k == p.bv_ox) Sf[k + 1] = p.ox_species_scale * Jn;
    Sf[0] = p.ox_charge_scale * Jn;
  } else if (tag == kDirichlet) {
    S kap = S(R(0)), T0 = S(R(0)), S0 = S(R(0));
#pragma unroll
    for (int k = 0; k < NF - 1; ++k) {
      const int f = k + 1;
      const C Dk = p.D[k], ak = p.acoef[k];
      const S jc = cm[f] - g[f];
      const S qn = un - p.mig[k] * dm[0];
      Tf[f] = (-Dk) * jc;
      Sf[f] = (-Dk) * dm[f] + (Dk * delta) * jc + R(0.5) * (cm[f] + g[f]) * qn +
              R(0.5) * absv(qn) * jc;
      kap += p.kcoef[k] * cm[f];
      T0 += (-ak) * jc;
      S0 += (-ak) * dm[f];
    }
    const S jphi = cm[0] - g[0];
    Tf[0] = T0 - kap * jphi;
    Sf[0] = S0 - kap * dm[0] + delta * (kap * jphi);
  }
}

// Adjoint of the linearised boundary own-row flux (this side only).
template <int NF, class R>
__device__ __forceinline__ void face_boundary_adjoint(const PhysT<R>& p, int tag, const R* cm,
                                                      const R* dm, const R* g, R un, R delta,
                                                      const R* x, R phiapp, const R* Sh,
                                                      const R* Th, R* acm, R* adm) {
  if (tag == kOutlet) {
#pragma unroll
    for (int k = 0; k < NF - 1; ++k) {
      const R mg = p.mig[k];
      acm[k + 1] += (un - mg * dm[0]) * Sh[k + 1];
      adm[0] += -mg * cm[k + 1] * Sh[k + 1];
    }
  } else if (tag >= kElectrode0) {
    if (p.bv_ox < 0) return;
    const R co = oxidant_conc<NF, R, R>(p, cm);
    const R eta = phiapp - cm[0];
    const R E1 = expv(p.e1 * eta), E2 = expv((-p.e2) * eta);
    R r = p.inv_cref * co, drdc = p.inv_cref;
    if (valof(p.gam) != R(1)) {
      const R rb = r;
      r = powv(rb, p.gam);
      drdc = p.gam * powv(rb, p.gam1) * p.inv_cref;
    }
    const R J0 = exchange_current(p, x);
    const R dJdphi = J0 * (-p.e1 * E1 - r * p.e2 * E2);
    const R dJdco = -J0 * E2 * drdc;
    R Jh = p.ox_charge_scale * Sh[0];
#pragma unroll
    for (int k = 0; k < NF - 1; ++k)
      if (k == p.bv_ox) Jh += p.ox_species_scale * Sh[k + 1];
    acm[0] += Jh * dJdphi;
    if (p.bv_ox < NF - 1) {
#pragma unroll
      for (int k = 0; k < NF - 1; ++k)
        if (k == p.bv_ox) acm[k + 1] += Jh * dJdco;
    } else {
#pragma unroll
      for (int k = 0; k < NF - 1; ++k) acm[k + 1] += Jh * dJdco * p.zratio[k];
    }
  } else if (tag == kDirichlet) {
    R kap = R(0);
#pragma unroll
    for (int k = 0; k < NF - 1; ++k) kap += p.kcoef[k] * cm[k + 1];
    const R jphi = cm[0] - g[0];
    const R S0 = Sh[0], T0 = Th[0];
#pragma unroll
    for (int k = 0; k < NF - 1; ++k) {
      const int f = k + 1;
      const R Dk = p.D[k], mg = p.mig[k], ak = p.acoef[k], kc = p.kcoef[k];
      const R jc = cm[f] - g[f];
      const R qn = un - mg * dm[0];
      const R sg = qn > R(0) ? R(1) : (qn < R(0) ? R(-1) : R(0));
      acm[f] += -Dk * Th[f] + (Dk * delta + R(0.5) * qn + R(0.5) * absv(qn)) * Sh[f];
      adm[f] += -Dk * Sh[f];
      adm[0] += -mg * (R(0.5) * (cm[f] + g[f]) + R(0.5) * sg * jc) * Sh[f];
      acm[f] += -ak * T0 - kc * jphi * T0 - kc * dm[0] * S0 + delta * kc * jphi * S0;
      adm[f] += -ak * S0;
    }
    acm[0] += -kap * T0 + delta * kap * S0;
    adm[0] += -kap * S0;
  }
}

}  // namespace enp
