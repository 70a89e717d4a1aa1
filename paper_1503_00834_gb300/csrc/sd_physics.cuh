// Point physics of the spectral-difference kernels (paper Section 2 Eqs. 5-9, Section 3 Rusanov flux).
//
// Two physics forms share the kernels:
//   PERT = false, R = double : Q is the total conserved state; plain fluxes.
//   PERT = true,  R = float  : Q is q' = Q - Q0 about the polytrope at rest; every nonlinear
//                              term is written as an exact algebraic difference F(Q0+q') - F(Q0)
//                              so that FP32 rounding is relative to the perturbation, and the
//                              FP64 background residual R(Q0) is added at the end.
#pragma once
#include "sd_device.cuh"

namespace chorus {

// ------------------------------------------------------------------ reciprocals

// Reciprocals of the point physics.  FP64: the correctly rounded quotient.  FP32 (the perturbation
// form, whose tolerance is relative 1e-5): the approximate reciprocal (error of one ulp for arguments
// of normal magnitude, one instruction); the quotients of a point share it.
__device__ __forceinline__ double qrcp(double a) { return 1.0 / a; }
__device__ __forceinline__ float qrcp(float a) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}

// ------------------------------------------------------------------ pairs

// Two values worked on together.  FP32: the packed two-lane FMA (fma.rn.f32x2), one issue slot for
// two correctly rounded FMAs; FP64: two FMAs.  The line contractions of the kernels (interpolation,
// derivative) run on pairs of components, which halves the instructions of the kernels' largest part.
template <class R>
struct Pair {
  R x, y;
};
template <class R>
__device__ __forceinline__ Pair<R> mul2(Pair<R> a, Pair<R> b) {
  if constexpr (sizeof(R) == 4) {
    unsigned long long ua, ub, ud;
    asm("mov.b64 %0, {%1, %2};" : "=l"(ua) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(ub) : "f"(b.x), "f"(b.y));
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(ud) : "l"(ua), "l"(ub));
    Pair<R> d;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(ud));
    return d;
  } else {
    return Pair<R>{a.x * b.x, a.y * b.y};
  }
}
template <class R>
__device__ __forceinline__ Pair<R> fma2(Pair<R> a, Pair<R> b, Pair<R> c) {
  if constexpr (sizeof(R) == 4) {
    unsigned long long ua, ub, uc, ud;
    asm("mov.b64 %0, {%1, %2};" : "=l"(ua) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(ub) : "f"(b.x), "f"(b.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(uc) : "f"(c.x), "f"(c.y));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(ud) : "l"(ua), "l"(ub), "l"(uc));
    Pair<R> d;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(ud));
    return d;
  } else {
    return Pair<R>{fma(a.x, b.x, c.x), fma(a.y, b.y, c.y)};
  }
}

// ------------------------------------------------------------------ point physics

template <class R>
struct Pt {
  R rho;    // total density
  R ir;     // 1 / rho
  R u[3];   // velocity
  R p;      // the form's pressure variable (p or p')
  R ptot;   // total pressure
  R Etot;   // total energy
};

template <bool PERT, class R>
__device__ __forceinline__ Pt<R> point_state(const R q[5], R rho0, R E0, const PhysArg<R>& ph) {
  Pt<R> s;
  s.rho = PERT ? rho0 + q[0] : q[0];
  s.ir = qrcp(s.rho);
  s.u[0] = q[1] * s.ir;
  s.u[1] = q[2] * s.ir;
  s.u[2] = q[3] * s.ir;
  const R ke = R(0.5) * (q[1] * s.u[0] + q[2] * s.u[1] + q[3] * s.u[2]);
  s.p = ph.gm1 * (q[4] - ke);
  if (PERT) {
    s.ptot = ph.gm1 * E0 + s.p;
    s.Etot = E0 + q[4];
  } else {
    s.ptot = s.p;
    s.Etot = q[4];
  }
  return s;
}

// s . (F, G, H)_inv (Eq. 6); in the perturbation form the difference from the background.
template <class R>
__device__ __forceinline__ void flux_inv(const R q[5], const Pt<R>& st, const R s[3], R F[5]) {
  F[0] = q[1] * s[0] + q[2] * s[1] + q[3] * s[2];
  const R Vn = F[0] * st.ir;
  F[1] = q[1] * Vn + st.p * s[0];
  F[2] = q[2] * Vn + st.p * s[1];
  F[3] = q[3] * Vn + st.p * s[2];
  F[4] = Vn * (st.Etot + st.ptot);
}

// Gradient record of a point, kG = 11 entries: g[0..2] the form's grad rho, g[3..7] the trace-free
// strain sigma = grad u + grad u^T - 2/3 (div u) I as (xx, yy, xy, yz, zx), zz = -(xx + yy), and
// g[8..10] the form's grad p.  tau = mu sigma (Eq. 9).

// sigma s
template <class R>
__device__ __forceinline__ void strain_dot(const R g[kG], const R s[3], R t[3]) {
  t[0] = g[3] * s[0] + g[5] * s[1] + g[7] * s[2];
  t[1] = g[5] * s[0] + g[4] * s[1] + g[6] * s[2];
  t[2] = g[7] * s[0] + g[6] * s[1] - (g[3] + g[4]) * s[2];
}

template <class R>
__device__ __forceinline__ R dot3(const R a[3], const R b[3]) {
  return a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
}

// s . (F, G, H)_v (Eqs. 7-9; energy entry u.tau - f as in Eq. 3), momentum and energy entries.
// gr0: background density gradient (perturbation form only).  With f = -C_p/R (kappa (grad p / gamma -
// p/rho grad rho) + kappa_r (grad p - p/rho grad rho)) only the three projections s.grad p, s.grad rho
// and s.grad rho0 enter.
template <bool PERT, class R>
__device__ __forceinline__ void flux_visc(const Pt<R>& st, const R q[5], const R g[kG], const R gr0[3], R rho0, R E0,
                                          const R s[3], const PhysArg<R>& ph, R kr, R Fv[4]) {
  const R mu = st.rho * ph.nu;
  R t[3];
  strain_dot(g, s, t);
#pragma unroll
  for (int a = 0; a < 3; ++a) Fv[a] = mu * t[a];
  R A = st.ptot * st.ir * dot3(g, s);  // s . (p/rho grad rho), of the form
  if (PERT) {
    const R T0 = ph.gm1 * E0 * qrcp(rho0);  // p0 / rho0
    A += (st.p - T0 * q[0]) * st.ir * dot3(gr0, s);  // p/rho - p0/rho0 = (p' - p0/rho0 rho') / rho
  }
  const R heat = ph.CpR * ((ph.kappa_g + kr) * dot3(g + 8, s) - (ph.kappa + kr) * A);  // -f . s
  Fv[3] = dot3(st.u, Fv) + heat;
}

// primitive gradient record from conserved gradients gq[3 v + n] = d q_v / d x_n:
//   grad u_a = (grad m_a - u_a grad rho) / rho,  grad p = (gamma-1)(grad E - u.grad m + |u|^2/2 grad rho)
template <bool PERT, class R>
__device__ __forceinline__ void grad_prim(const Pt<R>& st, const R gq[15], const R gr0[3], const PhysArg<R>& ph,
                                          R g[kG]) {
  R grt[3];
#pragma unroll
  for (int n = 0; n < 3; ++n) {
    grt[n] = PERT ? gr0[n] + gq[n] : gq[n];
    g[n] = gq[n];
  }
  R gu[3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int n = 0; n < 3; ++n) gu[a][n] = (gq[3 * (1 + a) + n] - st.u[a] * grt[n]) * st.ir;
  const R div = gu[0][0] + gu[1][1] + gu[2][2];
  g[3] = R(2) * gu[0][0] - R(2.0 / 3.0) * div;
  g[4] = R(2) * gu[1][1] - R(2.0 / 3.0) * div;
  g[5] = gu[0][1] + gu[1][0];
  g[6] = gu[1][2] + gu[2][1];
  g[7] = gu[0][2] + gu[2][0];
  const R ke = R(0.5) * (st.u[0] * st.u[0] + st.u[1] * st.u[1] + st.u[2] * st.u[2]);
#pragma unroll
  for (int n = 0; n < 3; ++n)
    g[8 + n] = ph.gm1 * (gq[12 + n] - (st.u[0] * gq[3 + n] + st.u[1] * gq[6 + n] + st.u[2] * gq[9 + n]) +
                         ke * grt[n]);
}

// |S| times the Rusanov flux along S / |S| from both sides' states: the fluxes projected on the
// (outward) S itself, which needs no unit normal, and the wave speed scaled by |S|.
template <bool PERT, class R>
__device__ __forceinline__ void rusanov(const R qL[5], const Pt<R>& sL, R rho0L, R E0L, const R qR[5],
                                        const Pt<R>& sR, R rho0R, R E0R, const R S[3], R mag, const PhysArg<R>& ph,
                                        R F[5]) {
  R FL[5], FR[5];
  flux_inv(qL, sL, S, FL);
  flux_inv(qR, sR, S, FR);
  const R cL = sqrt(ph.gamma * sL.ptot * sL.ir);
  const R cR = sqrt(ph.gamma * sR.ptot * sR.ir);
  const R vL = fabs(dot3(sL.u, S)) + cL * mag;
  const R vR = fabs(dot3(sR.u, S)) + cR * mag;
  const R lam = vL > vR ? vL : vR;
#pragma unroll
  for (int v = 0; v < 5; ++v) F[v] = R(0.5) * (FL[v] + FR[v]) - R(0.5) * lam * (qR[v] - qL[v]);
  if (PERT) {
    const R c0L = sqrt(ph.gamma * ph.gm1 * E0L * qrcp(rho0L));
    const R c0R = sqrt(ph.gamma * ph.gm1 * E0R * qrcp(rho0R));
    const R lam0 = (c0L > c0R ? c0L : c0R) * mag;
    F[0] -= R(0.5) * (lam - lam0) * (rho0R - rho0L);
    F[4] -= R(0.5) * (lam - lam0) * (E0R - E0L);
  }
}
}  // namespace chorus
