// Gas-kinetic flux at one Gauss point (Section 3.2, Eqs. flux-1 and flux-2) in the global frame:
// the unit normal n enters only through projections, so neither the reconstructed values nor
// their gradients are rotated and no tangential axes are formed. With Un = U . n, the half line
// u > 0 (left side) or u < 0 (right side) of the normal velocity, s = +1 or -1, and
//   A0 = <1> = erfc(-s sqrt(lam) Un) / 2,  B = exp(-lam Un^2) / (2 sqrt(pi lam)),
//   A1 = <u> = Un A0 + s B,  theta = p / rho,
// every moment is a vector or tensor expression in q = (rho, m, E), U and n:
//   rho <psi>      = A0 q + rho s B (0, n, Un / 2)
//   rho <u psi>    = A1 q + p (0, A0 n, (A1 + Un A0) / 2)
//   rho <u c>      = rho A1 U + p A0 n
//   rho <u c c^T>  = rho A1 U U^T + p (A0 (U n^T + n U^T) + A1 I + s B n n^T)
//   rho <u c |c|^2/2 (with xi)> = U ((E + 3p/2) A1 + Un p A0 / 2)
//                                 + n theta ((E + p) A0 + Un rho s B / 2)
// (the whole line is A0 = 1, B = 0, A1 = Un). A slope term rho <c_d (a psi) psi> with
// rho <a psi> = dq is the derivative of the moment along dq, and the sums over the axes,
// sum_d D<.. c_d ..>[dq_d], are divergences, formed from U . grad, n . grad and div of the
// conserved variables instead of one moment derivative per axis. Against the face-frame form
// this replaces: 1614 -> 941 flop per Gauss point (smooth, tau = 0), 3668 -> 1794 (full).
#pragma once

#include <type_traits>

#include "gks_kinetic.cuh"

namespace gks {

// One side of the interface: primitives and the half-line moments of its Maxwellian.
template <class R>
struct Side {
  Prim<R> w;
  R Un, A, sB, be, u2h;  // be = rho s B, u2h = |U|^2 / 2
};
// Derivatives of a side's normal velocity, pressure, A0 and s B along a conserved increment.
// (t: dsB = -s B t).
template <class R>
struct SideD {
  R dUn, dp, dA, dsB, t;
};

template <class R>
GKS_HD R dot3(const R a[3], const R b[3]) {
  return a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
}
template <class R>
GKS_HD R dotU(const Prim<R>& w, R x, R y, R z) {
  return w.U * x + w.V * y + w.W * z;
}

// s is an int, or a packed pair of signs when R carries both sides.
template <class R, class Sg>
GKS_HD void side_init(const double*, const R n[3], Sg s, Side<R>& h) {
  const Prim<R>& w = h.w;
  h.Un = dotU(w, n[0], n[1], n[2]);
  h.u2h = R(0.5) * dotU(w, w.U, w.V, w.W);
  const R sl = k_sqrt(w.lam);
  const R x = sl * h.Un;
  h.A = R(0.5) * k_erfc(-R(s) * x);
  h.sB = R(s) * k_div(R(0.28209479177387814) * k_exp(-x * x), sl);  // 1/(2 sqrt(pi))
  h.be = w.rho * h.sB;
}
GKS_HD void side_init(const double* tab, const double n[3], int s, Side<double>& h) {
  const Prim<double>& w = h.w;
  h.Un = dotU(w, n[0], n[1], n[2]);
  h.u2h = 0.5 * dotU(w, w.U, w.V, w.W);
#ifdef __CUDA_ARCH__
  const double rs = rsqrt(w.lam);
#else
  const double rs = 1.0 / sqrt(w.lam);
#endif
  const double x = w.lam * rs * h.Un;
  double d;
  if (!half_erfc(tab, -s * x, h.A, d)) {
    h.A = 0.5 * erfc(-s * x);
    d = -0.56418958354775629 * exp(-x * x);  // 1/sqrt(pi)
  }
  h.sB = -0.5 * s * d * rs;
  h.be = w.rho * h.sB;
}
// dA0 = s B z and d(s B) = -s B (Un z + dlam / (2 lam)), z = 2 lam dUn + Un dlam.
template <class R>
GKS_HD void side_der(const Side<R>& h, R gm1, const R n[3], R d0, R d1, R d2, R d3, R d4,
                     SideD<R>& o) {
  const Prim<R>& w = h.w;
  o.dUn = (n[0] * d1 + n[1] * d2 + n[2] * d3 - h.Un * d0) * w.ir;
  o.dp = gm1 * (d4 - dotU(w, d1, d2, d3) + h.u2h * d0);
  // FP64: with half of dlam / lam and the side's own factors on the right of each product, four
  // instructions fewer per axis (1.441 -> 1.390 ms per launch, smooth form, with the sums of
  // k_flux); FP32 holds the extra factors worse than it saves (302 against 304 us)
  if constexpr (std::is_same<R, double>::value) {
    const R hd = d0 * (R(0.5) * w.ir) - o.dp * (R(0.5) * w.ip);
    const R l2 = R(2) * w.lam;
    const R z = o.dUn * l2 + hd * (l2 * h.Un);
    o.dA = h.sB * z;
    o.t = h.Un * z + hd;
  } else {
    const R dll = d0 * w.ir - o.dp * w.ip;  // dlam / lam
    const R z = w.lam * (R(2) * o.dUn + h.Un * dll);
    o.dA = h.sB * z;
    o.t = h.Un * z + R(0.5) * dll;
  }
  o.dsB = -h.sB * o.t;
}
// Derivative of be = rho s B along the same increment.
template <class R>
GKS_HD R be_der(const Side<R>& h, const SideD<R>& e, R d0) {
  if constexpr (std::is_same<R, double>::value) return h.sB * d0 - h.be * e.t;
  return h.sB * d0 + h.w.rho * e.dsB;
}

// U . grad and div terms of a state whose gradient is g[v][axis] and pressure gradient dp.
template <class R>
struct Advect {
  R G[5], H[3];  // G = U . grad q, H_a = rho U . grad U_a
  R divm, divU, Gp;
};
template <class R>
GKS_HD void advect(const Prim<R>& w, const R g[5][3], const R dp[3], Advect<R>& a) {
#pragma unroll
  for (int v = 0; v < 5; ++v) a.G[v] = dotU(w, g[v][0], g[v][1], g[v][2]);
  a.H[0] = a.G[1] - w.U * a.G[0];
  a.H[1] = a.G[2] - w.V * a.G[0];
  a.H[2] = a.G[3] - w.W * a.G[0];
  a.divm = g[1][0] + g[2][1] + g[3][2];
  a.divU = (a.divm - a.G[0]) * w.ir;
  a.Gp = dotU(w, dp[0], dp[1], dp[2]);
}
// rho <A psi> = -sum_d A_d(W) dq_d, the Euler time derivative of the state (Ep = E + p).
template <class R>
GKS_HD void time_slope(const Prim<R>& w, R Ep, const Advect<R>& a, const R dp[3], R t[5]) {
  t[0] = -a.divm;
  t[1] = -(w.U * a.divm + a.H[0] + dp[0]);
  t[2] = -(w.V * a.divm + a.H[1] + dp[1]);
  t[3] = -(w.W * a.divm + a.H[2] + dp[2]);
  t[4] = -(Ep * a.divU + a.G[4] + a.Gp);
}

// One side's part of the interface state q0 and of its gradient dW[v][axis], and for the full
// form the non-equilibrium terms N[0] = F+(W), N[1] = sum_d D<u c_d psi>[dq_d],
// N[2] = DF+[rho <A psi>]; kAdd adds them to the other side's. The caller formed h.w from q
// (to_prim).
template <bool kAdd, class R>
GKS_HD void put(R& x, const R& y) {
  if (kAdd)
    x += y;
  else
    x = y;
}
template <bool kAdd, class R, class Sg>
GKS_HD void side_terms(bool full, const double* tab, R gm1, const R q[5], const R g[5][3],
                       const R n[3], Sg s, Side<R>& h, R q0[5], R dW[5][3], R N[3][5]) {
  const Prim<R>& w = h.w;
  side_init(tab, n, s, h);
  const R hU = R(0.5) * h.Un, hb = R(0.5) * h.be;
  // sums start from the other side's value, so that adding it costs nothing
  auto first = [](const R& x, const R& a, const R& b) -> R {
    return kAdd ? R(x + a * b) : R(a * b);
  };
  q0[0] = first(q0[0], h.A, q[0]);
#pragma unroll
  for (int a = 0; a < 3; ++a) q0[1 + a] = first(q0[1 + a], h.A, q[1 + a]) + h.be * n[a];
  q0[4] = first(q0[4], h.A, q[4]) + hU * h.be;
  const R U[3] = {w.U, w.V, w.W};
  R dp[3], dA1[3];  // full form only
  R UA, UsB, nA, nsB, nUn;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    SideD<R> e;
    side_der(h, gm1, n, g[0][d], g[1][d], g[2][d], g[3][d], g[4][d], e);
    const R dbe = be_der(h, e, g[0][d]);
    dW[0][d] = first(dW[0][d], e.dA, q[0]) + h.A * g[0][d];
#pragma unroll
    for (int a = 0; a < 3; ++a)
      dW[1 + a][d] = first(dW[1 + a][d], e.dA, q[1 + a]) + h.A * g[1 + a][d] + dbe * n[a];
    dW[4][d] = first(dW[4][d], e.dA, q[4]) + h.A * g[4][d] + hU * dbe + hb * e.dUn;
    if (full) {
      dp[d] = e.dp;
      dA1[d] = e.dUn * h.A + h.Un * e.dA + e.dsB;
      UA = d == 0 ? R(U[d] * e.dA) : R(UA + U[d] * e.dA);
      UsB = d == 0 ? R(U[d] * e.dsB) : R(UsB + U[d] * e.dsB);
      nA = d == 0 ? R(n[d] * e.dA) : R(nA + n[d] * e.dA);
      nsB = d == 0 ? R(n[d] * e.dsB) : R(nsB + n[d] * e.dsB);
      nUn = d == 0 ? R(n[d] * e.dUn) : R(nUn + n[d] * e.dUn);
    }
  }
  if (!full) return;
  const R A = h.A, A1 = h.Un * h.A + h.sB, E = q[4], p = w.p;
  const R F4 = R(0.5) * (A1 + h.Un * A);
  N[0][0] = first(N[0][0], A1, q[0]);
#pragma unroll
  for (int a = 0; a < 3; ++a) N[0][1 + a] = first(N[0][1 + a], A1, q[1 + a]) + (p * A) * n[a];
  N[0][4] = first(N[0][4], A1, E) + p * F4;
  Advect<R> c;
  advect(w, g, dp, c);
  {
    R Nn[5];  // n . grad q
#pragma unroll
    for (int v = 0; v < 5; ++v) Nn[v] = n[0] * g[v][0] + n[1] * g[v][1] + n[2] * g[v][2];
    const R Np = dot3(n, dp);
    const R UUn = dot3(n, c.H) * w.ir;              // U . grad Un
    const R UA1 = UUn * A + h.Un * UA + UsB;        // U . grad A1
    const R pn = A * Np + p * nA;                   // n . grad (p A0)
    // div (p A0 U) + n . grad (p s B)
    const R pd = p * (A * c.divU + UA) + A * c.Gp + h.sB * Np + p * nsB;
    const R N10 = A1 * c.divm + w.rho * UA1 + pn;
    put<kAdd>(N[1][0], N10);
    const R Ah = A * w.hil;
#pragma unroll
    for (int j = 0; j < 3; ++j)
      N[1][1 + j] = first(N[1][1 + j], U[j], N10) + A1 * (c.H[j] + dp[j]) +
                    Ah * (Nn[1 + j] - U[j] * Nn[0]) + n[j] * pd + p * dA1[j];
    const R E3 = E + R(1.5) * p, Ep = E + p;
    const R X = E3 * A1 + (p * A) * hU;
    const R Y = Ep * A + hU * h.be;
    const R nbe = h.sB * Nn[0] + w.rho * nsB;
    N[1][4] = first(N[1][4], X, c.divU) + (c.G[4] + R(1.5) * c.Gp) * A1 + E3 * UA1 +
              R(0.5) * (p * (UUn * A + h.Un * UA) + h.Un * A * c.Gp) +
              (Np - w.hil * Nn[0]) * w.ir * Y +
              w.hil * ((Nn[4] + Np) * A + Ep * nA + R(0.5) * (nUn * h.be + h.Un * nbe));
  }
  R t[5];
  time_slope(w, R(E + p), c, dp, t);
  SideD<R> e;
  side_der(h, gm1, n, t[0], t[1], t[2], t[3], t[4], e);
  const R x = e.dUn * A + h.Un * e.dA, y = x + e.dsB;  // d(Un A0), dA1
  const R z = A * e.dp + p * e.dA;                     // d(p A0)
  N[2][0] = first(N[2][0], y, q[0]) + A1 * t[0];
#pragma unroll
  for (int a = 0; a < 3; ++a)
    N[2][1 + a] = first(N[2][1 + a], y, q[1 + a]) + A1 * t[1 + a] + z * n[a];
  N[2][4] = first(N[2][4], y, E) + A1 * t[4] + e.dp * F4 + R(0.5) * p * (x + y);
}

// The non-equilibrium terms enter for the full form with a collision time only (tau = 0 leaves
// the equilibrium flux of the smooth form).
template <class R>
GKS_HD bool full_terms(const FluxParams<R>& P) {
  return P.full && P.tau_model != 0;
}

// exp(-dt / (2 tau)), 0 for tau = 0.
template <class R>
GKS_HD R relaxation(R dt, R tau) {
  return tau > R(0) ? k_exp(k_div(R(-0.5) * dt, tau)) : R(0);
}

// The two-point time fit of the full form (Eq. flux-1). With e = exp(-dt / (2 tau)) the fitted
// weights of the six time integrals, F^n = (4 F(dt/2) - F(dt)) / dt and
// dF/dt = 4 (F(dt) - 2 F(dt/2)) / dt^2, reduce to
//   F^n   = E0 - tau (E1 + E2) + n0 (N0 - E0) + n1 (N1 - E1) + n2 (N2 - E2)
//   dF/dt = E2                 + t0 (N0 - E0) + t1 (N1 - E1) + t2 (N2 - E2),
// the smooth form plus the departure from equilibrium: one exponential instead of two, and no
// difference of nearly equal integrals (FP32 dF/dt of 20,000 random points, tau_eps 0.01:
// 3.7e-6 rms of its largest component against 4.0e-6, largest 1.2e-4 against 2.4e-4).
template <class R>
struct FitWeights {
  R n[3], t[3];
};
template <class R>
GKS_HD void fit_weights(R tau, R dt, R idt0, FitWeights<R>& f) {
  const R e = relaxation(dt, tau);
  const R x = R(1) - e, s = x * x, m = x * (R(2) + x);
  const R idt = idt0 != R(0) ? idt0 : R(k_div(R(1), dt)), a = tau * idt, b = R(4) * a * idt;
  f.n[0] = a * m;
  f.t[0] = -b * s;
  f.n[2] = -tau * f.n[0];
  f.t[2] = -tau * f.t[0];
  f.n[1] = tau * (R(1) - s - R(2) * a * m);
  f.t[1] = b * (R(2) * a * s - e * x) * dt;
}

// F^n and dF/dt of the two-point time fit from the interface state q0, its gradient dW, the two
// sides' summed non-equilibrium terms N (full form) and pressures; w the primitives of q0.
template <class R>
GKS_HD void interface_flux(const FluxParams<R>& P, const Prim<R>& w, const R q0[5],
                           const R dW[5][3], const R N[3][5], R pl, R pr, const R n[3], R dt,
                           R Fn[5], R Ft[5]) {
  const R gm1 = P.gamma - R(1), E = q0[4], p = w.p, Ep = E + p;
  const R U[3] = {w.U, w.V, w.W};
  const R Un = dotU(w, n[0], n[1], n[2]);
  const R u2h = R(0.5) * dotU(w, w.U, w.V, w.W);
  R dp[3];
#pragma unroll
  for (int d = 0; d < 3; ++d)
    dp[d] = gm1 * (dW[4][d] - dotU(w, dW[1][d], dW[2][d], dW[3][d]) + u2h * dW[0][d]);
  Advect<R> c;
  advect(w, dW, dp, c);
  R t[5], E1[5], E2[5];  // t = rho0 <Ab psi>_0
  time_slope(w, Ep, c, dp, t);
  // E2 = rho0 <u Ab psi>_0, the Euler flux Jacobian along n applied to t
  {
    const R dmn = n[0] * t[1] + n[1] * t[2] + n[2] * t[3];
    const R r = dmn - Un * t[0];
    const R dpt = gm1 * (t[4] - dotU(w, t[1], t[2], t[3]) + u2h * t[0]);
    E2[0] = dmn;
#pragma unroll
    for (int a = 0; a < 3; ++a) E2[1 + a] = U[a] * r + Un * t[1 + a] + dpt * n[a];
    E2[4] = r * w.ir * Ep + Un * (t[4] + dpt);
  }
  const R x = k_abs(k_div(pl - pr, pl + pr));
  const R tau = collision_time(P, p, w.ip, w.ir, x, dt);
  // E1 = rho0 <u (ab . c) psi>_0; multiplied by tau, so zero without a collision-time model
  if (P.tau_model != 0) {
    R Nn[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) Nn[v] = dot3(n, dW[v]);
    const R Np = dot3(n, dp), nH = dot3(n, c.H);
    const R pd = p * c.divU + c.Gp;  // div (p U)
    E1[0] = Un * c.divm + nH + Np;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      // rho (n . grad U_j + d_j Un)
      const R r = Nn[1 + j] - U[j] * Nn[0] +
                  (n[0] * dW[1][j] + n[1] * dW[2][j] + n[2] * dW[3][j] - Un * dW[0][j]);
      E1[1 + j] = U[j] * E1[0] + Un * (c.H[j] + dp[j]) + w.hil * r + n[j] * pd;
    }
    E1[4] = (Ep + p) * (Un * c.divU + nH * w.ir) + Un * (c.G[4] + R(2) * c.Gp) +
            w.hil * (Nn[4] + Np) + Ep * ((Np - w.hil * Nn[0]) * w.ir);
  } else {
#pragma unroll
    for (int q = 0; q < 5; ++q) E1[q] = R(0);
  }
  const R mn = w.rho * Un;
  const R E0[5] = {mn, mn * U[0] + p * n[0], mn * U[1] + p * n[1], mn * U[2] + p * n[2], Un * Ep};
  // smooth form (Eq. flux-2): F(delta) = E0 delta - tau delta (E1 + E2) + delta^2/2 E2, so the
  // two-point fit is exact
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    Fn[q] = E0[q] - tau * (E1[q] + E2[q]);
    Ft[q] = E2[q];
  }
  if (full_terms(P)) {
    FitWeights<R> f;
    fit_weights(tau, dt, P.idt, f);
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      const R d0 = N[0][q] - E0[q], d1 = N[1][q] - E1[q], d2 = N[2][q] - E2[q];
      Fn[q] += f.n[0] * d0 + f.n[1] * d1 + f.n[2] * d2;
      Ft[q] += f.t[0] * d0 + f.t[1] * d1 + f.t[2] * d2;
    }
    return;
  }
  if (P.pr_fix != R(0)) {
    // the energy components gain pr_fix times the heat flux relative to the interface velocity,
    // from the flux moments F and the conserved moments m of the time-integrated distribution
    // (m^n = q0, dm/dt = t; the tau terms of m vanish by the compatibility condition)
    auto heat = [&](const R F[5], const R m[5]) {
      return F[4] - dotU(w, F[1], F[2], F[3]) + u2h * F[0] -
             Un * (m[4] - dotU(w, m[1], m[2], m[3]) + u2h * m[0]);
    };
    const R qn = heat(Fn, q0);
    const R qt = heat(Ft, t);
    Fn[4] += P.pr_fix * qn;
    Ft[4] += P.pr_fix * qt;
  }
}

// Whole Gauss-point contribution: values and gradients [v][axis] of both sides, unit normal n
// out of the left side and quadrature weight w: acc[0..4] = w F^n, acc[5..9] = w dF/dt. Returns
// false for a non-physical side or interface state.
template <class R>
GKS_HD bool gp_flux_global(const FluxParams<R>& P, const R vl[5], const R gl[5][3], const R vr[5],
                           const R gr[5][3], const R n[3], R w, R dt, R acc[10]) {
  Side<R> hl, hr;
  if (!(to_prim(vl, P.gamma, hl.w) & to_prim(vr, P.gamma, hr.w))) return false;
  const R gm1 = P.gamma - R(1);
  const bool full = full_terms(P);
  R q0[5], dW[5][3], N[3][5];
  side_terms<false>(full, P.erfc_tab, gm1, vl, gl, n, +1, hl, q0, dW, N);
  side_terms<true>(full, P.erfc_tab, gm1, vr, gr, n, -1, hr, q0, dW, N);
  Prim<R> w0;
  if (!to_prim(q0, P.gamma, w0)) return false;
  R Fn[5], Ft[5];
  interface_flux(P, w0, q0, dW, N, hl.w.p, hr.w.p, n, dt, Fn, Ft);
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    acc[q] = w * Fn[q];
    acc[5 + q] = w * Ft[q];
  }
  return true;
}

}  // namespace gks
