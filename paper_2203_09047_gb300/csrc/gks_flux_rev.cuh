// Vector-Jacobian product of the Gauss-point flux of gks_flux.cuh: its statements reversed by
// hand, in reverse order. The forward is recomputed with its own helpers (no tape): both sides
// and the interface once, then one reverse pass of the interface and one of each side. Every
// slope term is a divergence of a closed form, so its reverse is a handful of products per
// gradient component. Against the reverse in the face frame this replaces, which ran the
// reverse of each moment function in dual numbers along each axis: about 11 -> 3 kflop per
// Gauss point (smooth form).
#pragma once

#include "gks_flux.cuh"

namespace gks {

// Cotangents of a state's primitives and of the functions of it that the forward keeps.
struct StateG {
  double rho = 0, U[3] = {0, 0, 0}, p = 0, E = 0;
  double ir = 0, ip = 0, lam = 0, hil = 0, Un = 0, u2h = 0;
};
// Folds them into the cotangent of the conserved state (accumulated): Un = U . n,
// u2h = |U|^2 / 2, hil = p / rho, lam = rho / (2 p), ir = 1 / rho, ip = 1 / p, U = m / rho,
// p = (gamma - 1) (E - |m|^2 / (2 rho)).
GKS_HD void state_rev(const Prim<double>& w, double u2h, double gm1, const double n[3], StateG& s,
                      double gq[5]) {
  const double U[3] = {w.U, w.V, w.W};
#pragma unroll
  for (int a = 0; a < 3; ++a) s.U[a] += s.Un * n[a] + s.u2h * U[a];
  s.p += s.hil * w.ir - w.ip * (s.ip * w.ip + s.lam * w.lam);
  s.ir += s.hil * w.p;
  const double gp = gm1 * s.p;
  const double gr = s.rho + 0.5 * s.lam * w.ip - s.ir * w.ir * w.ir;
  gq[0] += gr + gp * u2h - w.ir * dot3(s.U, U);
#pragma unroll
  for (int a = 0; a < 3; ++a) gq[1 + a] += s.U[a] * w.ir - gp * U[a];
  gq[4] += s.E + gp;
}

// Cotangents of Advect, accumulated by the reverses of its users.
struct AdvectG {
  double G4 = 0, H[3] = {0, 0, 0}, divm = 0, divU = 0, Gp = 0;
};
// Reverse of time_slope: cotangent gt of t.
GKS_HD void time_slope_rev(const Prim<double>& w, double Ep, const Advect<double>& a,
                           const double gt[5], StateG& s, AdvectG& g, double gdp[3]) {
  g.divm -= gt[0] + dotU(w, gt[1], gt[2], gt[3]);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    s.U[j] -= gt[1 + j] * a.divm;
    g.H[j] -= gt[1 + j];
    gdp[j] -= gt[1 + j];
  }
  const double gEp = gt[4] * a.divU;
  s.E -= gEp;
  s.p -= gEp;
  g.divU -= gt[4] * Ep;
  g.G4 -= gt[4];
  g.Gp -= gt[4];
}
// Reverse of advect and of n . grad q (cotangents gNn): into gg[v][axis], the velocity and gdp.
GKS_HD void advect_rev(const Prim<double>& w, const double q[5][3], const double dp[3],
                       const Advect<double>& a, const AdvectG& g, const double n[3],
                       const double gNn[5], StateG& s, double gdp[3], double gg[5][3]) {
  const double U[3] = {w.U, w.V, w.W};
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    s.U[d] += g.Gp * dp[d];
    gdp[d] += g.Gp * U[d];
  }
  const double r = g.divU * w.ir;
  s.ir += g.divU * (a.divm - a.G[0]);
  double gG[5];
  gG[0] = -r - dotU(w, g.H[0], g.H[1], g.H[2]);
  gG[4] = g.G4;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    gG[1 + d] = g.H[d];
    s.U[d] -= g.H[d] * a.G[0];
  }
#pragma unroll
  for (int v = 0; v < 5; ++v)
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      s.U[d] += gG[v] * q[v][d];
      gg[v][d] += gG[v] * U[d] + gNn[v] * n[d];
    }
  const double gm = g.divm + r;
#pragma unroll
  for (int d = 0; d < 3; ++d) gg[1 + d][d] += gm;
}
// Reverse of dp = (gamma - 1) (d4 - U . (d1, d2, d3) + |U|^2 d0 / 2).
GKS_HD void dp_rev(const Prim<double>& w, double u2h, double gm1, double gdp, double d0, double d1,
                   double d2, double d3, StateG& s, double& g0, double& g1, double& g2,
                   double& g3, double& g4) {
  const double x = gm1 * gdp;
  g4 += x;
  g1 -= x * w.U;
  g2 -= x * w.V;
  g3 -= x * w.W;
  g0 += x * u2h;
  s.U[0] -= x * d1;
  s.U[1] -= x * d2;
  s.U[2] -= x * d3;
  s.u2h += x * d0;
}
// Reverse of side_der: cotangents of (dUn, dp, dA, dsB) -> those of the increment and of the
// side (gsB: of s B).
GKS_HD void side_der_rev(const Side<double>& h, double gm1, const double n[3], double d0,
                         double d1, double d2, double d3, const SideD<double>& e,
                         double gdUn, double gdp, double gdA, double gdsB, StateG& s, double& gsB,
                         double& g0, double& g1, double& g2, double& g3, double& g4) {
  const Prim<double>& w = h.w;
  const double dll = d0 * w.ir - e.dp * w.ip;
  const double y = 2.0 * e.dUn + h.Un * dll, z = w.lam * y;
  gsB += gdA * z - gdsB * (h.Un * z + 0.5 * dll);
  const double gz = h.sB * (gdA - h.Un * gdsB);
  s.Un -= h.sB * z * gdsB;
  s.lam += gz * y;
  const double lz = w.lam * gz;
  gdUn += 2.0 * lz;
  const double gdll = lz * h.Un - 0.5 * h.sB * gdsB;
  s.Un += lz * dll;
  s.ir += gdll * d0;
  s.ip -= gdll * e.dp;
  gdp -= gdll * w.ip;
  const double u = gdUn * w.ir;
  g0 += gdll * w.ir - u * h.Un;
  g1 += u * n[0];
  g2 += u * n[1];
  g3 += u * n[2];
  s.Un -= u * d0;
  s.ir += gdUn * e.dUn * w.rho;
  dp_rev(w, h.u2h, gm1, gdp, d0, d1, d2, d3, s, g0, g1, g2, g3, g4);
}

// Reverse of side_terms: cotangents gq0, gdW, gN (full form) and gp (of the side's pressure) ->
// gq, gg (accumulated). h holds the side of the forward pass.
GKS_HD void side_terms_rev(bool full, double gm1, const double q[5], const double g[5][3],
                           const double n[3], const Side<double>& h, const double gq0[5],
                           const double gdW[5][3], const double gN[3][5], double gp, double gq[5],
                           double gg[5][3]) {
  const Prim<double>& w = h.w;
  const double U[3] = {w.U, w.V, w.W};
  const double A = h.A, sB = h.sB, be = h.be, hU = 0.5 * h.Un;
  SideD<double> e[3];
#pragma unroll
  for (int d = 0; d < 3; ++d)
    side_der(h, gm1, n, g[0][d], g[1][d], g[2][d], g[3][d], g[4][d], e[d]);
  StateG s;
  s.p = gp;
  double gA = 0, gsB = 0, gbe = 0;
  double gdp[3] = {0, 0, 0}, gdA1[3] = {0, 0, 0};
  double gUA = 0, gUsB = 0, gnA = 0, gnsB = 0, gnUn = 0;
  if (full) {
    const double p = w.p, E = q[4], Ep = E + p, A1 = h.Un * A + sB;
    const double F4 = 0.5 * (A1 + h.Un * A);
    const double dp[3] = {e[0].dp, e[1].dp, e[2].dp};
    double dA1[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) dA1[d] = e[d].dUn * A + h.Un * e[d].dA + e[d].dsB;
    const double UA = U[0] * e[0].dA + U[1] * e[1].dA + U[2] * e[2].dA;
    const double UsB = U[0] * e[0].dsB + U[1] * e[1].dsB + U[2] * e[2].dsB;
    const double nA = n[0] * e[0].dA + n[1] * e[1].dA + n[2] * e[2].dA;
    const double nsB = n[0] * e[0].dsB + n[1] * e[1].dsB + n[2] * e[2].dsB;
    const double nUn = n[0] * e[0].dUn + n[1] * e[1].dUn + n[2] * e[2].dUn;
    Advect<double> c;
    advect(w, g, dp, c);
    AdvectG ga;
    double gA1 = 0, gF4 = 0;
    // N[0] = A1 q + p (0, A0 n, F4)
    {
      const double* y = gN[0];
      const double m = n[0] * y[1] + n[1] * y[2] + n[2] * y[3];
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        gA1 += y[v] * q[v];
        gq[v] += A1 * y[v];
      }
      s.p += A * m + F4 * y[4];
      gA += p * m;
      gF4 += p * y[4];
    }
    // N[2] = DF+[t]
    {
      const double* y = gN[2];
      double t[5], gt[5];
      time_slope(w, Ep, c, dp, t);
      SideD<double> f;
      side_der(h, gm1, n, t[0], t[1], t[2], t[3], t[4], f);
      const double x1 = f.dUn * A + h.Un * f.dA, y1 = x1 + f.dsB;
      const double h4 = 0.5 * p * y[4];
      double gy = h4;
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        gy += y[v] * q[v];
        gq[v] += y1 * y[v];
        gA1 += y[v] * t[v];
        gt[v] = A1 * y[v];
      }
      const double gz = n[0] * y[1] + n[1] * y[2] + n[2] * y[3], gx = h4 + gy;
      gF4 += y[4] * f.dp;
      s.p += 0.5 * (x1 + y1) * y[4] + f.dA * gz;
      gA += gx * f.dUn + gz * f.dp;
      s.Un += gx * f.dA;
      side_der_rev(h, gm1, n, t[0], t[1], t[2], t[3], f, gx * A, y[4] * F4 + A * gz,
                   gx * h.Un + gz * p, gy, s, gsB, gt[0], gt[1], gt[2], gt[3], gt[4]);
      time_slope_rev(w, Ep, c, gt, s, ga, gdp);
    }
    // N[1]
    {
      const double* y = gN[1];
      double Nn[5], gNn[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) Nn[v] = dot3(n, g[v]);
      const double Np = dot3(n, dp), nH = dot3(n, c.H), UUn = nH * w.ir;
      const double UA1 = UUn * A + h.Un * UA + UsB;
      const double N10 = A1 * c.divm + w.rho * UA1 + A * Np + p * nA;
      const double E3 = E + 1.5 * p, X = E3 * A1 + (p * A) * hU, Y = Ep * A + hU * be;
      const double nbe = sB * Nn[0] + w.rho * nsB;
      const double y4 = y[4];
      double gUUn, gUA1, gNp, gEp = 0, ghU = 0;
      ga.divU += y4 * X;
      ga.G4 += y4 * A1;
      ga.Gp += y4 * (1.5 * A1 + hU * A);
      gA1 += y4 * (c.G[4] + 1.5 * c.Gp);
      const double gX = y4 * c.divU;
      const double gE3 = y4 * UA1 + gX * A1;
      gUA1 = y4 * E3;
      const double hy = 0.5 * y4;
      s.p += hy * (UUn * A + h.Un * UA);
      gUUn = hy * p * A;
      gA += hy * (p * UUn + h.Un * c.Gp);
      s.Un += hy * (p * UA + A * c.Gp);
      gUA += hy * p * h.Un;
      const double nth = Np - w.hil * Nn[0], k = y4 * w.ir;
      gNp = k * Y;
      s.hil -= gNp * Nn[0];
      gNn[0] = -gNp * w.hil;
      s.ir += y4 * nth * Y;
      const double gY = k * nth;
      const double Lx = (Nn[4] + Np) * A + Ep * nA + 0.5 * (nUn * be + h.Un * nbe);
      const double gL = y4 * w.hil;
      s.hil += y4 * Lx;
      gNn[4] = gL * A;
      gNp += gL * A;
      gA += gL * (Nn[4] + Np) + gY * Ep + gX * p * hU;
      gEp += gL * nA + gY * A;
      gnA += gL * Ep;
      gnUn += 0.5 * gL * be;
      gbe += 0.5 * gL * nUn + gY * hU;
      s.Un += 0.5 * gL * nbe;
      const double gnbe = gL * hU;
      gsB += gnbe * Nn[0];
      gNn[0] += gnbe * sB;
      s.rho += gnbe * nsB;
      gnsB += gnbe * w.rho;
      ghU += gY * be + gX * p * A;
      gA1 += gX * E3;
      s.p += gX * A * hU + 1.5 * gE3 + gEp;
      s.E += gE3 + gEp;
      s.Un += 0.5 * ghU;
      double g0 = y[0], gAh = 0, gpd = 0;
      const double Ah = A * w.hil;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const double yj = y[1 + j], m = Ah * yj;
        g0 += U[j] * yj;
        s.U[j] += yj * N10 - m * Nn[0];
        gA1 += yj * (c.H[j] + dp[j]);
        ga.H[j] += A1 * yj;
        gdp[j] += A1 * yj;
        gAh += yj * (Nn[1 + j] - U[j] * Nn[0]);
        gNn[1 + j] = m;
        gNn[0] -= m * U[j];
        gpd += yj * n[j];
        s.p += yj * dA1[j];
        gdA1[j] = p * yj;
      }
      s.hil += gAh * A;
      gA1 += g0 * c.divm;
      ga.divm += g0 * A1;
      s.rho += g0 * UA1;
      gUA1 += g0 * w.rho;
      gNp += g0 * A + gpd * sB;
      s.p += g0 * nA + gpd * (A * c.divU + UA + nsB);
      gnA += g0 * p;
      gA += gAh * w.hil + g0 * Np + gpd * (p * c.divU + c.Gp) + gUA1 * UUn;
      ga.divU += gpd * p * A;
      gUA += gpd * p + gUA1 * h.Un;
      ga.Gp += gpd * A;
      gsB += gpd * Np;
      gnsB += gpd * p;
      gUUn += gUA1 * A;
      s.Un += gUA1 * UA;
      gUsB += gUA1;
      s.ir += gUUn * nH;
      const double u = gUUn * w.ir;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        ga.H[j] += u * n[j];
        gdp[j] += gNp * n[j];
      }
      advect_rev(w, g, dp, c, ga, n, gNn, s, gdp, gg);
    }
    // F4 = (A1 + Un A0) / 2, A1 = Un A0 + s B
    gA1 += 0.5 * gF4;
    const double gUA0 = gA1 + 0.5 * gF4;
    s.Un += gUA0 * A;
    gA += gUA0 * h.Un;
    gsB += gA1;
  }
  // dW per axis and the sums over the axes
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const double dbe = sB * g[0][d] + w.rho * e[d].dsB;
    double gdA = 0;
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      gdA += gdW[v][d] * q[v];
      gq[v] += gdW[v][d] * e[d].dA;
      gA += gdW[v][d] * g[v][d];
      gg[v][d] += A * gdW[v][d];
    }
    const double y4 = gdW[4][d];
    const double gdbe = n[0] * gdW[1][d] + n[1] * gdW[2][d] + n[2] * gdW[3][d] + hU * y4;
    s.Un += 0.5 * dbe * y4;
    gbe += 0.5 * e[d].dUn * y4;
    gsB += g[0][d] * gdbe;
    gg[0][d] += sB * gdbe;
    s.rho += e[d].dsB * gdbe;
    double gdUn = 0.5 * be * y4, gdsB = w.rho * gdbe, gdpd = 0;
    if (full) {
      const double x = gdA1[d];
      gA += x * e[d].dUn;
      s.Un += x * e[d].dA;
      s.U[d] += gUA * e[d].dA + gUsB * e[d].dsB;
      gdUn += x * A + gnUn * n[d];
      gdA += x * h.Un + gUA * U[d] + gnA * n[d];
      gdsB += x + gUsB * U[d] + gnsB * n[d];
      gdpd = gdp[d];
    }
    side_der_rev(h, gm1, n, g[0][d], g[1][d], g[2][d], g[3][d], e[d], gdUn, gdpd, gdA, gdsB, s,
                 gsB, gg[0][d], gg[1][d], gg[2][d], gg[3][d], gg[4][d]);
  }
  // q0 = A0 q + rho s B (0, n, Un / 2)
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    gA += gq0[v] * q[v];
    gq[v] += A * gq0[v];
  }
  gbe += n[0] * gq0[1] + n[1] * gq0[2] + n[2] * gq0[3] + hU * gq0[4];
  s.Un += 0.5 * be * gq0[4];
  s.rho += gbe * sB;
  gsB += gbe * w.rho;
  // A0 and s B of (Un, lam)
  s.Un += 2.0 * w.lam * sB * (gA - h.Un * gsB);
  s.lam += sB * (h.Un * gA - (h.Un * h.Un + w.hil) * gsB);
  state_rev(w, h.u2h, gm1, n, s, gq);
}

// d/dtau of the weights of fit_weights.
GKS_HD void fit_weights_dtau(double tau, double dt, FitWeights<double>& f) {
  const double e = tau > 0.0 ? exp(-0.5 * dt / tau) : 0.0;
  const double x = 1.0 - e, s = x * x, m = x * (2.0 + x);
  const double idt = 1.0 / dt, a = tau * idt, b = 4.0 * a * idt;
  const double de = tau > 0.0 ? e * 0.5 * dt / (tau * tau) : 0.0;
  const double ds = -2.0 * x * de, dm = -(2.0 + 2.0 * x) * de, db = 4.0 * idt * idt;
  f.n[0] = idt * m + a * dm;
  f.t[0] = -db * s - b * ds;
  f.n[2] = -a * m - tau * f.n[0];
  f.t[2] = b * s - tau * f.t[0];
  f.n[1] = (1.0 - s - 2.0 * a * m) - tau * (ds + 2.0 * idt * m + 2.0 * a * dm);
  f.t[1] = db * (2.0 * a * s - e * x) * dt +
           b * dt * (2.0 * idt * s + 2.0 * a * ds - de * x + e * de);
}

// Vector-Jacobian product of gp_flux_global (FP64): gacc[10] -> cotangents of both sides' values
// and gradients (accumulated). Returns false for a non-physical side or interface state. The
// heat-flux correction (Pr != 1) is not reversed.
GKS_HD bool gp_flux_global_vjp(const FluxParams<double>& P, const double vl[5],
                               const double gl[5][3], const double vr[5], const double gr[5][3],
                               const double n[3], double wq, double dt, const double gacc[10],
                               double gvl[5], double ggl[5][3], double gvr[5], double ggr[5][3]) {
  // ---- forward
  const double gm1 = P.gamma - 1.0;
  const bool full = full_terms(P);
  Side<double> hl, hr;
  if (!(to_prim(vl, P.gamma, hl.w) & to_prim(vr, P.gamma, hr.w))) return false;
  double q0[5], dW[5][3], N[3][5];
  side_terms<false>(full, P.erfc_tab, gm1, vl, gl, n, +1, hl, q0, dW, N);
  side_terms<true>(full, P.erfc_tab, gm1, vr, gr, n, -1, hr, q0, dW, N);
  double gq0[5] = {0, 0, 0, 0, 0}, gdW[5][3], gN[3][5], gpl = 0, gpr = 0;
#pragma unroll
  for (int v = 0; v < 5; ++v)
#pragma unroll
    for (int a = 0; a < 3; ++a) gdW[v][a] = 0.0;
  {
    Prim<double> w;
    if (!to_prim(q0, P.gamma, w)) return false;
    const double E = q0[4], p = w.p, Ep = E + p;
    const double U[3] = {w.U, w.V, w.W};
    const double Un = dotU(w, n[0], n[1], n[2]);
    const double u2h = 0.5 * dotU(w, w.U, w.V, w.W);
    double dp[3];
#pragma unroll
    for (int d = 0; d < 3; ++d)
      dp[d] = gm1 * (dW[4][d] - dotU(w, dW[1][d], dW[2][d], dW[3][d]) + u2h * dW[0][d]);
    Advect<double> c;
    advect(w, dW, dp, c);
    double t[5];
    time_slope(w, Ep, c, dp, t);
    const double dmn = n[0] * t[1] + n[1] * t[2] + n[2] * t[3];
    const double r2 = dmn - Un * t[0];
    const double dpt = gm1 * (t[4] - dotU(w, t[1], t[2], t[3]) + u2h * t[0]);
    const double sdp = hl.w.p >= hr.w.p ? 1.0 : -1.0, spp = hl.w.p + hr.w.p;
    const double jump = sdp * (hl.w.p - hr.w.p) / spp;
    const double tau = collision_time(P, p, w.ip, w.ir, jump, dt);
    // ---- reverse of the combination
    double gE0[5], gE1[5], gE2[5], gtau = 0.0;
    double Nn[5] = {0, 0, 0, 0, 0}, rj[3], Np = 0, nH = 0, E10 = 0;
    if (P.tau_model != 0) {
#pragma unroll
      for (int v = 0; v < 5; ++v) Nn[v] = dot3(n, dW[v]);
      Np = dot3(n, dp);
      nH = dot3(n, c.H);
      E10 = Un * c.divm + nH + Np;
      const double pd = p * c.divU + c.Gp;
#pragma unroll
      for (int j = 0; j < 3; ++j)
        rj[j] = Nn[1 + j] - U[j] * Nn[0] +
                (n[0] * dW[1][j] + n[1] * dW[2][j] + n[2] * dW[3][j] - Un * dW[0][j]);
      double E0[5], E1[5], E2[5];
      const double mn = w.rho * Un;
      E0[0] = mn;
      E0[4] = Un * Ep;
      E1[0] = E10;
      E1[4] = (Ep + p) * (Un * c.divU + nH * w.ir) + Un * (c.G[4] + 2.0 * c.Gp) +
              w.hil * (Nn[4] + Np) + Ep * ((Np - w.hil * Nn[0]) * w.ir);
      E2[0] = dmn;
      E2[4] = r2 * w.ir * Ep + Un * (t[4] + dpt);
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        E0[1 + j] = mn * U[j] + p * n[j];
        E1[1 + j] = U[j] * E10 + Un * (c.H[j] + dp[j]) + w.hil * rj[j] + n[j] * pd;
        E2[1 + j] = U[j] * r2 + Un * t[1 + j] + dpt * n[j];
      }
      FitWeights<double> f, df;
      if (full) {
        fit_weights(tau, dt, P.idt, f);
        fit_weights_dtau(tau, dt, df);
      }
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        const double a = wq * gacc[q], b = wq * gacc[5 + q];
        gE0[q] = a;
        gE1[q] = -tau * a;
        gE2[q] = b - tau * a;
        gtau -= a * (E1[q] + E2[q]);
        if (full) {
#pragma unroll
          for (int k = 0; k < 3; ++k) gN[k][q] = f.n[k] * a + f.t[k] * b;
          gE0[q] -= gN[0][q];
          gE1[q] -= gN[1][q];
          gE2[q] -= gN[2][q];
          const double d0 = N[0][q] - E0[q], d1 = N[1][q] - E1[q], d2 = N[2][q] - E2[q];
          gtau += a * (df.n[0] * d0 + df.n[1] * d1 + df.n[2] * d2) +
                  b * (df.t[0] * d0 + df.t[1] * d1 + df.t[2] * d2);
        }
      }
      if (full && !(tau > 0.0)) gtau = 0.0;  // the full form's branch at tau = 0 is constant
    } else {
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        gE0[q] = wq * gacc[q];
        gE2[q] = wq * gacc[5 + q];
      }
    }
    // ---- reverse of the interface terms
    StateG s;
    AdvectG ga;
    double gEp = 0, gdp[3] = {0, 0, 0}, gNn[5] = {0, 0, 0, 0, 0}, gt[5];
    // E2
    {
      const double* y = gE2;
      const double ny = n[0] * y[1] + n[1] * y[2] + n[2] * y[3];
      const double x = gm1 * (ny + y[4] * Un);  // cotangent of dpt times gamma - 1
      const double gr = dotU(w, y[1], y[2], y[3]) + y[4] * w.ir * Ep;
      s.ir += y[4] * r2 * Ep;
      gEp += y[4] * r2 * w.ir;
      s.Un += y[1] * t[1] + y[2] * t[2] + y[3] * t[3] + y[4] * (t[4] + dpt) - gr * t[0];
      const double gd = y[0] + gr;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        s.U[a] += y[1 + a] * r2 - x * t[1 + a];
        gt[1 + a] = Un * y[1 + a] + gd * n[a] - x * U[a];
      }
      gt[4] = y[4] * Un + x;
      gt[0] = x * u2h - gr * Un;
      s.u2h += x * t[0];
    }
    time_slope_rev(w, Ep, c, gt, s, ga, gdp);
    // E0
    {
      const double* y = gE0;
      const double gm = y[0] + dotU(w, y[1], y[2], y[3]), mn = w.rho * Un;
#pragma unroll
      for (int a = 0; a < 3; ++a) s.U[a] += mn * y[1 + a];
      s.p += n[0] * y[1] + n[1] * y[2] + n[2] * y[3];
      s.Un += y[4] * Ep + gm * w.rho;
      gEp += y[4] * Un;
      s.rho += gm * Un;
    }
    if (P.tau_model != 0) {
      // E1
      const double* y = gE1;
      const double y4 = y[4], X = Ep + p, nth = Np - w.hil * Nn[0];
      const double gX = y4 * (Un * c.divU + nH * w.ir);
      gEp += gX + y4 * nth * w.ir;
      s.p += gX;
      s.Un += y4 * (X * c.divU + c.G[4] + 2.0 * c.Gp);
      ga.divU += y4 * X * Un;
      double gnH = y4 * X * w.ir;
      s.ir += y4 * (X * nH + Ep * nth);
      ga.G4 += y4 * Un;
      ga.Gp += 2.0 * y4 * Un;
      const double k = y4 * Ep * w.ir;
      s.hil += y4 * (Nn[4] + Np) - k * Nn[0];
      gNn[4] = y4 * w.hil;
      double gNp = gNn[4] + k;
      gNn[0] = -k * w.hil;
      double g0 = y[0], gpd = 0;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const double yj = y[1 + j], z = yj * w.hil;
        g0 += U[j] * yj;
        s.U[j] += yj * E10 - z * Nn[0];
        s.Un += yj * (c.H[j] + dp[j]) - z * dW[0][j];
        ga.H[j] += yj * Un;
        gdp[j] += yj * Un;
        s.hil += yj * rj[j];
        gpd += yj * n[j];
        gNn[1 + j] = z;
        gNn[0] -= z * U[j];
#pragma unroll
        for (int b = 0; b < 3; ++b) gdW[1 + b][j] += z * n[b];
        gdW[0][j] -= z * Un;
      }
      s.Un += g0 * c.divm;
      ga.divm += g0 * Un;
      gnH += g0;
      gNp += g0;
      s.p += gpd * c.divU;
      ga.divU += gpd * p;
      ga.Gp += gpd;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        ga.H[j] += gnH * n[j];
        gdp[j] += gNp * n[j];
      }
      // collision time tau(p0, rho0, jump), jump = |pl - pr| / (pl + pr) (d|x|/dx = sign, +1
      // at 0)
      const double gj = gtau * P.tau_C * dt;
      if (P.tau_model == 2) {
        s.p -= gtau * P.mu * w.ip * w.ip;
      } else if (P.tau_model == 3) {
        // mu (p0 / (rho0 T_ref))^mu_pow / p0
        const double a = P.mu * k_pow(w.p * w.ir / P.T_ref, P.mu_pow) * w.ip;
        s.p += gtau * a * (P.mu_pow - 1.0) * w.ip;
        s.rho -= gtau * a * P.mu_pow * w.ir;
      }
      gpl = gj * (sdp - jump) / spp;
      gpr = gj * (-sdp - jump) / spp;
    }
    s.E += gEp;
    s.p += gEp;
    advect_rev(w, dW, dp, c, ga, n, gNn, s, gdp, gdW);
#pragma unroll
    for (int d = 0; d < 3; ++d)
      dp_rev(w, u2h, gm1, gdp[d], dW[0][d], dW[1][d], dW[2][d], dW[3][d], s, gdW[0][d], gdW[1][d],
             gdW[2][d], gdW[3][d], gdW[4][d]);
    state_rev(w, u2h, gm1, n, s, gq0);
  }
  // ---- reverse of both sides
  side_terms_rev(full, gm1, vl, gl, n, hl, gq0, gdW, gN, gpl, gvl, ggl);
  side_terms_rev(full, gm1, vr, gr, n, hr, gq0, gdW, gN, gpr, gvr, ggr);
  return true;
}

}  // namespace gks
