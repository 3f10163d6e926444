// Shared parts of the Gauss-point flux (Section 3.2): scalar functions per type, primitives,
// flux parameters, collision time, boundary ghosts and the evaluation of the reconstruction. The
// flux itself is in gks_flux.cuh.
#pragma once

#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstring>

#include "gks_internal.h"

namespace gks {

#define GKS_HD __host__ __device__ __forceinline__

GKS_HD double k_exp(double x) { return exp(x); }
GKS_HD float k_exp(float x) { return expf(x); }
GKS_HD double k_erfc(double x) { return erfc(x); }
GKS_HD float k_erfc(float x) { return erfcf(x); }
GKS_HD double k_sqrt(double x) { return sqrt(x); }
GKS_HD float k_sqrt(float x) { return sqrtf(x); }
GKS_HD double k_abs(double x) { return fabs(x); }
GKS_HD float k_abs(float x) { return fabsf(x); }
GKS_HD double k_pow(double x, double y) { return pow(x, y); }
GKS_HD float k_pow(float x, float y) { return powf(x, y); }
// Quotients of the per-state terms (reciprocals of rho and p, the half-line B, the pressure
// jump): the IEEE division, except for FP32 on the device, which takes the fast division intrinsic
// (within 2 ulp for divisors below 2^126). Against IEEE divisions, in the face-frame form of the
// flux that preceded this one: smooth 0.438 -> 0.421 ms per launch on the 64^3-cube mesh, full
// 6.52 -> 6.06 ms on the 128^3-cube explosion.
template <class R>
GKS_HD R k_div(R a, R b) {
  return a / b;
}
GKS_HD float k_div(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fdividef(a, b);
#else
  return a / b;
#endif
}

template <class R>
struct Prim {
  R rho, U, V, W, p, lam;
  R ir, ip, hil;  // 1/rho, 1/p, 1/(2 lam) = p/rho
};

// Primitives and the reciprocals the flux reuses (two divisions per state).
template <class R>
GKS_HD bool to_prim(const R q[5], R gamma, Prim<R>& w) {
  w.rho = q[0];
  w.ir = k_div(R(1), q[0]);
  w.U = q[1] * w.ir;
  w.V = q[2] * w.ir;
  w.W = q[3] * w.ir;
  w.p = (gamma - R(1)) * (q[4] - R(0.5) * (q[1] * w.U + q[2] * w.V + q[3] * w.W));
  w.ip = k_div(R(1), w.p);
  w.lam = R(0.5) * w.rho * w.ip;
  w.hil = w.p * w.ir;
  return (w.rho > R(0)) && (w.p > R(0));  // false also for NaN
}
// Whether a positive x lies well inside the FP64 range (2^-940 to 2^940), by its exponent bits.
GKS_HD bool mid_range(double x) {
#ifdef __CUDA_ARCH__
  const uint32_t hi = (uint32_t)__double2hiint(x);
#else
  uint64_t u;
  memcpy(&u, &x, sizeof(u));
  const uint32_t hi = (uint32_t)(u >> 32);
#endif
  return hi - 0x05300000u < 0x75800000u;  // false for negative, zero, infinite and NaN as well
}
// FP64: both reciprocals from one division, 1 / (rho rho p) (a division is a chain of about ten
// instructions on the FP64 pipe, which bounds the FP64 kernels), where that product is positive
// and far from the ends of the range.
GKS_HD bool to_prim(const double q[5], double gamma, Prim<double>& w) {
  w.rho = q[0];
  const double rp = (gamma - 1.0) *
                    (q[0] * q[4] - 0.5 * (q[1] * q[1] + q[2] * q[2] + q[3] * q[3]));  // rho p
  const double rrp = q[0] * rp;
  if (!mid_range(rrp) || !mid_range(rp)) return to_prim<double>(q, gamma, w);
  const double r = 1.0 / rrp;
  w.ir = rp * r;
  w.U = q[1] * w.ir;
  w.V = q[2] * w.ir;
  w.W = q[3] * w.ir;
  w.p = rp * w.ir;
  w.ip = q[0] * (q[0] * r);
  w.lam = 0.5 * w.rho * w.ip;
  w.hil = w.p * w.ir;
  return (w.rho > 0.0) && (w.p > 0.0);
}

// erfc(z) / 2 and its derivative -exp(-z^2) / sqrt(pi) in FP64 from one table: Taylor
// polynomials of degree 9 about the points i / 64, |i| <= 256 (coefficients f^(k) / k! from the
// Hermite recurrence, filled on the host in extended precision). |z - i/64| <= 1/128, so the
// remainder is below 2^-53 of either value up to |z| = 4; beyond it the library functions. Both
// values take 17 FMAs and one record of 80 bytes, where erfc and exp take about five times that
// on the FP64 pipe (k_flux FP64 1.77 -> 1.49 ms with the single division of to_prim, smooth form,
// 299 k faces); largest errors over 20,000 points 1.9 and 2.8 times 2^-53.
constexpr int kErfcSteps = 64, kErfcMax = 4, kErfcTerms = 10;
constexpr int kErfcRecords = 2 * kErfcSteps * kErfcMax + 1;
GKS_HD bool half_erfc(const double* tab, double z, double& f, double& d) {
  if (!(tab && k_abs(z) < (double)kErfcMax)) return false;
  const int i = (int)(z * kErfcSteps + (z < 0.0 ? -0.5 : 0.5));
  const double t = z - (double)i * (1.0 / kErfcSteps);
  const double2* c = reinterpret_cast<const double2*>(tab + kErfcTerms * (i + kErfcSteps * kErfcMax));
  double k[kErfcTerms];
#pragma unroll
  for (int j = 0; j < kErfcTerms / 2; ++j) {
    const double2 x = c[j];
    k[2 * j] = x.x;
    k[2 * j + 1] = x.y;
  }
  f = k[kErfcTerms - 1];
  d = f;
  f = f * t + k[kErfcTerms - 2];
#pragma unroll
  for (int j = kErfcTerms - 3; j >= 0; --j) {
    d = d * t + f;
    f = f * t + k[j];
  }
  return true;
}

template <class R>
struct FluxParams {
  R gamma, mu, tau_eps, tau_C;
  int full, tau_model;
  R pr_fix = R(0);  // 1/Pr - 1 (heat-flux correction of the smooth flux; 0 for the BGK value)
  R T_ref = R(1), mu_pow = R(0.7);  // power law mu (T / T_ref)^mu_pow (collision time 3)
  const double* erfc_tab = nullptr; // table of half_erfc (FP64 path; null: the library functions)
  R idt = R(0);                     // 1/dt where the caller has it (0: formed per point)
};

// One boundary plane: no-slip wall velocity and temperature (<= 0: adiabatic), far-field state
// (rho, U, V, W, p). The kernels read it from a [6][kPlaneStride] device table (plane axis +
// 3 side: uw[3], Tw, finf[5], padding) only at boundary faces, so that the parameter block
// holds no array indexed at run time.
template <class R>
struct WallData {
  R uw[3] = {R(0), R(0), R(0)};
  R Tw = R(0);
  const R* finf = nullptr;  // far-field planes: (rho, U, V, W, p) in the table
};
template <class R>
GKS_HD WallData<R> wall_data(const R* table, int code) {
  WallData<R> d;
  if (code >= 6) {
    const R* t = table + kPlaneStride * (code % 6);
#pragma unroll
    for (int a = 0; a < 3; ++a) d.uw[a] = t[a];
    d.Tw = t[3];
    d.finf = t + 4;
  }
  return d;
}

// Flux parameters from the solver's kernel parameters (any struct with the same field names).
template <class R, template <class> class KP>
inline FluxParams<R> flux_params(const KP<R>& p) {
  FluxParams<R> fp;
  fp.gamma = p.gamma;
  fp.mu = p.mu;
  fp.tau_eps = p.tau_eps;
  fp.tau_C = p.tau_C;
  fp.full = p.flux_mode;
  fp.tau_model = p.tau_model;
  fp.pr_fix = p.pr_fix;
  fp.T_ref = p.T_ref;
  fp.mu_pow = p.mu_pow;
  return fp;
}

// Collision time of the interface (Section 5): zero; inviscid (eps + C dp) dt; viscous
// mu / p0 + C dp dt, with mu constant or the power law of Section 5.4 at T0 = p0 / rho0.
template <class R>
GKS_HD R collision_time(const FluxParams<R>& P, R p0, R ip0, R ir0, R dp, R dt) {
  if (P.tau_model == 1) return (P.tau_eps + P.tau_C * dp) * dt;
  if (P.tau_model == 2) return P.mu * ip0 + P.tau_C * dp * dt;
  if (P.tau_model == 3)
    return P.mu * k_pow(k_div(p0 * ir0, P.T_ref), P.mu_pow) * ip0 + P.tau_C * dp * dt;
  return R(0);
}

// Far-field state at a plane of axis ax with outward normal sign sg (Section 5.4, Riemann
// invariants): R+ = u_n + 2c/(gamma-1) from the inside state q, R- = u_n - 2c/(gamma-1) from
// the far field; u_n and c of the boundary are their mean and (gamma-1)/4 of their difference;
// entropy p/rho^gamma and tangential velocity from the upwind side; supersonic inflow takes the
// far field, supersonic outflow q. Conserved variables in and out.
template <class R>
GKS_HD void farfield_state(const FluxParams<R>& P, const R finf[5], int ax, R sg, const R q[5],
                           R out[5]) {
  const R g = P.gamma, gm1 = P.gamma - R(1);
  const R ir = R(1) / q[0];
  const R U[3] = {q[1] * ir, q[2] * ir, q[3] * ir};
  const R p = gm1 * (q[4] - R(0.5) * (q[1] * U[0] + q[2] * U[1] + q[3] * U[2]));
  const R c = k_sqrt(g * p * ir);
  const R un = sg * U[ax];
  const R rinf = finf[0], pinf = finf[4];
  const R Uinf[3] = {finf[1], finf[2], finf[3]};
  const R uninf = sg * Uinf[ax];
  const R cinf = k_sqrt(g * pinf / rinf);
  R rb, pb, Ub[3];
  if (un >= c) {
#pragma unroll
    for (int v = 0; v < 5; ++v) out[v] = q[v];
    return;
  }
  if (un <= -c) {
    rb = rinf;
    pb = pinf;
#pragma unroll
    for (int a = 0; a < 3; ++a) Ub[a] = Uinf[a];
  } else {
    const R Rp = un + R(2) * c / gm1, Rm = uninf - R(2) * cinf / gm1;
    const R unb = R(0.5) * (Rp + Rm), cb = R(0.25) * gm1 * (Rp - Rm);
    const bool out_flow = unb >= R(0);
    const R s = out_flow ? p / k_pow(q[0], g) : pinf / k_pow(rinf, g);
#pragma unroll
    for (int a = 0; a < 3; ++a) Ub[a] = out_flow ? U[a] : Uinf[a];
    Ub[ax] = sg * unb;  // tangential components kept, the normal one from the invariants
    rb = k_pow(cb * cb / (g * s), R(1) / gm1);
    pb = rb * cb * cb / g;
  }
  out[0] = rb;
#pragma unroll
  for (int a = 0; a < 3; ++a) out[1 + a] = rb * Ub[a];
  out[4] = pb / gm1 + R(0.5) * rb * (Ub[0] * Ub[0] + Ub[1] * Ub[1] + Ub[2] * Ub[2]);
}

// Ghost value and gradient at a Gauss point of wall `code` (global frame; code as in
// gks_internal.h: axis + 3 side, + 6 for a no-slip wall). Geometry is mirrored (d/dx_axis
// changes sign); the flow variables: slip, the normal momentum negated; no-slip with (U_w, T_w),
// rho_g = rho, m_g = 2 U_w rho - m and E_g = E + 2 |U_w|^2 rho - 2 U_w . m (adiabatic, p_g = p)
// or E_g = 2 rho T_w / (gamma-1) - E + |m|^2/rho + 2 |U_w|^2 rho - 2 U_w . m (isothermal,
// T_g = 2 T_w - T); the gradient is mapped by the Jacobian of that map.
// kFar = false leaves the far-field branch out (for callers that never see far-field planes).
template <class R, bool kFar = true>
GKS_HD void wall_ghost(const FluxParams<R>& P, int code, const WallData<R>& wd, const R v[5],
                       const R g[5][3], R vg[5], R gg[5][3]) {
  const int ax = code % 3;
  if (kFar && code >= 12) {  // far field: the characteristic state, uniform
    farfield_state(P, wd.finf, ax, (code % 6) >= 3 ? R(1) : R(-1), v, vg);
#pragma unroll
    for (int r = 0; r < 5; ++r)
#pragma unroll
      for (int b = 0; b < 3; ++b) gg[r][b] = R(0);
    return;
  }
  if (code < 6) {
#pragma unroll
    for (int r = 0; r < 5; ++r) {
      const R sv = (r == 1 + ax) ? R(-1) : R(1);
      vg[r] = sv * v[r];
#pragma unroll
      for (int b = 0; b < 3; ++b) gg[r][b] = (b == ax ? -sv : sv) * g[r][b];
    }
    return;
  }
  const R u0 = wd.uw[0], u1 = wd.uw[1], u2 = wd.uw[2], Tw = wd.Tw;
  const R uw2 = u0 * u0 + u1 * u1 + u2 * u2;
  const R uw[3] = {u0, u1, u2};
  // row 4 of the Jacobian: dE_g = j0 drho + jm . dm + j4 dE
  R j0, jm[3], j4;
  const R rho = v[0];
  const R um = u0 * v[1] + u1 * v[2] + u2 * v[3];
  if (Tw > R(0)) {
    const R ir = R(1) / rho;
    const R U[3] = {v[1] * ir, v[2] * ir, v[3] * ir};
    const R U2 = U[0] * U[0] + U[1] * U[1] + U[2] * U[2];
    const R cT = R(2) * Tw / (P.gamma - R(1));
    vg[4] = cT * rho - v[4] + U2 * rho + R(2) * uw2 * rho - R(2) * um;
    j0 = cT - U2 + R(2) * uw2;
#pragma unroll
    for (int a = 0; a < 3; ++a) jm[a] = R(2) * (U[a] - uw[a]);
    j4 = R(-1);
  } else {
    vg[4] = v[4] + R(2) * uw2 * rho - R(2) * um;
    j0 = R(2) * uw2;
#pragma unroll
    for (int a = 0; a < 3; ++a) jm[a] = R(-2) * uw[a];
    j4 = R(1);
  }
  vg[0] = rho;
#pragma unroll
  for (int a = 0; a < 3; ++a) vg[1 + a] = R(2) * uw[a] * rho - v[1 + a];
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    const R sb = b == ax ? R(-1) : R(1);
    gg[0][b] = sb * g[0][b];
#pragma unroll
    for (int a = 0; a < 3; ++a) gg[1 + a][b] = sb * (R(2) * uw[a] * g[0][b] - g[1 + a][b]);
    gg[4][b] = sb * (j0 * g[0][b] + jm[0] * g[1][b] + jm[1] * g[2][b] + jm[2] * g[3][b] +
                     j4 * g[4][b]);
  }
}

// The wall flux (after the Gauss-point sum): no mass; a slip wall passes normal momentum only;
// an adiabatic no-slip wall conducts no heat, so its energy flux is U_w . (momentum flux).
template <class R>
GKS_HD void wall_flux_fix(int code, const WallData<R>& wd, R acc[10]) {
  if (code >= 12) return;  // a far-field plane passes the GKS flux of its ghost pair
  acc[0] = acc[5] = R(0);
  const int ax = code % 3;
  if (code < 6) {
#pragma unroll
    for (int v = 1; v < 5; ++v)
      if (v != 1 + ax) acc[v] = acc[5 + v] = R(0);
    return;
  }
  if (wd.Tw <= R(0)) {
    acc[4] = wd.uw[0] * acc[1] + wd.uw[1] * acc[2] + wd.uw[2] * acc[3];
    acc[9] = wd.uw[0] * acc[6] + wd.uw[1] * acc[7] + wd.uw[2] * acc[8];
  }
}

// The ten coefficients of variable v through the accessor; accessors over device memory
// provide their own (vector-load) version, found by argument-dependent lookup.
template <class Coef, class R>
GKS_HD void load_coefs(const Coef& coef, int v, R k[10]) {
#pragma unroll
  for (int j = 0; j < 10; ++j) k[j] = coef(v, j);
}

// Value and gradient at offset d of a cell polynomial c[v][j] in physical offsets from the
// centroid: Q = c0 + c1 dx + c2 dy + c3 dz + c4 dx^2 + c5 dy^2 + c6 dz^2 + c7 dxdy + c8 dxdz
// + c9 dydz. `coef(v, j)` returns coefficient j of variable v.
template <class R, class Coef>
GKS_HD void eval_poly(const Coef& coef, const R d[3], R val[5], R grad[5][3]) {
  const R tx = R(2) * d[0], ty = R(2) * d[1], tz = R(2) * d[2];
  const R hx = R(0.5) * d[0], hy = R(0.5) * d[1], hz = R(0.5) * d[2];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    R k[10];
    load_coefs(coef, v, k);
    grad[v][0] = k[1] + k[4] * tx + k[7] * d[1] + k[8] * d[2];
    grad[v][1] = k[2] + k[5] * ty + k[7] * d[0] + k[9] * d[2];
    grad[v][2] = k[3] + k[6] * tz + k[8] * d[0] + k[9] * d[1];
    // Q(d) = c0 + d . (grad Q(0) + grad Q(d)) / 2 for a quadratic: 15 instructions a variable
    // against 21 with the products of the offsets
    val[v] = k[0] + hx * (k[1] + grad[v][0]) + hy * (k[2] + grad[v][1]) + hz * (k[3] + grad[v][2]);
  }
}

}  // namespace gks
