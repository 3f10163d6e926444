// FP32 Gauss-point flux on packed f32x2 arithmetic, the flux templates instantiated with the pair
// type P2, in two forms:
//  - gp_flux_pair (smooth form, Eq. flux-2): the halves carry two Gauss points of a face, so that
//    everything -- both sides, the interface, the polynomials, which are loaded once for both
//    points -- runs two points per instruction;
//  - gp_flux_sides (full form, Eq. flux-1): the halves carry the two sides of one point; the
//    interface part stays scalar. The full form's terms of two points do not fit the registers
//    (its pair form took 285 us at best against 231, 48^3-cube explosion).
// Division, square root, exp and erfc run per half.
#pragma once
#include "gks_f32x2.cuh"
#include "gks_flux.cuh"

namespace gks {

// Which of the two points hold (bit 0, bit 1).
__device__ __forceinline__ unsigned physical_halves(const Prim<P2>& w) {
  return (w.rho.lo() > 0.f && w.p.lo() > 0.f ? 1u : 0u) |
         (w.rho.hi() > 0.f && w.p.hi() > 0.f ? 2u : 0u);
}
__device__ __forceinline__ P2 relaxation(const P2& dt, const P2& tau) {
  return P2(relaxation(dt.lo(), tau.lo()), relaxation(dt.hi(), tau.hi()));
}
__device__ __forceinline__ FluxParams<P2> pair_params(const FluxParams<float>& P) {
  FluxParams<P2> o;
  o.gamma = P2(P.gamma);
  o.mu = P2(P.mu);
  o.tau_eps = P2(P.tau_eps);
  o.tau_C = P2(P.tau_C);
  o.full = P.full;
  o.tau_model = P.tau_model;
  o.pr_fix = P2(P.pr_fix);
  o.T_ref = P2(P.T_ref);
  o.mu_pow = P2(P.mu_pow);
  o.idt = P2(P.idt);
  return o;
}

// Value and gradient of a cell polynomial at two offsets.
template <class Coef>
__device__ __forceinline__ void eval_poly2(const Coef& coef, const P2 d[3], P2 val[5],
                                           P2 grad[5][3]) {
  const P2 tx = d[0] + d[0], ty = d[1] + d[1], tz = d[2] + d[2];
  const P2 hx = P2(0.5f) * d[0], hy = P2(0.5f) * d[1], hz = P2(0.5f) * d[2];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    float c[10];
    load_coefs(coef, v, c);
    P2 k[10];
#pragma unroll
    for (int j = 0; j < 10; ++j) k[j] = P2(c[j]);
    grad[v][0] = k[1] + k[4] * tx + k[7] * d[1] + k[8] * d[2];
    grad[v][1] = k[2] + k[5] * ty + k[7] * d[0] + k[9] * d[2];
    grad[v][2] = k[3] + k[6] * tz + k[8] * d[0] + k[9] * d[1];
    val[v] = k[0] + hx * (k[1] + grad[v][0]) + hy * (k[2] + grad[v][1]) + hz * (k[3] + grad[v][2]);
  }
}

// Contributions of two Gauss points, per point (as gp_flux_global): acc[0..4] = w F^n,
// acc[5..9] = w dF/dt, zero for a point whose side or interface state is non-physical. Returns
// the points that are physical (bits). right(v, g) forms the right side's values and gradients
// into the arrays that held the left side's, after they were used.
template <class Right>
__device__ __forceinline__ unsigned gp_flux_pair(const FluxParams<float>& Pf, P2 v[5], P2 g[5][3],
                                                 Right right, const P2 n[3], const P2& w, float dt,
                                                 P2 acc[10]) {
  const FluxParams<P2> P = pair_params(Pf);
  const bool full = full_terms(P);
  const P2 gm1(Pf.gamma - 1.f);
  P2 q0[5], dW[5][3], N[3][5], pl, pr;
  unsigned ok;
  {
    Side<P2> h;
    to_prim(v, P.gamma, h.w);
    ok = physical_halves(h.w);
    side_terms<false>(full, nullptr, gm1, v, g, n, +1, h, q0, dW, N);
    pl = h.w.p;
  }
  right(v, g);
  {
    Side<P2> h;
    to_prim(v, P.gamma, h.w);
    ok &= physical_halves(h.w);
    side_terms<true>(full, nullptr, gm1, v, g, n, -1, h, q0, dW, N);
    pr = h.w.p;
  }
  Prim<P2> w0;
  to_prim(q0, P.gamma, w0);
  ok &= physical_halves(w0);
  P2 Fn[5], Ft[5];
  interface_flux(P, w0, q0, dW, N, pl, pr, n, P2(dt), Fn, Ft);
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    const P2 a = w * Fn[q], b = w * Ft[q];
    acc[q] = P2(ok & 1u ? a.lo() : 0.f, ok & 2u ? a.hi() : 0.f);
    acc[5 + q] = P2(ok & 1u ? b.lo() : 0.f, ok & 2u ? b.hi() : 0.f);
  }
  return ok;
}

// One Gauss point with its two sides in the two halves (as gp_flux_global): the sides' work is
// packed, the interface part scalar. It holds half the values of gp_flux_pair.
__device__ __forceinline__ bool gp_flux_sides(const FluxParams<float>& P, const float vl[5],
                                              const float gl[5][3], const float vr[5],
                                              const float gr[5][3], const float n1[3], float w,
                                              float dt, float acc[10]) {
  const bool full = full_terms(P);
  float q0[5], dW[5][3], N[3][5], pl, pr;
  {
    const P2 n[3] = {P2(n1[0]), P2(n1[1]), P2(n1[2])}, sg(1.f, -1.f);  // u > 0 left, u < 0 right
    P2 q[5], g[5][3];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      q[v] = P2(vl[v], vr[v]);
#pragma unroll
      for (int a = 0; a < 3; ++a) g[v][a] = P2(gl[v][a], gr[v][a]);
    }
    Side<P2> h;
    if (!to_prim(q, P2(P.gamma), h.w)) return false;
    P2 Q[5], D[5][3], M[3][5];
    side_terms<false>(full, nullptr, P2(P.gamma - 1.f), q, g, n, sg, h, Q, D, M);
    pl = h.w.p.lo();
    pr = h.w.p.hi();
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      q0[v] = hsum(Q[v]);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        dW[v][a] = hsum(D[v][a]);
        if (full) N[a][v] = hsum(M[a][v]);
      }
    }
  }
  Prim<float> w0;
  if (!to_prim(q0, P.gamma, w0)) return false;
  float Fn[5], Ft[5];
  interface_flux(P, w0, q0, dW, N, pl, pr, n1, dt, Fn, Ft);
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    acc[q] = w * Fn[q];
    acc[5 + q] = w * Ft[q];
  }
  return true;
}

}  // namespace gks
