// FP32 Gauss-point flux (both forms, Eq. flux-1 and Eq. flux-2) with the two sides' work on
// packed f32x2 arithmetic: side_terms is instantiated with the pair type P2, one half of every
// pair carrying the left side and the other the right. The interface part (the state q0, its
// gradient, the equilibrium terms, the time-fit weights) is a function of the sums of the two
// halves and stays scalar, shared with the scalar instantiation.
#pragma once
#include "gks_f32x2.cuh"
#include "gks_flux.cuh"

namespace gks {

// Whole Gauss-point contribution (as gp_flux_global): acc[0..4] = w F^n, acc[5..9] = w dF/dt.
// Returns false for a non-physical side or interface state.
__device__ __forceinline__ bool gp_flux_global2(const FluxParams<float>& P, const float vl[5],
                                                const float gl[5][3], const float vr[5],
                                                const float gr[5][3], const float n1[3],
                                                float w, float dt, float acc[10]) {
  const bool full = full_terms(P);
  float q0[5], dW[5][3], N[3][5], pl, pr;
  {
    const P2 n[3] = {P2(n1[0]), P2(n1[1]), P2(n1[2])}, sg(1.f, -1.f);  // sg: u > 0 left, u < 0 right
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
    side_terms(full, nullptr, P2(P.gamma - 1.f), q, g, n, sg, h, Q, D, M);
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
  float Fn[5], Ft[5];
  if (!interface_flux(P, q0, dW, N, pl, pr, n1, dt, Fn, Ft)) return false;
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    acc[q] = w * Fn[q];
    acc[5 + q] = w * Ft[q];
  }
  return true;
}

}  // namespace gks
