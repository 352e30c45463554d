// Per-bus arithmetic of the load gradient (adjoint.cu), FP64.
#pragma once

#include <cuda_runtime.h>

#include "loads.cuh"

namespace zbus {

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cconj(double2 a) { return make_double2(a.x, -a.y); }
// acc + a b with four FMAs
__device__ __forceinline__ double2 cfma(double2 a, double2 b, double2 acc) {
  return make_double2(fma(a.x, b.x, fma(-a.y, b.y, acc.x)), fma(a.x, b.y, fma(a.y, b.x, acc.y)));
}
__device__ __forceinline__ double2 csub(double2 a, double2 b) {
  return make_double2(a.x - b.x, a.y - b.y);
}

// conj(S / u^2) = conj(S) u^2 / |u|^4; zero for an absent load.
__device__ __forceinline__ double2 load_slope(double2 S, double2 u) {
  if (!has_load(S)) return make_double2(0.0, 0.0);
  const double q = u.x * u.x + u.y * u.y;
  const double2 u2 = cmul(u, u);
  const double2 r = cmul(cconj(S), u2);
  const double inv = 1.0 / (q * q);
  return make_double2(r.x * inv, r.y * inv);
}

// x / conj(u) = x u / |u|^2; zero where u = 0 (an absent phase of a padded
// partial-phase bus).
__device__ __forceinline__ double2 div_conj(double2 x, double2 u) {
  const double q = u.x * u.x + u.y * u.y;
  if (q == 0.0) return make_double2(0.0, 0.0);
  const double2 r = cmul(x, u);
  return make_double2(r.x / q, r.y / q);
}

// Operand of one bus of an adjoint sweep: conj(lambda), lambda = G inv_s +
// A^T mu at the converged voltages v (m valid phases; absent loads zeros).  A
// bus with loads of one kind forms three slopes whichever kind it is.
__device__ __forceinline__ void adjoint_rhs(const double2* v, const double2* mu, const double2* g,
                                            double inv_s, const double2* sw, const double2* sd,
                                            int m, double2* out) {
  bool wye = false, delta = false;
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    wye = wye || has_load(sw[p]);
    delta = delta || has_load(sd[p]);
  }
  delta = delta && m == 3;
  double2 lam[3];
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    lam[p] = make_double2(g[p].x * inv_s, g[p].y * inv_s);
    if (wye && delta && p < m) {
      const double2 d = cmul(load_slope(sw[p], v[p]), mu[p]);
      lam[p].x += d.x;
      lam[p].y += d.y;
    }
  }
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    const int q = p == 2 ? 0 : p + 1;
    const double2 d = cmul(load_slope(delta ? sd[p] : sw[p], delta ? csub(v[p], v[q]) : v[p]),
                           delta ? csub(mu[p], mu[q]) : mu[p]);
    lam[p].x += d.x;
    lam[p].y += d.y;
    if (delta) {
      lam[q].x -= d.x;
      lam[q].y -= d.y;
    }
  }
#pragma unroll
  for (int p = 0; p < 3; ++p) out[p] = cconj(lam[p]);
}

}  // namespace zbus
