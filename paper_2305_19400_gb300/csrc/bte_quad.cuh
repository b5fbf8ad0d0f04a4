// bte_quad.cuh -- band equilibrium intensity by Gauss-Legendre quadrature (FP64).
#pragma once
#include "bte_internal.h"

namespace bte {

// Band quadrature.  I0_b(T) = sum_i C_i / expm1(c_i / T) (Gauss-Legendre on the
// band).  With n = 1/(e^x - 1), x = c/T, q = n(1+n) x and u = (1+2n) x - 2:
// dn/dT = q/T, d2n/dT2 = q u/T^2, d3n/dT3 = q (u^2 - 2u - 2 + 2 q x)/T^3.
__device__ __forceinline__ double band_I0(const double* __restrict__ c, const double* __restrict__ C, int ng,
                                          double rT) {
  double s = 0.0;
  for (int i = 0; i < ng; ++i) s = fma(C[i], 1.0 / expm1(c[i] * rT), s);
  return s;
}

// One node's terms: n, q, q u and q (u^2 - 2u - 2 + 2 q x).
__device__ __forceinline__ void node_terms(double x, double (&t)[4]) {
  const double n = 1.0 / expm1(x);
  const double q = fma(n, n, n) * x;
  const double u = fma(2.0 * n, x, x) - 2.0;
  t[0] = n;
  t[1] = q;
  t[2] = q * u;
  t[3] = q * fma(2.0 * q, x, fma(u, u - 2.0, -2.0));
}

// I0_b and its first three temperature derivatives.
__device__ __forceinline__ void band_I0_d3(const double* __restrict__ c, const double* __restrict__ C, int ng,
                                           double rT, double (&f)[4]) {
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  for (int i = 0; i < ng; ++i) {
    double t[4];
    node_terms(c[i] * rT, t);
#pragma unroll
    for (int k = 0; k < 4; ++k) s[k] = fma(C[i], t[k], s[k]);
  }
  f[0] = s[0];
  f[1] = s[1] * rT;
  f[2] = s[2] * rT * rT;
  f[3] = s[3] * rT * rT * rT;
}

}  // namespace bte
