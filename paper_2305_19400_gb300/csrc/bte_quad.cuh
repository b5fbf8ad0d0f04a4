// bte_quad.cuh -- band equilibrium intensity by Gauss-Legendre quadrature (FP64).
#pragma once
#include "bte_ff.cuh"
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

// 1/q for q > 0: an FP32 reciprocal and one third-order step, y (1 + e + e^2) with
// e = 1 - q y (three FP64 FMAs, error 2^-66 before the last rounding; an IEEE
// division issues about ten FP64 instructions, and the FP64 pipe is what these
// solves wait for).  Values whose reciprocal leaves the FP32 range are divided.
__device__ __forceinline__ double rcp_pos(double q) {
  const unsigned e = (unsigned)__double2hiint(q) >> 20;  // sign and exponent
  if (e - 949u > 174u) return 1.0 / q;                   // not in [2^-74, 2^101)
  float h, l, r;
  ff::split(q, h, l);
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(h));
  const double y = ff::to_double(r, 0.0f);
  const double d = fma(-q, y, 1.0);
  return fma(fma(d, d, d), y, y);
}

// One node's terms: n, q, q u and q (u^2 - 2u - 2 + 2 q x).
__device__ __forceinline__ void node_terms(double x, double (&t)[4]) {
  const double n = rcp_pos(expm1(x));
  const double q = fma(n, n, n) * x;
  const double u = fma(2.0 * n, x, x) - 2.0;
  t[0] = n;
  t[1] = q;
  t[2] = q * u;
  t[3] = q * fma(2.0 * q, x, fma(u, u - 2.0, -2.0));
}

// Factors of the nodes' sums: Taylor coefficients f, f', f''/2, f'''/6 of I0_b at T.
__device__ __forceinline__ double taylor_scale(int k, double rT) {
  return k == 0 ? 1.0 : (k == 1 ? rT : (k == 2 ? 0.5 * rT * rT : rT * rT * rT * (1.0 / 6.0)));
}

// Taylor coefficients of I0_b at T = 1/rT.
__device__ __forceinline__ void band_taylor(const double* __restrict__ c, const double* __restrict__ C, int ng,
                                            double rT, double (&f)[4]) {
  double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
  for (int i = 0; i < ng; ++i) {
    double t[4];
    node_terms(c[i] * rT, t);
#pragma unroll
    for (int k = 0; k < 4; ++k) s[k] = fma(C[i], t[k], s[k]);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) f[k] = s[k] * taylor_scale(k, rT);
}

}  // namespace bte
