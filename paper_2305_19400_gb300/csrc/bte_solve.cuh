// bte_solve.cuh -- exact FP64 solve of the T_p equation for one cell, by one warp or one thread-block cluster.
#pragma once
#include <cooperative_groups.h>

#include <cmath>

#include "bte_ff.cuh"
#include "bte_quad.cuh"

namespace bte {

// Relative trust radius of a cell's third-order Taylor model of I0_b(T) for a
// solve tolerance rtol.  For the bands up to 1e14 rad/s the remainder is at most
// 0.4 (d/T)^4 I0_b at 300 K and 5.7 (d/T)^4 I0_b at 100 K: at the radius
// (rtol/32)^(1/4), 1.33e-4 for 1e-14, that is 1.2e-16 and 1.8e-15.  The
// second-order model took (rtol/4)^(1/3) = 1.36e-5 (2.1e-15 and 6.0e-14 there,
// and no less than this one's down to 26 K); cells drift out of the ten times
// wider radius ten times less often.
inline double model_trust(double rtol) { return std::pow(rtol / 32.0, 0.25); }

// Root nearest 0 of F + F1 d + F2 d^2 / 2 + F3 d^3 / 6, the step of the cell's
// cached temperature model: an FP32 estimate from the stable form of the
// quadratic's root, -2F / (F1 + sqrt(F1^2 - 2 F F2)) (-F / F1 without a real
// root), then one Newton step on the cubic in FP64 with the FP32 reciprocal of
// the derivative.  The estimate is good to about 2e-7 of d (FP32 rounding and,
// inside the trust radius, the cubic term) and the step to about 1e-13 of d,
// while an accepted d is below 2e-4 T.  The FP64 pipe of GB300 takes about 76
// cycles per warp instruction: this form issues eight FP64 operations where a
// square root and a division take twenty-odd, and its conversions run on the
// integer pipe (bte_ff.cuh).
__device__ __forceinline__ double model_step(double F, double F1, double F2, double F3) {
  float f, f1, f2, lo;
  ff::split(F, f, lo);
  ff::split(F1, f1, lo);
  ff::split(F2, f2, lo);
  const float disc = fmaf(f1, f1, -2.0f * f * f2);
  const float d0f = (disc >= 0.0f && f1 > 0.0f) ? -2.0f * f / (f1 + sqrtf(disc)) : -f / f1;
  const double d0 = ff::to_double(d0f, 0.0f);
  const double h = fma(F3 * (1.0 / 6.0), d0, 0.5 * F2);
  const double q = fma(fma(h, d0, F1), d0, F);
  float qp;
  ff::split(fma(fma(0.5 * F3, d0, F2), d0, F1), qp, lo);
  const double r = ff::to_double(1.0f / qp, 0.0f);
  return fma(-q, r, d0);
}

// The model's value at T_e + d from one band's column of the cell's rows ([4][ld]).
__device__ __forceinline__ double model_I0(const double* Jb, int ld, double d) {
  return fma(fma(fma(Jb[3 * ld] * (1.0 / 6.0), d, 0.5 * Jb[2 * ld]), d, Jb[ld]), d, Jb[0]);
}

struct SolveResult {
  double Te;     // last exact evaluation point (its I0 and three derivatives are in Jrow)
  double delta;  // accepted step from Te: T_p = Te + delta
  int evals;     // exact band-quadrature evaluations
  int fallback;  // 1 when bisection was needed
  int bad;       // 1 when no temperature in [1, 5000] K was found
  double M[4];   // sum_b w_b of I0_b and its first three derivatives at Te: the cell's model sums
};

// Control of the exact solve of sum_b w_b I0_b(T) = Ep: Halley steps from T0
// on the exact band quadrature (F and three derivatives from one evaluation),
// bisection on [1, 5000] K as the fallback.  A step delta is accepted when
// |delta| <= trust_rel * T, where the third-order Taylor model at the
// evaluation point is accurate to the solve tolerance; an accepted step takes
// one Newton step on that model's cubic (the Halley step itself leaves an
// error of third order in delta).  Shared by the warp and the CTA forms
// below, so both take the same decisions from the same sums.
struct SolveCtl {
  double T, lo, hi, delta;
  int mode, iters;  // mode 0 Halley, 1 bisection, 2 final
  bool done;
  SolveResult r;

  __device__ explicit SolveCtl(double T0)
      : T((T0 >= kTmin && T0 <= kTmax && isfinite(T0)) ? T0 : 300.0), lo(kTmin), hi(kTmax), delta(0.0), mode(0),
        iters(0), done(false), r{T, 0.0, 0, 0, 0, {0.0, 0.0, 0.0, 0.0}} {}

  // One evaluation's sums at T; moves T to the next evaluation point or sets done.
  __device__ void advance(double F, double F1, double F2, double F3, double Ep, double trust_rel, int maxit) {
    r.M[0] = F;
    r.M[1] = F1;
    r.M[2] = F2;
    r.M[3] = F3;
    F -= Ep;
    ++r.evals;
    r.Te = T;
    if (mode == 0) {
      ++iters;
      bool badstep = !(isfinite(F) && isfinite(F1) && F1 > 0.0);
      double Tn = T;
      if (!badstep) {
        const double newton = -F / F1;
        const double h = F * F2 / (2.0 * F1 * F1);
        delta = fabs(h) < 0.5 ? newton / (1.0 - h) : newton;
        Tn = T + delta;
        badstep = !(Tn >= kTmin && Tn <= kTmax) || iters > maxit;
      }
      if (badstep) {
        mode = 1;
        lo = kTmin;
        hi = kTmax;
        T = 0.5 * (lo + hi);
        r.fallback = 1;
      } else if (fabs(delta) <= trust_rel * Tn) {
        const double g = fma(fma(fma(F3 * (1.0 / 6.0), delta, 0.5 * F2), delta, F1), delta, F);
        delta -= g / fma(fma(0.5 * F3, delta, F2), delta, F1);
        done = true;
      } else {
        T = Tn;
      }
    } else if (mode == 1) {
      if (F < 0.0) lo = T; else hi = T;
      T = 0.5 * (lo + hi);
      ++iters;
      if (hi - lo <= 4e-16 * hi || iters >= maxit + 200) mode = 2;
    } else {
      delta = 0.0;
      done = true;
      if (T <= kTmin * (1.0 + 1e-9) || T >= kTmax * (1.0 - 1e-9)) r.bad = 1;
    }
  }

  __device__ SolveResult finish() {
    if (!done) {
      r.bad = 1;
      delta = 0.0;
    }
    r.delta = delta;
    return r;
  }
};

// Exact solve by one warp (w = a_p unless given): lanes over bands.  Each
// evaluation's I0 and three derivatives per band are written to Jrow ([4][nbp],
// may be null).  All 32 lanes of the warp must call it.
__device__ inline SolveResult exact_solve_warp(const ThermoTables& th, double Ep, double T0, double trust_rel, int maxit,
                                               double* Jrow, const double* wts = nullptr) {
  const double* wb = wts ? wts : th.a_p;
  const int lane = threadIdx.x & 31;
  const int nbp = th.nbp, ng = th.ng;
  SolveCtl c(T0);
  for (int loop = 0; loop < maxit + 224 && !c.done; ++loop) {
    const double rT = 1.0 / c.T;
    double F[4] = {0.0, 0.0, 0.0, 0.0};
    for (int b = lane; b < nbp; b += 32) {
      double f[4];
      band_I0_d3(th.node_c + b * ng, th.node_C + b * ng, ng, rT, f);
      const double ap = wb[b];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (Jrow) Jrow[k * nbp + b] = f[k];
        F[k] = fma(ap, f[k], F[k]);
      }
    }
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
      for (int k = 0; k < 4; ++k) F[k] += __shfl_xor_sync(0xffffffffu, F[k], o);
    }
    c.advance(F[0], F[1], F[2], F[3], Ep, trust_rel, maxit);
  }
  return c.finish();
}

// Shared memory (doubles) of exact_solve_cluster, per CTA.
// (band, node) pairs per chunk of a CTA of a cluster of nr: all of its bands'
// nodes, 768 (42 KB of scratch with 256 bands) at most.
__host__ __device__ inline int cta_solve_pairs(int nbp, int ng, int nr) {
  const int all = (nbp + nr - 1) / nr * ng;
  return all < 768 ? all : 768;
}
__host__ __device__ inline int cta_solve_smem_doubles(int nbp, int ng, int nr) {
  return 4 * cta_solve_pairs(nbp, ng, nr) + 8 * nbp + 4;
}

// The same solve by a thread-block cluster, bit for bit the warp form's
// results.  CTA r of the C in the cluster evaluates the bands
// [r nbp / C, (r + 1) nbp / C): the costly per-node terms (expm1, the
// reciprocal, the derivative factors) are spread over its threads, and each
// band's node sums run in node order on one thread, writing the four values to the
// CTA's own shared memory (and the cell's model row Jrow).  After one cluster
// barrier warp 0 of every CTA adds all bands through distributed shared
// memory in the warp form's order, so every CTA holds the same sums and
// advances the same controller, and the loop ends on the same evaluation
// everywhere.  The band values alternate between two buffers over the
// cluster's successive evaluations (par counts them across calls): evaluation
// k writes buffer k % 2 after the barrier of evaluation k - 1, which every
// reader of buffer (k - 2) % 2 has passed.  One cell's evaluation thus runs
// on C SMs' FP64 units.  sm: cta_solve_smem_doubles doubles per CTA.
// Every thread of every CTA of the cluster must call it (it synchronises the
// cluster).
__device__ inline SolveResult exact_solve_cluster(const ThermoTables& th, double Ep, double T0, double trust_rel,
                                                  int maxit, double* Jrow, double* sm, unsigned& par) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), nr = (int)cl.num_blocks();
  const double* wb = th.a_p;
  const int nbp = th.nbp, ng = th.ng;
  const int own0 = rank * nbp / nr, own1 = (rank + 1) * nbp / nr;  // this CTA's bands
  const int pairs = cta_solve_pairs(nbp, ng, nr), cb = pairs / ng;  // bands per chunk (ng <= kMaxGauss)
  double* pt = sm;                        // [4][pairs] node_terms of each pair
  double* bv2 = pt + 4 * pairs;  // [2][4][nbp] per band I0 and three derivatives (own bands), two buffers
  double* sums = bv2 + 8 * nbp;           // [4] this CTA's copy of F and its derivatives
  SolveCtl c(T0);
  for (int loop = 0; loop < maxit + 224 && !c.done; ++loop) {
    double* bv = bv2 + (size_t)(par++ & 1u) * 4 * nbp;
    const double rT = 1.0 / c.T;
    for (int b0 = own0; b0 < own1; b0 += cb) {
      const int npair = min(cb, own1 - b0) * ng;
      const double* cn = th.node_c + b0 * ng;
#pragma unroll 1
      for (int p = threadIdx.x; p < npair; p += blockDim.x) {
        double t[4];
        node_terms(cn[p] * rT, t);
#pragma unroll
        for (int q = 0; q < 4; ++q) pt[q * pairs + p] = t[q];
      }
      __syncthreads();
#pragma unroll 1
      for (int k = threadIdx.x; k < npair / ng; k += blockDim.x) {
        const int b = b0 + k;
        const double* C = th.node_C + b * ng;
        double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 2
        for (int i = 0; i < ng; ++i)
#pragma unroll
          for (int q = 0; q < 4; ++q) s[q] = fma(C[i], pt[q * pairs + k * ng + i], s[q]);
        const double f[4] = {s[0], s[1] * rT, s[2] * rT * rT, s[3] * rT * rT * rT};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          bv[q * nbp + b] = f[q];
          if (Jrow) Jrow[q * nbp + b] = f[q];
        }
      }
      __syncthreads();
    }
    cl.sync();  // every CTA's bands are in its bv
    if (threadIdx.x < 32) {
      const int lane = threadIdx.x;
      double F[4] = {0.0, 0.0, 0.0, 0.0};
      for (int b = lane; b < nbp; b += 32) {
        int o = (int)(((long long)b * nr) / nbp);  // the CTA whose range holds b
        while (o + 1 < nr && (o + 1) * nbp / nr <= b) ++o;
        while (o > 0 && o * nbp / nr > b) --o;
        const double* ob = cl.map_shared_rank(bv, (unsigned)o);
        const double ap = wb[b];
#pragma unroll
        for (int q = 0; q < 4; ++q) F[q] = fma(ap, ob[q * nbp + b], F[q]);
      }
      for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int q = 0; q < 4; ++q) F[q] += __shfl_xor_sync(0xffffffffu, F[q], o);
      }
      if (lane == 0) {
#pragma unroll
        for (int q = 0; q < 4; ++q) sums[q] = F[q];
      }
    }
    __syncthreads();
    c.advance(sums[0], sums[1], sums[2], sums[3], Ep, trust_rel, maxit);
  }
  return c.finish();
}

}  // namespace bte
