// bte_solve.cuh -- exact FP64 solve of the T_p equation for one cell, by one warp or one thread-block cluster.
#pragma once
#include <cooperative_groups.h>

#include <cmath>

#include "bte_ff.cuh"
#include "bte_quad.cuh"

namespace bte {

// Relative trust radius of a cell's third-order Taylor model of I0_b(T) for a
// solve tolerance rtol, (rtol/32)^(1/4) = 1.33e-4 for 1e-14, and (rtol/x)^(1/4)
// where x = hbar omega_max / (k_B T) is above 32: below T_knee (ThermoTables), 24 K for
// bands up to 1e14 rad/s.  A second-order model at (rtol/4)^(1/3) = 1.36e-5 leaves a
// remainder of 2.1e-15 I0_b at 300 K (x = 2.5) and 5.6e-14 at 100 K, this one 1.2e-16
// and 1.8e-15, and at no x more (where x is large they are x^3 rtol/24 and
// x^4/24 times the fourth power of the radius); cells drift out of the ten
// times wider radius ten times less often.
inline double model_trust(double rtol) { return std::pow(rtol / 32.0, 0.25); }

__device__ __forceinline__ bool finite(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }

// Root nearest 0 of c0 + c1 d + c2 d^2 + c3 d^3, the step of a cell's cached
// temperature model (NaN where c1 is not positive or leaves 2^-100 .. 2^101).  The
// coefficients are proportional to the relaxation rates, and c1^2 alone leaves the FP32
// range above 1.8e19 (rates of about 1e13 1/s in silicon), so they are divided by c1
// first: with a, b, c = c0, c2, c3 over c1 an FP32 estimate from the stable form of the
// quadratic's root, -2 a / (1 + sqrt(1 - 4 a b)) (-a without a real root), then
// one Newton step on the cubic in FP64 with the derivative and its reciprocal in
// FP32.  The estimate is good to about 3e-7 of d (FP32 rounding and, inside the
// trust radius, the cubic term) and the step to about 2e-13 of d, while an
// accepted d is below 2e-4 T.  The FP64 pipe of GB300 takes about 73 cycles per
// warp instruction: this form issues four FP64 operations where a square root
// and a division take twenty-odd, and its conversions run on the integer pipe.
__device__ __forceinline__ double model_step(double c0, double c1, double c2, double c3) {
  float f0, f1, f2, f3, lo;
  ff::split(c1, f1, lo);
  ff::split(c2, f2, lo);
  ff::split(c3, f3, lo);
  const float r = 1.0f / f1, b = f2 * r, c = f3 * r;  // not behind the energies
  ff::split(c0, f0, lo);
  const float a = f0 * r, disc = fmaf(-4.0f * a, b, 1.0f);
  const float df = disc >= 0.0f ? -2.0f * a / (1.0f + sqrtf(disc)) : -a;
  const double d = ff::to_double(df, 0.0f);
  const double g = fma(fma(fma(c3, d, c2), d, c1), d, c0);
  const float dg = fmaf(fmaf(3.0f * c, df, 2.0f * b), df, 1.0f);
  const double step = fma(-g, ff::to_double(r / dg, 0.0f), d);
  const int e1 = __double2hiint(c1) >> 20;  // sign and exponent
  return (unsigned)(e1 - 923) <= 200u ? step : __hiloint2double(0x7ff80000, 0);
}

// Whether a step d to T > 0 stays inside the trust radius (R float or double).
template <typename R>
__device__ __forceinline__ bool in_radius(R d, R T, R trust, R T_knee) {
  const R a = d < R(0) ? -d : d, r = trust * T;
  if (!(a <= r)) return false;
  if (T >= T_knee) return true;
  const R a2 = a * a, r2 = r * r;
  return a2 * a2 * T_knee <= r2 * r2 * T;
}
// The same for T finite, decided in FP32: the radius is not sharp to 1e-7.
__device__ __forceinline__ bool in_trust(double d, double T, float trust, float T_knee) {
  float df, Tf, lo;
  ff::split(d, df, lo);
  ff::split(T, Tf, lo);
  return finite(T) && in_radius(df, Tf, trust, T_knee);
}

// The model's value at T_e + d from one band's column of the cell's rows ([4][ld]).
__device__ __forceinline__ double model_I0(const double* Jb, int ld, double d) {
  return fma(fma(fma(Jb[3 * ld], d, Jb[2 * ld]), d, Jb[ld]), d, Jb[0]);
}

struct SolveResult {
  double Te;     // last exact evaluation point (its Taylor coefficients are in Jrow)
  double delta;  // accepted step from Te: T_p = Te + delta
  int evals;     // exact band-quadrature evaluations
  int fallback;  // 1 when bisection was needed
  int bad;       // 1 when no temperature in [1, 5000] K was found
  double M[4];   // sum_b w_b of the bands' Taylor coefficients at Te: the cell's model sums
  double ML[4];  // the same with the T_L weights (exact_solve_cluster with Jrow)
};

// Control of the exact solve of sum_b w_b I0_b(T) = Ep: Halley steps from T0
// on the exact band quadrature (F and three derivatives from one evaluation),
// bisection on [1, 5000] K as the fallback.  A step delta is accepted inside
// the trust radius, where the third-order Taylor model at the
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
        iters(0), done(false), r{T, 0.0, 0, 0, 0, {0.0, 0.0, 0.0, 0.0}, {0.0, 0.0, 0.0, 0.0}} {}

  // One evaluation's sums at T (Taylor coefficients); moves T to the next
  // evaluation point or sets done.
  __device__ void advance(const double* c, double Ep, double trust_rel, double T_knee, int maxit) {
#pragma unroll
    for (int k = 0; k < 4; ++k) r.M[k] = c[k];
    const double F = c[0] - Ep, F1 = c[1];
    ++r.evals;
    r.Te = T;
    if (mode == 0) {
      ++iters;
      bool badstep = !(finite(F) && finite(F1) && F1 > 0.0);
      double Tn = T;
      if (!badstep) {
        const double r1 = rcp_pos(F1);
        const double newton = -F * r1;
        const double h = -newton * c[2] * r1;
        delta = fabs(h) < 0.5 ? newton * rcp_pos(1.0 - h) : newton;
        Tn = T + delta;
        badstep = !(Tn >= kTmin && Tn <= kTmax) || iters > maxit;
      }
      if (badstep) {
        mode = 1;
        lo = kTmin;
        hi = kTmax;
        T = 0.5 * (lo + hi);
        r.fallback = 1;
      } else if (in_radius(delta, Tn, trust_rel, T_knee)) {
        const double g = fma(fma(fma(c[3], delta, c[2]), delta, F1), delta, F);
        const double dg = fma(fma(3.0 * c[3], delta, 2.0 * c[2]), delta, F1);
        delta = dg > 0.0 ? fma(-g, rcp_pos(dg), delta) : delta;
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
// evaluation's Taylor coefficients per band are written to Jrow ([4][nbp],
// may be null).  All 32 lanes of the warp must call it.
__device__ inline SolveResult exact_solve_warp(const ThermoTables& th, double Ep, double T0, double trust_rel, int maxit,
                                               double* Jrow, const double* wts = nullptr) {
  const double* wb = wts ? wts : th.a_p;
  const int lane = threadIdx.x & 31;
  const int nbp = th.nbp, ng = th.ng;
  SolveCtl c(T0);
  for (int loop = 0; loop < maxit + 224 && !c.done; ++loop) {
    const double rT = rcp_pos(c.T);
    double F[4] = {0.0, 0.0, 0.0, 0.0};
    for (int b = lane; b < nbp; b += 32) {
      double f[4];
      band_taylor(th.node_c + b * ng, th.node_C + b * ng, ng, rT, f);
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
    c.advance(F, Ep, trust_rel, th.T_knee, maxit);
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
  return 4 * cta_solve_pairs(nbp, ng, nr) + 8 * nbp + 8;
}

// The same solve by a thread-block cluster, or (COOP false) by one CTA alone with
// all bands and no cluster barrier.  CTA r of the C in the cluster
// evaluates the bands [r nbp / C, (r + 1) nbp / C): the costly per-node terms
// (expm1, the reciprocal, the derivative factors) are spread over its threads,
// and each of a band's four node sums runs in node order on one thread, writing
// the coefficient to the CTA's own shared memory (and the cell's model row Jrow).
// After one cluster barrier warp 0 of every CTA adds all bands through
// distributed shared memory in the warp form's order (warp 1 with the T_L
// weights when a model is kept), so every CTA holds the same sums and advances
// the same controller, and the loop ends on the same evaluation everywhere.  The
// band values alternate between two buffers over the cluster's successive
// evaluations (par counts them across calls): evaluation k writes buffer k % 2
// after the barrier of evaluation k - 1, which every reader of buffer (k - 2) % 2
// has passed.  One cell's evaluation thus runs on C SMs' FP64 units.  sm:
// cta_solve_smem_doubles doubles per CTA.  Every thread of every CTA of the
// cluster must call it (it synchronises the cluster).
template <bool COOP>
__device__ inline SolveResult exact_solve_cluster(const ThermoTables& th, const double* wb, double Ep, double T0,
                                                  double trust_rel, int maxit, double* Jrow, double* sm, unsigned& par) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = COOP ? (int)cl.block_rank() : 0, nr = COOP ? (int)cl.num_blocks() : 1;
  const int nbp = th.nbp, ng = th.ng;
  const int own0 = rank * nbp / nr, own1 = (rank + 1) * nbp / nr;  // this CTA's bands
  const int pairs = cta_solve_pairs(nbp, ng, nr), cb = pairs / ng;  // bands per chunk (ng <= kMaxGauss)
  double* pt = sm;                // [4][pairs] node_terms of each pair
  double* bv2 = pt + 4 * pairs;   // [2][4][nbp] per band Taylor coefficients (own bands), two buffers
  double* sums = bv2 + 8 * nbp;   // [8] this CTA's copy of the sums with wb, and with the T_L weights
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  SolveCtl c(T0);
  for (int loop = 0; loop < maxit + 224 && !c.done; ++loop) {
    double* bv = bv2 + (size_t)(par++ & 1u) * 4 * nbp;
    const double rT = rcp_pos(c.T);
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
      for (int e = threadIdx.x; e < npair / ng * 4; e += blockDim.x) {
        const int k = e >> 2, q = e & 3, b = b0 + k;
        const double* C = th.node_C + b * ng;
        double s = 0.0;
#pragma unroll 4
        for (int i = 0; i < ng; ++i) s = fma(C[i], pt[q * pairs + k * ng + i], s);
        s *= taylor_scale(q, rT);
        bv[q * nbp + b] = s;
        if (Jrow) Jrow[q * nbp + b] = s;
      }
      __syncthreads();
    }
    if constexpr (COOP) cl.sync();  // every CTA's bands are in its bv
    if (wid == 0 || (wid == 1 && Jrow)) {
      const double* wt = wid == 0 ? wb : th.a_L;
      double F[4] = {0.0, 0.0, 0.0, 0.0};
      for (int b = lane; b < nbp; b += 32) {
        const double* ob = bv;
        if constexpr (COOP) {
          int o = (int)(((long long)b * nr) / nbp);  // the CTA whose range holds b
          while (o + 1 < nr && (o + 1) * nbp / nr <= b) ++o;
          while (o > 0 && o * nbp / nr > b) --o;
          ob = cl.map_shared_rank(bv, (unsigned)o);
        }
        const double ap = wt[b];
#pragma unroll
        for (int q = 0; q < 4; ++q) F[q] = fma(ap, ob[q * nbp + b], F[q]);
      }
      for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int q = 0; q < 4; ++q) F[q] += __shfl_xor_sync(0xffffffffu, F[q], o);
      }
      if (lane == 0) {
#pragma unroll
        for (int q = 0; q < 4; ++q) sums[4 * wid + q] = F[q];
      }
    }
    __syncthreads();
    c.advance(sums, Ep, trust_rel, th.T_knee, maxit);
  }
  SolveResult r = c.finish();
#pragma unroll
  for (int q = 0; q < 4; ++q) r.ML[q] = sums[4 + q];
  return r;
}

}  // namespace bte
