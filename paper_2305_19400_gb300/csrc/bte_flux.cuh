// bte_flux.cuh -- the heat flow through one wall face (Sec. 3.1, surface term of
// Eq. 5), shared by bte_get_flux and the no-allocation wall flux, which so
// agree bit for bit.
#pragma once
#include "bte_store.cuh"

namespace bte {

constexpr int kFluxThreads = 256;

// Deterministic block sum of one value per thread (blockDim.x a power of two <= 1024).
__device__ __forceinline__ double block_sum(double v, double* sh) {
  sh[threadIdx.x] = v;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
    __syncthreads();
  }
  const double r = sh[0];
  __syncthreads();
  return r;
}

// Net outgoing flux sum_b sum_d (S_d . n_out) I_face through face f of a side,
// by a CTA of kFluxThreads threads (every thread calls it; the sum is returned
// to all).  Lane l of group g holds two bands and sums every groups-th leaving
// direction of the side's list, eight loads in flight; what enters is the ghost
// row times the sum of the entering weights (isothermal, diffuse), the leaving
// values themselves (mirror: their difference, zero unless not finite), or the
// face's per-direction ghosts (partially specular).  Bound by one face's
// latency.  Walking all directions and testing each took 116 us for the four
// sides of the 128x128 x 400 x 55 grid, 385 us for the six of a 23x18x13 one.
template <typename S>
__device__ double face_flux(const S* I, const double* I0ref, const double* I0wall, const DevGeom& g, int side, int f,
                            const WallDirs& wd, const double* Sd, int nd, int nbp, double* sh) {
  const int ax = side / 2;
  const double nsign = (side & 1) ? 1.0 : -1.0;
  int i, j, k;
  if (side < 2) { j = f % g.ny; k = f / g.ny; i = (side & 1) ? g.nx - 1 : 0; }
  else if (side < 4) { i = f % g.nx; k = f / g.nx; j = (side & 1) ? g.ny - 1 : 0; }
  else { i = f % g.nx; j = f / g.nx; k = (side & 1) ? g.nz - 1 : 0; }
  const int lpc = nbp / 2, groups = kFluxThreads / lpc, grp = threadIdx.x / lpc, b = 2 * (threadIdx.x - grp * lpc);
  const S* row = I + (g.cell0 + i + (long long)g.nx * (j + (long long)g.ny * k)) * nd * nbp + b;
  const int bc = g.bc[side];
  double acc = 0.0;
  if (grp < groups) {
    auto walk = [&](const S* from, const int* list, int n, bool diff) {
#pragma unroll 8
      for (int q = grp; q < n; q += groups) {
        const int d = list[q];
        double x0, x1;
        ld_pair(from + (long long)d * nbp, x0, x1);
        acc = fma(Sd[3 * d + ax] * nsign, diff ? (x0 - x0) + (x1 - x1) : x0 + x1, acc);
      }
    };
    walk(row, wd.out, wd.nout, bc == 1);
    if (bc == 3) walk(reinterpret_cast<const S*>(g.gdir[side]) + (long long)f * nd * nbp + b, wd.rest, nd - wd.nout, false);
    if (grp == 0 && bc != 1) {
      const double* gw = I0wall + (g.face0[side] + f) * nbp + b;
      double ref = 0.0;  // the reference part of the reduced modes' storage
      if constexpr (sizeof(S) != 8) ref = I0ref[b] + I0ref[b + 1];
      const double in = bc == 3 ? ref : gw[0] + gw[1];
      acc = fma(wd.sum_out, ref, fma(-wd.sum_in, in, acc));
      acc = fma(wd.sum_out_lo, ref, fma(-wd.sum_in_lo, in, acc));
    }
  }
  return block_sum(acc, sh);
}

}  // namespace bte
