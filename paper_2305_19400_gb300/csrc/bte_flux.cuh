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
// to all).  A thread keeps one band and walks every (threads / nbp)-th
// direction, four loads in flight and no index division; a ghost that does not
// depend on the direction is read once.  One thread per (direction, band)
// element with a 64-bit division each took 58-69 us per side of the 128x128 x
// 400 x 55 grid.
template <typename S>
__device__ double face_flux(const S* I, const double* I0ref, const double* I0wall, const DevGeom& g, int side, int f,
                            const DirInfo* dirs, const double* Sd, int nd, int nbp, double* sh) {
  const int ax = side / 2;
  const double nsign = (side & 1) ? 1.0 : -1.0;
  int i, j, k;
  if (side < 2) { j = f % g.ny; k = f / g.ny; i = (side & 1) ? g.nx - 1 : 0; }
  else if (side < 4) { i = f % g.nx; k = f / g.nx; j = (side & 1) ? g.ny - 1 : 0; }
  else { i = f % g.nx; j = f / g.nx; k = (side & 1) ? g.nz - 1 : 0; }
  const long long base = (g.cell0 + i + (long long)g.nx * (j + (long long)g.ny * k)) * nd * nbp;
  const int rows = kFluxThreads / nbp, r = threadIdx.x / nbp, b = threadIdx.x - r * nbp;
  const int bc = g.bc[side];
  double acc = 0.0;
  if (r < rows) {
    const double gv = bc == 0 ? I0wall[(g.face0[side] + f) * nbp + b] : 0.0;
    const S* gd = bc == 3 ? reinterpret_cast<const S*>(g.gdir[side]) : nullptr;
#pragma unroll 4
    for (int d = r; d < nd; d += rows) {
      const double sn = Sd[3 * d + ax] * nsign;
      double v = gv;
      if (sn > 0.0 || bc == 1) {
        const int m = sn > 0.0 ? d : (ax == 0 ? dirs[d].rx : (ax == 1 ? dirs[d].ry : dirs[d].rz));
        v = full_I(I, base + (long long)m * nbp + b, b, I0ref);
      } else if (bc == 3) {
        v = full_I(gd, ((long long)f * nd + d) * nbp + b, b, I0ref);
      }
      acc = fma(sn, v, acc);
    }
  }
  return block_sum(acc, sh);
}

}  // namespace bte
