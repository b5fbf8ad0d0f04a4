// bte_kernels.cu -- CUDA kernels around the sweep (sm_103a).  The sweeps (upwind
// update, walls, band sums; Sec. 3.1, Eq. 4-6) live in bte_sweep.cuh and
// bte_sweep_ff.cuh, the per-cell T_p step in bte_cells.cu.  Here:
//   gs_reduce_kernel    band sums after a sweep-ordered pass (bte_gs.cu) or an
//                       unstructured sweep;
//   init_cells / state_from_Tp / wall_I0 / wall_dev
//                       equilibrium state, cached models and Eq. 6 ghosts;
//   solve_TL_kernel     T_L on request (cached model first, exact otherwise);
//   flux_cells / flux_faces / mean / pack / unpack / energy_L
//                       heat flux, FP64 <-> storage packing, E_L after a restore.
#include <algorithm>
#include <type_traits>

#include "bte_ff.cuh"
#include "bte_flux.cuh"
#include "bte_quad.cuh"
#include "bte_solve.cuh"
#include "bte_store.cuh"

namespace bte {

namespace {

// ---------------------------------------------------------------------------
// Per-cell thermodynamic state at temperature T: I0cell, cached model J at T
// with its T_p sums Msum, T_e = T_p = T.  One CTA per cell (grid-stride);
// bands over threads.
__device__ void cell_state_at(double* I0cell, double* J, double* Msum, long long P, double T, ThermoTables th,
                              double* row) {
  const double rT = 1.0 / T;
  double* Jrow = J + (P * 4) * th.nbp;
  for (int b = threadIdx.x; b < th.nbp; b += blockDim.x) {  // every band (the temperature model)
    double f[4];
    band_I0_d3(th.node_c + b * th.ng, th.node_C + b * th.ng, th.ng, rT, f);
    row[b] = f[0];
#pragma unroll
    for (int k = 0; k < 4; ++k) Jrow[k * th.nbp + b] = f[k];
  }
  __syncthreads();
  for (int b = threadIdx.x; b < th.nbo; b += blockDim.x)  // stored bands
    I0cell[P * th.nbo + b] = b < th.nbr ? row[th.band0 + b] : 0.0;
  if (threadIdx.x < 32) {  // the model's sums with the T_p weights
    double m[4] = {0.0, 0.0, 0.0, 0.0};
    for (int b = threadIdx.x; b < th.nbp; b += 32) {
      const double ap = th.a_p[b];
#pragma unroll
      for (int k = 0; k < 4; ++k) m[k] = fma(ap, Jrow[k * th.nbp + b], m[k]);
    }
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
      for (int k = 0; k < 4; ++k) m[k] += __shfl_xor_sync(0xffffffffu, m[k], o);
    }
    if (threadIdx.x == 0)
      for (int k = 0; k < 4; ++k) Msum[4 * P + k] = m[k];
  }
}

// Equilibrium initial state: I = I0_b(T_P) for every direction (stored as the
// deviation I0_b(T_P) - I0_b(T_ref) in the reduced modes).
template <typename S>
__global__ void init_cells_kernel(S* I, double* I0cell, double* J, double* Msum, double* Tp, double* Te, double* TL,
                                  double* EL, const double* Tcells, const double* I0ref, long long cell0, int ncells,
                                  int nd, ThermoTables th) {
  extern __shared__ double row[];  // [nbp]
  for (int c = blockIdx.x; c < ncells; c += gridDim.x) {
    const long long P = cell0 + c;
    const double T = Tcells[c];
    cell_state_at(I0cell, J, Msum, P, T, th, row);
    __syncthreads();
    const long long n = (long long)nd * th.nbo;
    for (long long e = threadIdx.x; e < n; e += blockDim.x) {
      const int b = (int)(e % th.nbo);  // stored band; I0ref holds the stored bands
      const double v = b < th.nbr ? (sizeof(S) == 8 ? row[th.band0 + b] : row[th.band0 + b] - I0ref[b]) : 0.0;
      set_I(I, P * n + e, v);
    }
    if (threadIdx.x == 0) {
      double e = 0.0;
      for (int b = 0; b < th.nbp; ++b) e = fma(th.a_L[b], row[b], e);
      Tp[P] = T;
      Te[P] = T;
      TL[P] = T;
      EL[P] = e;
    }
    __syncthreads();
  }
}

// Thermodynamic state from T_p after a state restore: I0cell, J, T_e.
__global__ void state_from_Tp_kernel(double* I0cell, double* J, double* Msum, const double* Tp, double* Te,
                                     long long ncells, ThermoTables th) {
  extern __shared__ double row[];
  for (long long P = blockIdx.x; P < ncells; P += gridDim.x) {
    cell_state_at(I0cell, J, Msum, P, Tp[P], th, row);
    if (threadIdx.x == 0) Te[P] = Tp[P];
    __syncthreads();
  }
}

// Wall ghost intensities (FP64): one thread per (face, band).
__global__ void wall_I0_kernel(double* I0wall, const double* Tf, long long nfaces, ThermoTables th) {
  const long long n = nfaces * th.nbo;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    const long long f = e / th.nbo;
    const int b = (int)(e - f * th.nbo);
    const int bg = th.band0 + b;
    I0wall[e] = b < th.nbr ? band_I0(th.node_c + bg * th.ng, th.node_C + bg * th.ng, th.ng, 1.0 / Tf[f]) : 0.0;
  }
}

// Deviation ghosts for the reduced modes: I0wall - I0ref as FP32.
__global__ void wall_dev_kernel(float* out, const double* I0wall, const double* I0ref, long long n, int nbp) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
    out[e] = (float)(I0wall[e] - I0ref[e % nbp]);
}

// Lattice temperature: sum_b a_L,b I0_b(T) = E_L per cell (evaluated on
// request).  One warp per cell: the root of the cell's cached cubic model
// of I0_b(T) around T_e (the one the T_p solve keeps) when it lies inside the
// trust radius, else Halley on the exact band quadrature from there (or from
// the guess), bisection as the fallback.
__global__ void solve_TL_kernel(double* TL, const double* EL, const double* Tguess, const double* J,
                                const double* Teval, long long ncells, ThermoTables th, double trust_rel, int maxit,
                                DevCounters* counters) {
  const int warps = blockDim.x / 32, lane = threadIdx.x & 31;
  const int nbp = th.nbp;
  for (long long P = blockIdx.x * (long long)warps + threadIdx.x / 32; P < ncells; P += (long long)gridDim.x * warps) {
    const double E = EL[P];
    if (!isfinite(E)) {
      if (lane == 0) {
        TL[P] = E;
        if (counters) atomicAdd(&counters->nonfinite, 1ULL);
      }
      continue;
    }
    double F[4] = {0.0, 0.0, 0.0, 0.0};
    for (int b = lane; b < nbp; b += 32) {
      const double w = th.a_L[b];
#pragma unroll
      for (int k = 0; k < 4; ++k) F[k] = fma(w, J[(P * 4 + k) * nbp + b], F[k]);
    }
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
      for (int k = 0; k < 4; ++k) F[k] += __shfl_xor_sync(0xffffffffu, F[k], o);
    }
    const double Te = Teval[P];
    const double delta = model_step(F[0] - E, F[1], F[2], F[3]);
    const double Tn = Te + delta;
    if (isfinite(Tn) && fabs(delta) <= trust_rel * Tn) {
      if (lane == 0) TL[P] = Tn;
      continue;
    }
    const double start = (isfinite(Tn) && Tn >= kTmin && Tn <= kTmax) ? Tn : Tguess[P];
    const SolveResult r = exact_solve_warp(th, E, start, trust_rel, maxit, nullptr, th.a_L);
    if (lane == 0) {
      TL[P] = r.Te + r.delta;
      if (counters && r.fallback) atomicAdd(&counters->fallbacks, 1ULL);
      if (counters && r.bad) atomicAdd(&counters->nonfinite, 1ULL);
    }
  }
}

// Cell heat flux q(P) = sum_b sum_d S_d I_{d,b}: one CTA per cell.  A lane holds
// the V bands of one 16-byte vector and takes every (threads / lanes)-th group of
// four rows, (+,+), (-,+), (-,-), (+,-) of one |S|: the four values' sums and
// differences first, then one FMA per axis, 1.5 FP64 operations per value in
// 2-D where S_d I for every direction takes two (the FP64 pipe is the bound).
// The reference part of the reduced modes' storage drops out: sum_d S_d = 0.
// On 128x128 x 400 x 55: 2014 us with one 64-bit division and two FMAs per value.
template <typename S, int V>
__device__ __forceinline__ double vector_sum(const S* p) {  // sum of V consecutive values
  double s = 0.0;
  if constexpr (sizeof(S) == 8) {
    if constexpr (std::is_same<S, FFElem>::value) {
      double a, b;
      ff::to_doubles(ff::ldg(p), a, b);
      s = a + b;
    } else {
      double x[2];
      Tr<double>::ld(p, x);
      s = x[0] + x[1];
    }
  } else {
    float x[V];
    Tr<S>::ld(p, x);
#pragma unroll
    for (int v = 0; v < V; ++v) s += (double)x[v];
  }
  return s;
}

template <typename S, int V, int DIM>
__global__ void __launch_bounds__(256) flux_cells_kernel(const S* I, double* q, const double* Sd, long long cell0,
                                                         int ncells, int nd, int nbp) {
  __shared__ double sh[3][8];
  const int lpc = nbp / V, groups = 256 / lpc, grp = threadIdx.x / lpc, b0 = V * (threadIdx.x - grp * lpc);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int c = blockIdx.x; c < ncells; c += gridDim.x) {
    const S* row = I + (cell0 + c) * (long long)nd * nbp + b0;
    double acc[3] = {0.0, 0.0, 0.0};
    if (grp < groups) {
#pragma unroll 2
      for (int r = 4 * grp; r < nd; r += 4 * groups) {
        double v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = vector_sum<S, V>(row + (r + k) * nbp);
        const double a = v[0] + v[3], b = v[1] + v[2];
        acc[0] = fma(Sd[3 * r], a - b, acc[0]);
        acc[1] = fma(Sd[3 * r + 1], (v[0] - v[3]) + (v[1] - v[2]), acc[1]);
        if (DIM == 3) acc[2] = fma(Sd[3 * r + 2], a + b, acc[2]);
      }
    }
#pragma unroll
    for (int ax = 0; ax < DIM; ++ax) {
      for (int o = 16; o > 0; o >>= 1) acc[ax] += __shfl_xor_sync(0xffffffffu, acc[ax], o);
      if (lane == 0) sh[ax][wid] = acc[ax];
    }
    __syncthreads();
    if (threadIdx.x < DIM) {
      double t = 0.0;
      for (int w = 0; w < 8; ++w) t += sh[threadIdx.x][w];
      q[(long long)c * DIM + threadIdx.x] = t;
    }
    __syncthreads();
  }
}

// Net outgoing flux through every face of every side of a geometry (blockIdx.y: side).
template <typename S>
__global__ void __launch_bounds__(kFluxThreads) flux_faces_kernel(const S* I, const double* I0ref, const double* I0wall,
                                                                  const DevGeom* geoms, int geom, const DirInfo* dirs,
                                                                  const double* Sd, int nd, int nbp, double* face_out,
                                                                  int max_faces) {
  __shared__ double sh[kFluxThreads];
  const DevGeom g = geoms[geom];
  const int side = blockIdx.y;
  const int nfaces = side < 2 ? g.ny * g.nz : (side < 4 ? g.nx * g.nz : g.nx * g.ny);
  for (int f = blockIdx.x; f < nfaces; f += gridDim.x) {
    const double t = face_flux(I, I0ref, I0wall, g, side, f, dirs, Sd, nd, nbp, sh);
    if (threadIdx.x == 0) face_out[(long long)side * max_faces + f] = t;
  }
}

struct SideFaces {
  int n[6];
};
__global__ void mean_kernel(const double* v, int max_faces, SideFaces nf, double* out) {  // a CTA per side
  __shared__ double sh[256];
  const int n = nf.n[blockIdx.x];
  double acc = 0.0;
  for (int e = threadIdx.x; e < n; e += blockDim.x) acc += v[(long long)blockIdx.x * max_faces + e];
  const double t = block_sum(acc, sh);
  if (threadIdx.x == 0) out[blockIdx.x] = t / (double)n;
}

// FP64 [cell][caller's d][nb] <-> internal rows [cell][dir][nbp] (deviation in the
// reduced modes): one CTA per cell, a thread per band walking every
// (threads / nbp)-th direction, so consecutive lanes touch consecutive bands on
// both sides and no index is divided.
template <typename S>
__global__ void __launch_bounds__(256) unpack_kernel(const S* I, double* out, const double* I0ref, const int* perm,
                                                     long long ncells, int nd, int nb, int nbp) {
  const int rows = 256 / nbp, r = threadIdx.x / nbp, b = threadIdx.x - r * nbp;
  if (r >= rows || b >= nb) return;
  for (long long P = blockIdx.x; P < ncells; P += gridDim.x) {
    double* o = out + P * nd * nb + b;
#pragma unroll 8
    for (int d = r; d < nd; d += rows) __stcs(o + (long long)perm[d] * nb, full_I(I, (P * nd + d) * nbp + b, b, I0ref));
  }
}

template <typename S>
__global__ void __launch_bounds__(256) pack_kernel(const double* in, S* I, const double* I0ref, const int* perm,
                                                   long long ncells, int nd, int nb, int nbp) {
  const int rows = 256 / nbp, r = threadIdx.x / nbp, b = threadIdx.x - r * nbp;
  if (r >= rows) return;
  const double ref = sizeof(S) == 8 || b >= nb ? 0.0 : I0ref[b];
  for (long long P = blockIdx.x; P < ncells; P += gridDim.x) {
    const double* x = in + P * nd * nb + b;
#pragma unroll 8
    for (int d = r; d < nd; d += rows) {
      const double v = b < nb ? __ldcs(x + (long long)perm[d] * nb) - ref : 0.0;
      set_I(I, (P * nd + d) * nbp + b, v);
    }
  }
}

// E_L of every cell from its intensity row (used after a state restore).
template <typename S>
__global__ void energy_L_kernel(const S* I, const double* I0ref, double* EL, const double* wdir, long long ncells,
                                int nd, ThermoTables th) {
  extern __shared__ double sh[];
  for (long long P = blockIdx.x; P < ncells; P += gridDim.x) {
    const long long base = P * (long long)nd * th.nbo;
    double acc = 0.0;
    for (int b = threadIdx.x; b < th.nbo; b += blockDim.x) {
      double G = 0.0;
      for (int d = 0; d < nd; ++d) G = fma(wdir[d], full_I(I, base + (long long)d * th.nbo + b, b, I0ref), G);
      acc = fma(G, th.inv_v[b], acc);
    }
    const double t = block_sum(acc, sh);
    if (threadIdx.x == 0) EL[P] = t;
  }
}

// Band sums after a separate sweep (the sweep-ordered pass, the unstructured
// sweep): one CTA of 8 warps per cell.  Warp w sums the directions
// [w nd/8, (w+1) nd/8) for every stored band (lanes over band pairs); the 8
// partials are added in warp order (deterministic) and
// G_b = sum_d w_d I^{k+1}_{d,b} goes to Gc for cells_kernel.
// Within a warp the sums over a run of equal-weight directions are exact
// 64-bit fixed-point additions on the integer pipe (unit 2^(E-50) for the
// cell's I0 of exponent E; a value up to 32 I0 adds at most 2^55, so a run of
// 256 cannot overflow), closed by one FP64 FMA (sum x w x unit).  Values
// beyond that range (or negative, NaN) take the FP64 FMA directly.
// Reduced storage (deviations from I0_b(T_ref)): each lane sums w_d x deviation
// in FP32, flushed to FP64 every 16 directions, and G_b gets W I0_b(T_ref).
constexpr int kRedWarps = 8;

template <typename S>
__device__ __forceinline__ void reduce_dev_warp(const SweepArgs& a, const S* row, int d0, int d1, int lane,
                                                double* gpart_w) {
  const int nbo = a.th.nbo;
  for (int b0 = 2 * lane; b0 < nbo; b0 += 64) {  // two bands per lane
    double G0 = 0.0, G1 = 0.0;
    for (int d = d0; d < d1; d += 16) {  // 16 directions: loads first, then the float sums
      const int m = min(16, d1 - d);
      float x0[16], x1[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        x0[k] = x1[k] = 0.f;
        if (k < m) {
          const S* p = row + (long long)(d + k) * nbo + b0;
          x0[k] = Tr<S>::to_float(p[0]);
          x1[k] = Tr<S>::to_float(p[1]);
        }
      }
      float acc0 = 0.f, acc1 = 0.f;
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const float w = k < m ? a.wdir32[d + k] : 0.f;
        acc0 = fmaf(w, x0[k], acc0);
        acc1 = fmaf(w, x1[k], acc1);
      }
      G0 += (double)acc0;
      G1 += (double)acc1;
    }
    gpart_w[b0] = G0;
    gpart_w[b0 + 1] = G1;
  }
}

template <typename S>
__global__ void __launch_bounds__(256, 4) gs_reduce_kernel(SweepArgs a, long long ncells) {
  extern __shared__ double gpart[];  // [kRedWarps][nbo]
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nbo = a.th.nbo, nd = a.nd, lpc = nbo / 2;
  const int d0 = (int)((long long)wid * nd / kRedWarps), d1 = (int)((long long)(wid + 1) * nd / kRedWarps);
  for (long long P = blockIdx.x; P < ncells; P += gridDim.x) {
    if constexpr (sizeof(S) != 8) {
      reduce_dev_warp<S>(a, reinterpret_cast<const S*>(a.Iout) + P * (long long)nd * nbo, d0, d1, lane, gpart + wid * nbo);
    } else {
    const double* row = reinterpret_cast<const double*>(a.Iout) + P * (long long)nd * nbo;
    for (int lp = lane; lp < lpc; lp += 32) {
      const int b0 = 2 * lp;
      double G[2] = {0.0, 0.0};
      unsigned long long facc[2] = {0ull, 0ull};
      long long fsc[2];
      int fe0[2];
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        const int e0 = (int)((unsigned long long)__double_as_longlong(a.I0cell[P * nbo + b0 + v]) >> 52);
        const bool on = e0 >= 200 && e0 <= 1900;
        fe0[v] = on ? e0 + 4 : -1;
        fsc[v] = on ? (long long)(e0 - 1073) * (1LL << 52) : 0;
      }
      long long wrun = d0 < d1 ? __double_as_longlong(a.wdir[d0]) : 0;
      int nrun = 0;
      auto add = [&](double2 x, int d) {
        const long long wb = __double_as_longlong(a.wdir[d]);
        if (wb != wrun || nrun == 256) {  // close the run: sum x (w x unit)
#pragma unroll
          for (int v = 0; v < 2; ++v) {
            if (facc[v] != 0ull) G[v] = fma(__ull2double_rn(facc[v]), __longlong_as_double(wrun + fsc[v]), G[v]);
            facc[v] = 0ull;
          }
          wrun = wb;
          nrun = 0;
        }
        ++nrun;
        const double xv[2] = {x.x, x.y};
        bool big = false;
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          const unsigned long long rb = (unsigned long long)__double_as_longlong(xv[v]);
          const int e = (int)(rb >> 52);  // sign bit included: negative values take the FP64 path
          const unsigned long long m = ((rb & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull) << 2;
          const int sh = e == 0 ? 63 : min(fe0[v] - e, 63);  // zero (and subnormal) adds nothing
          facc[v] += sh >= 0 ? (m >> sh) : 0ull;
          big |= sh < 0;
        }
        // rare: a value beyond the fixed-point range (a warp-uniform branch, so
        // no FP64 instruction is issued in the common case)
        if (__any_sync(__activemask(), big)) {
#pragma unroll
          for (int v = 0; v < 2; ++v) {
            const int e = (int)((unsigned long long)__double_as_longlong(xv[v]) >> 52);
            if (e != 0 && fe0[v] - e < 0) G[v] = fma(a.wdir[d], xv[v], G[v]);
          }
        }
      };
      int d = d0;
      for (; d + 4 <= d1; d += 4) {
        double2 x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = __ldcs(reinterpret_cast<const double2*>(row + (long long)(d + u) * nbo + b0));
#pragma unroll
        for (int u = 0; u < 4; ++u) add(x[u], d + u);
      }
      for (; d < d1; ++d) add(__ldcs(reinterpret_cast<const double2*>(row + (long long)d * nbo + b0)), d);
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        if (facc[v] != 0ull) G[v] = fma(__ull2double_rn(facc[v]), __longlong_as_double(wrun + fsc[v]), G[v]);
        gpart[wid * nbo + b0 + v] = G[v];
      }
    }
    }
    __syncthreads();
    for (int b = threadIdx.x; b < nbo; b += blockDim.x) {
      double G = gpart[b];
      for (int w = 1; w < kRedWarps; ++w) G += gpart[w * nbo + b];
      if constexpr (sizeof(S) != 8) G = fma(a.Wtot, a.I0ref[b], G);  // the reference part, sum_d w_d I0_b(T_ref)
      a.Gc[P * nbo + b] = G;
    }
    __syncthreads();
  }
}

// Wall ghosts of one side of one geometry from the wall cells' current iterate:
// one CTA of 256 threads per face.  Bound by the FP64 pipe (one FMA per
// outgoing direction and band) and, below a few hundred faces, by the latency
// of one face, so a face's directions are spread over the CTA: lane l of group
// g holds the V bands of one 16-byte vector and sums the outgoing directions
// g, g + groups, ... of the side's list (WallDirs, built on the host with the
// two weight sums, so no thread walks or tests all directions), four loads in
// flight; the groups' partials are added in order in shared memory.  One warp
// per face walking every direction, each thread forming the weight sum again,
// took 280 us (diffuse) and 204 us (partially specular) on the 67 faces of a
// 67x45 grid with 400 directions x 55 bands; this form takes 8-9 us.
// Reduced modes sum the stored deviations: the reference part of the ratio is
// I0_b(T_ref) (sum_out - sum_in) / sum_in.
constexpr int kWallThreads = 256;

template <typename S>
struct WallArgs {
  const S* I;
  const double* I0ref;
  const DevGeom* geoms;
  const double* Sd;
  int geom, side, nd, nbp, nfaces;
  WallDirs wd;
};

__device__ __forceinline__ long long wall_cell(const DevGeom& g, int side, int f) {
  const int ax = side >> 1;
  const bool high = side & 1;
  int i, j, k;  // wall cell of face f (x sides: j + ny k, y sides: i + nx k, z sides: i + nx j)
  if (ax == 0) { i = high ? g.nx - 1 : 0; j = f % g.ny; k = f / g.ny; }
  else if (ax == 1) { j = high ? g.ny - 1 : 0; i = f % g.nx; k = f / g.nx; }
  else { k = high ? g.nz - 1 : 0; i = f % g.nx; j = f / g.nx; }
  return g.cell0 + ((long long)k * g.ny + j) * g.nx + i;
}

// D[b] = sum_out |S_ax| I_b / sum_in |S_ax| of the cell whose row is given (a
// deviation in the reduced modes).  Every thread calls it; D is complete on return.
template <typename S>
__device__ __forceinline__ void wall_diffuse(const WallArgs<S>& w, const S* row, double* part, double* D) {
  using T = Tr<S>;
  constexpr int V = T::V;
  const int lpc = w.nbp / V, groups = kWallThreads / lpc;
  const int grp = threadIdx.x / lpc, b0 = V * (threadIdx.x - grp * lpc);
  const int ax = w.side >> 1;
  if (grp < groups) {
    double acc[V];
#pragma unroll
    for (int v = 0; v < V; ++v) acc[v] = 0.0;
    int k = grp;
    for (; k + 3 * groups < w.wd.nout; k += 4 * groups) {
      typename T::A x[4][V];
      double sd[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int d = w.wd.out[k + u * groups];
        sd[u] = fabs(w.Sd[3 * d + ax]);
        T::ld(row + (long long)d * w.nbp + b0, x[u]);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < V; ++v) acc[v] = fma(sd[u], (double)x[u][v], acc[v]);
    }
    for (; k < w.wd.nout; k += groups) {
      const int d = w.wd.out[k];
      const double sd = fabs(w.Sd[3 * d + ax]);
      typename T::A x[V];
      T::ld(row + (long long)d * w.nbp + b0, x);
#pragma unroll
      for (int v = 0; v < V; ++v) acc[v] = fma(sd, (double)x[v], acc[v]);
    }
#pragma unroll
    for (int v = 0; v < V; ++v) part[grp * w.nbp + b0 + v] = acc[v];
  }
  __syncthreads();
  for (int b = threadIdx.x; b < w.nbp; b += kWallThreads) {
    double num = part[b];
    for (int g = 1; g < groups; ++g) num += part[g * w.nbp + b];
    if constexpr (sizeof(S) != 8) num = fma(w.wd.sum_out - w.wd.sum_in, w.I0ref[b], num);
    D[b] = num / w.wd.sum_in;
  }
  __syncthreads();
}

// Diffuse side: the FP64 ghost row of every face (and the FP32 deviation row in
// the reduced modes).
template <typename S>
__global__ void __launch_bounds__(kWallThreads) diffuse_ghost_kernel(WallArgs<S> w, double* I0wall, float* I0wall_dev) {
  extern __shared__ double part[];  // [groups][nbp], then D [nbp]
  double* D = part + (kWallThreads / (w.nbp / Tr<S>::V)) * w.nbp;
  const DevGeom g = w.geoms[w.geom];
  for (int f = blockIdx.x; f < w.nfaces; f += gridDim.x) {
    wall_diffuse<S>(w, w.I + wall_cell(g, w.side, f) * ((long long)w.nd * w.nbp), part, D);
    for (int b = threadIdx.x; b < w.nbp; b += kWallThreads) {
      const long long e = (g.face0[w.side] + f) * w.nbp + b;
      if constexpr (sizeof(S) == 8) {
        I0wall[e] = D[b];
      } else {
        I0wall[e] = w.I0ref[b] + D[b];
        I0wall_dev[e] = (float)D[b];
      }
    }
    __syncthreads();
  }
}

// Partially specular side: for every direction that enters through it (or runs
// along it) and every band, the ghost p I(mirror of d) + (1 - p) D_b, in the
// storage type (a deviation from I0_b(T_ref) in the reduced modes).  Rows of
// outgoing directions are never read and stay as they are.
template <typename S>
__global__ void __launch_bounds__(kWallThreads) partial_ghost_kernel(WallArgs<S> w, const DirInfo* dirs, double p,
                                                                     S* out) {
  using T = Tr<S>;
  constexpr int V = T::V;
  extern __shared__ double part[];  // [groups][nbp], then D [nbp]
  const int lpc = w.nbp / V, groups = kWallThreads / lpc;
  const int grp = threadIdx.x / lpc, b0 = V * (threadIdx.x - grp * lpc);
  const int ax = w.side >> 1;
  double* D = part + groups * w.nbp;
  const DevGeom g = w.geoms[w.geom];
  const long long row = (long long)w.nd * w.nbp;
  for (int f = blockIdx.x; f < w.nfaces; f += gridDim.x) {
    const S* cell = w.I + wall_cell(g, w.side, f) * row;
    wall_diffuse<S>(w, cell, part, D);
    if (grp < groups) {
      double q[V];
#pragma unroll
      for (int v = 0; v < V; ++v) q[v] = (1.0 - p) * D[b0 + v];
#pragma unroll 4
      for (int k = grp; k < w.nd - w.wd.nout; k += groups) {
        const int d = w.wd.rest[k];
        const int r = ax == 0 ? dirs[d].rx : (ax == 1 ? dirs[d].ry : dirs[d].rz);
        typename T::A x[V];
        T::ld(cell + (long long)r * w.nbp + b0, x);
#pragma unroll
        for (int v = 0; v < V; ++v) x[v] = (typename T::A)fma(p, (double)x[v], q[v]);
        T::st(out + f * row + (long long)d * w.nbp + b0, x);
      }
    }
    __syncthreads();
  }
}

inline int grid_for(long long n, int threads) {
  long long g = (n + threads - 1) / threads;
  if (g > 152LL * 64) g = 152LL * 64;
  return (int)(g < 1 ? 1 : g);
}

inline int cell_grid(long long ncells) { return (int)(ncells < 152 * 16 ? (ncells < 1 ? 1 : ncells) : 152 * 16); }

}  // namespace

int values_per_lane(int precision) { return precision == 0 ? 2 : (precision == 1 ? 4 : 8); }

cudaError_t launch_sweep(int precision, int pd, const SweepArgs& a, int dim, int threads, int grid, cudaStream_t s) {
  if (precision == 0) return launch_sweep_fp64(a, dim, threads, grid, s);
  if (precision == 1) return launch_sweep_fp32(a, dim, threads, grid, s);
  return launch_sweep_bf16(pd, a, dim, threads, grid, s);
}

namespace {
template <typename S>
WallArgs<S> wall_args(const void* I, const double* I0ref, const DevGeom* geoms, int geom, int side, const double* Sd,
                      const WallDirs& wd, int nd, int nbp, int nfaces) {
  return WallArgs<S>{(const S*)I, I0ref, geoms, Sd, geom, side, nd, nbp, nfaces, wd};
}
template <typename S>
size_t wall_smem(int nbp) {
  return (size_t)(kWallThreads / (nbp / Tr<S>::V) + 1) * nbp * sizeof(double);
}
}  // namespace

cudaError_t launch_diffuse_ghosts(int precision, const void* I, const double* I0ref, double* I0wall, float* I0wall_dev,
                                  const DevGeom* geoms, int geom, int side, const double* Sd, const WallDirs& wd, int nd,
                                  int nbp, int nfaces, cudaStream_t s) {
  const int grid = (int)std::min<long long>(std::max(nfaces, 1), 152LL * 16);
  auto go = [&](auto tag) {
    using S = decltype(tag);
    diffuse_ghost_kernel<S><<<grid, kWallThreads, wall_smem<S>(nbp), s>>>(
        wall_args<S>(I, I0ref, geoms, geom, side, Sd, wd, nd, nbp, nfaces), I0wall, I0wall_dev);
  };
  if (precision == 0) go(double{});
  else if (precision == 1) go(float{});
  else go(__nv_bfloat16{});
  return cudaGetLastError();
}

cudaError_t launch_partial_ghosts(int precision, const void* I, const double* I0ref, const DevGeom* geoms, int geom,
                                  int side, const double* Sd, const WallDirs& wd, const DirInfo* dirs, int nd, int nbp,
                                  int nfaces, double p, void* out, cudaStream_t s) {
  const int grid = (int)std::min<long long>(std::max(nfaces, 1), 152LL * 16);
  auto go = [&](auto tag) {
    using S = decltype(tag);
    partial_ghost_kernel<S><<<grid, kWallThreads, wall_smem<S>(nbp), s>>>(
        wall_args<S>(I, I0ref, geoms, geom, side, Sd, wd, nd, nbp, nfaces), dirs, p, (S*)out);
  };
  if (precision == 0) go(double{});
  else if (precision == 1) go(float{});
  else go(__nv_bfloat16{});
  return cudaGetLastError();
}

cudaError_t launch_gs_reduce(int precision, const SweepArgs& a, long long ncells, cudaStream_t s) {
  const int grid = (int)std::min<long long>(std::max(ncells, 1LL), 152LL * 64);
  const size_t sm = (size_t)kRedWarps * a.th.nbo * sizeof(double);
  if (precision == 0) gs_reduce_kernel<double><<<grid, 32 * kRedWarps, sm, s>>>(a, ncells);
  else if (precision == 1) gs_reduce_kernel<float><<<grid, 32 * kRedWarps, sm, s>>>(a, ncells);
  else gs_reduce_kernel<__nv_bfloat16><<<grid, 32 * kRedWarps, sm, s>>>(a, ncells);
  return cudaGetLastError();
}

cudaError_t launch_init_cells(int precision, bool state_ff, void* I, double* I0cell, double* J, double* Msum, double* Tp,
                              double* Te, double* TL, double* EL, const double* Tcells, const double* I0ref,
                              long long cell0, int ncells, int nd, ThermoTables th, cudaStream_t s) {
  auto go = [&](auto tag) {
    using T = decltype(tag);
    init_cells_kernel<T><<<cell_grid(ncells), 256, th.nbp * sizeof(double), s>>>((T*)I, I0cell, J, Msum, Tp, Te, TL, EL, Tcells,
                                                                                 I0ref, cell0, ncells, nd, th);
  };
  if (precision == 0 && state_ff) go(FFElem{});
  else if (precision == 0) go(double{});
  else if (precision == 1) go(float{});
  else go(__nv_bfloat16{});
  return cudaGetLastError();
}

cudaError_t launch_state_from_Tp(double* I0cell, double* J, double* Msum, const double* Tp, double* Te,
                                 long long ncells, ThermoTables th, cudaStream_t s) {
  state_from_Tp_kernel<<<cell_grid(ncells), 64, th.nbp * sizeof(double), s>>>(I0cell, J, Msum, Tp, Te, ncells,
                                                                               th);  // row: all bands
  return cudaGetLastError();
}

cudaError_t launch_wall_I0(double* I0wall, const double* Tfaces, long long nfaces, ThermoTables th, cudaStream_t s) {
  wall_I0_kernel<<<grid_for(nfaces * th.nbo, 256), 256, 0, s>>>(I0wall, Tfaces, nfaces, th);
  return cudaGetLastError();
}

cudaError_t launch_wall_dev(float* out, const double* I0wall, const double* I0ref, long long nfaces, int nbp,
                            cudaStream_t s) {
  wall_dev_kernel<<<grid_for(nfaces * nbp, 256), 256, 0, s>>>(out, I0wall, I0ref, nfaces * nbp, nbp);
  return cudaGetLastError();
}

cudaError_t launch_solve_TL(double* TL, const double* EL, const double* Tguess, const double* J, const double* Teval,
                            long long ncells, ThermoTables th, double trust_rel, int maxit, DevCounters* counters,
                            cudaStream_t s) {
  solve_TL_kernel<<<cell_grid(ncells / 4 + 1), 128, 0, s>>>(TL, EL, Tguess, J, Teval, ncells, th, trust_rel, maxit,
                                                            counters);
  return cudaGetLastError();
}

cudaError_t launch_flux_cells(int precision, bool state_ff, const void* I, double* q, const double* S, long long cell0,
                              int ncells, int nd, int nbp, int dim, cudaStream_t s) {
  const int grid = cell_grid(ncells);
  auto go = [&](auto tag, auto vec) {
    using T = decltype(tag);
    constexpr int V = decltype(vec)::value;
    if (dim == 3) flux_cells_kernel<T, V, 3><<<grid, 256, 0, s>>>((const T*)I, q, S, cell0, ncells, nd, nbp);
    else flux_cells_kernel<T, V, 2><<<grid, 256, 0, s>>>((const T*)I, q, S, cell0, ncells, nd, nbp);
  };
  if (precision == 0 && state_ff) go(FFElem{}, std::integral_constant<int, 2>{});
  else if (precision == 0) go(double{}, std::integral_constant<int, 2>{});
  else if (precision == 1) go(float{}, std::integral_constant<int, 4>{});
  else go(__nv_bfloat16{}, std::integral_constant<int, 8>{});
  return cudaGetLastError();
}

cudaError_t launch_flux_walls(int precision, bool state_ff, const void* I, const double* I0ref, const double* I0wall,
                              const DevGeom* geoms, int geom, const DirInfo* dirs, const double* S, int nd, int nbp,
                              double* face_out, int max_faces, const int (&nfaces)[6], int nsides, double* out,
                              cudaStream_t s) {
  int most = 1;
  SideFaces nf{};
  for (int k = 0; k < nsides; ++k) {
    nf.n[k] = nfaces[k];
    most = std::max(most, nfaces[k]);
  }
  const dim3 grid(cell_grid(most), nsides);
  auto go = [&](auto tag) {
    using T = decltype(tag);
    flux_faces_kernel<T><<<grid, kFluxThreads, 0, s>>>((const T*)I, I0ref, I0wall, geoms, geom, dirs, S, nd, nbp, face_out,
                                                       max_faces);
  };
  if (precision == 0 && state_ff) go(FFElem{});
  else if (precision == 0) go(double{});
  else if (precision == 1) go(float{});
  else go(__nv_bfloat16{});
  mean_kernel<<<nsides, 256, 0, s>>>(face_out, max_faces, nf, out);
  return cudaGetLastError();
}

namespace {
__global__ void ff_to_doubles_kernel(ulonglong2* buf, long long npairs) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < npairs; i += (long long)gridDim.x * blockDim.x) {
    const ulonglong2 v = buf[i];
    double a, b;
    ff::to_doubles(ff::P2{v.x, v.y}, a, b);
    buf[i] = make_ulonglong2((unsigned long long)__double_as_longlong(a), (unsigned long long)__double_as_longlong(b));
  }
}
__global__ void doubles_to_ff_kernel(const double2* src, ulonglong2* dst, long long npairs) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < npairs; i += (long long)gridDim.x * blockDim.x) {
    const double2 v = src[i];
    const ff::P2 p = ff::from_doubles(v.x, v.y);
    dst[i] = make_ulonglong2(p.h, p.l);
  }
}
}  // namespace

cudaError_t launch_doubles_to_ff(const void* src, void* dst, long long npairs, cudaStream_t s) {
  if (npairs <= 0) return cudaSuccess;
  doubles_to_ff_kernel<<<grid_for(npairs, 256), 256, 0, s>>>(reinterpret_cast<const double2*>(src),
                                                             reinterpret_cast<ulonglong2*>(dst), npairs);
  return cudaGetLastError();
}

cudaError_t launch_ff_to_doubles(void* buf, long long npairs, cudaStream_t s) {
  if (npairs <= 0) return cudaSuccess;
  ff_to_doubles_kernel<<<grid_for(npairs, 256), 256, 0, s>>>(reinterpret_cast<ulonglong2*>(buf), npairs);
  return cudaGetLastError();
}

cudaError_t launch_unpack(int precision, bool state_ff, const void* I, double* out, const double* I0ref, const int* perm,
                          long long ncells, int nd, int nb, int nbp, cudaStream_t s) {
  auto go = [&](auto tag) {
    using T = decltype(tag);
    unpack_kernel<T><<<cell_grid(ncells), 256, 0, s>>>((const T*)I, out, I0ref, perm, ncells, nd, nb, nbp);
  };
  if (precision == 0 && state_ff) go(FFElem{});
  else if (precision == 0) go(double{});
  else if (precision == 1) go(float{});
  else go(__nv_bfloat16{});
  return cudaGetLastError();
}

cudaError_t launch_pack(int precision, bool state_ff, const double* in, void* I, const double* I0ref, const int* perm,
                        long long ncells, int nd, int nb, int nbp, cudaStream_t s) {
  auto go = [&](auto tag) {
    using T = decltype(tag);
    pack_kernel<T><<<cell_grid(ncells), 256, 0, s>>>(in, (T*)I, I0ref, perm, ncells, nd, nb, nbp);
  };
  if (precision == 0 && state_ff) go(FFElem{});
  else if (precision == 0) go(double{});
  else if (precision == 1) go(float{});
  else go(__nv_bfloat16{});
  return cudaGetLastError();
}

cudaError_t launch_energy_L(int precision, bool state_ff, const void* I, const double* I0ref, double* EL, const double* wdir,
                            long long ncells, int nd, ThermoTables th, cudaStream_t s) {
  auto go = [&](auto tag) {
    using T = decltype(tag);
    energy_L_kernel<T><<<cell_grid(ncells), 64, 64 * sizeof(double), s>>>((const T*)I, I0ref, EL, wdir, ncells, nd, th);
  };
  if (precision == 0 && state_ff) go(FFElem{});
  else if (precision == 0) go(double{});
  else if (precision == 1) go(float{});
  else go(__nv_bfloat16{});
  return cudaGetLastError();
}

}  // namespace bte
