// bte_kernels.cu -- CUDA kernels around the sweep (sm_103a).  The sweeps (upwind
// update, walls, band sums; Sec. 3.1, Eq. 4-6) live in bte_sweep.cuh and
// bte_rows.cuh, the per-cell T_p step in bte_cells.cu.  Here:
//   gs_reduce_kernel    energies after a sweep-ordered pass (bte_gs.cu) or an
//                       unstructured sweep;
//   init_cells / state_from_Tp / wall_I0 / wall_dev
//                       equilibrium state, cached models and Eq. 6 ghosts;
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
// with its T_p and T_L sums, T_e = T_p = T.  One CTA per cell (grid-stride); bands
// over threads.
__device__ void cell_state_at(double* I0cell, double* J, double* Msum, double* MsumL, long long P, double T,
                              ThermoTables th, double* row) {
  const double rT = rcp_pos(T);
  double* Jrow = J + (P * 4) * th.nbp;
  for (int b = threadIdx.x; b < th.nbp; b += blockDim.x) {  // every band (the temperature model)
    double f[4];
    band_taylor(th.node_c + b * th.ng, th.node_C + b * th.ng, th.ng, rT, f);
    row[b] = f[0];
#pragma unroll
    for (int k = 0; k < 4; ++k) Jrow[k * th.nbp + b] = f[k];
  }
  __syncthreads();
  for (int b = threadIdx.x; b < th.nbo; b += blockDim.x)  // stored bands
    I0cell[P * th.nbo + b] = b < th.nbr ? row[th.band0 + b] : 0.0;
  if (threadIdx.x < 64) {  // the model's sums: warp 0 with the T_p weights, warp 1 with T_L's
    const int lane = threadIdx.x & 31;
    const double* wt = threadIdx.x < 32 ? th.a_p : th.a_L;
    double m[4] = {0.0, 0.0, 0.0, 0.0};
    for (int b = lane; b < th.nbp; b += 32) {
      const double ap = wt[b];
#pragma unroll
      for (int k = 0; k < 4; ++k) m[k] = fma(ap, Jrow[k * th.nbp + b], m[k]);
    }
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
      for (int k = 0; k < 4; ++k) m[k] += __shfl_xor_sync(0xffffffffu, m[k], o);
    }
    if (lane == 0)
      for (int k = 0; k < 4; ++k) (threadIdx.x < 32 ? Msum : MsumL)[4 * P + k] = m[k];
  }
}

// One row of stored bands (less ref in the reduced modes) into every direction of a cell: a
// thread keeps one pair of bands and walks the rows (16-byte stores in FP64).
template <typename S>
__device__ __forceinline__ void fill_cell(S* cell, const double* row, const double* ref, int nd, int nbo, int nbr) {
  const int pairs = nbo / 2, groups = (int)blockDim.x / pairs;
  const int grp = groups ? threadIdx.x / pairs : 0;
  for (int p = threadIdx.x - grp * pairs; grp < max(groups, 1) && p < pairs; p += groups ? pairs : blockDim.x) {
    double v[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int b = 2 * p + k;
      v[k] = b < nbr ? (sizeof(S) == 8 ? row[b] : row[b] - ref[b]) : 0.0;
    }
    for (int r = grp; r < nd; r += max(groups, 1)) st_pair(cell + (long long)r * nbo + 2 * p, v[0], v[1]);
  }
}

// Equilibrium initial state: I = I0_b(T_P) for every direction (stored as the
// deviation I0_b(T_P) - I0_b(T_ref) in the reduced modes).
template <typename S>
__global__ void init_cells_kernel(S* I, double* I0cell, double* J, double* Msum, double* MsumL, double* Tp, double* Te, double* TL,
                                  double* EL, const double* Tcells, const double* I0ref, long long cell0, int ncells,
                                  int nd, ThermoTables th) {
  extern __shared__ double row[];  // [nbp]
  for (int c = blockIdx.x; c < ncells; c += gridDim.x) {
    const long long P = cell0 + c;
    const double T = Tcells[c];
    cell_state_at(I0cell, J, Msum, MsumL, P, T, th, row);
    __syncthreads();
    fill_cell(I + P * (long long)nd * th.nbo, row + th.band0, I0ref, nd, th.nbo, th.nbr);  // I0ref: the stored bands
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

// The intensities of an FP64 initial state again, from I0cell, in another form.
template <typename S>
__global__ void __launch_bounds__(256) refill_kernel(S* I, const double* I0cell, long long ncells, int nd, int nbo) {
  for (long long P = blockIdx.x; P < ncells; P += gridDim.x)
    fill_cell(I + P * (long long)nd * nbo, I0cell + P * nbo, nullptr, nd, nbo, nbo);
}

// Thermodynamic state from T_p after a state restore: I0cell, J, T_e.
__global__ void state_from_Tp_kernel(double* I0cell, double* J, double* Msum, double* MsumL, const double* Tp, double* Te,
                                     long long ncells, ThermoTables th) {
  extern __shared__ double row[];
  for (long long P = blockIdx.x; P < ncells; P += gridDim.x) {
    cell_state_at(I0cell, J, Msum, MsumL, P, Tp[P], th, row);
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

// Cell heat flux q(P) = sum_b sum_d S_d I_{d,b}: one CTA per cell.  A lane holds
// the V bands of one 16-byte vector and takes every (threads / lanes)-th group of
// four rows, (+,+), (-,+), (-,-), (+,-) of one |S|: the four values' sums and
// differences first, then one FMA per axis, 1.5 FP64 operations per value in
// 2-D where S_d I for every direction takes two (the FP64 pipe is the bound).
// The reference part of the reduced modes' storage drops out: sum_d S_d = 0.
// On 128x128 x 400 x 55: 2014 us with one 64-bit division and two FMAs per value.
template <typename S, int V>
struct Vec {  // V consecutive values, loaded and summed
  typename RawPair<S>::R x[V / 2];
  __device__ __forceinline__ void load(const S* p) {
    const uint4 w = __ldg(reinterpret_cast<const uint4*>(p));
    memcpy(x, &w, 16);
  }
  __device__ __forceinline__ double sum() const {
    double s = 0.0;
#pragma unroll
    for (int v = 0; v < V / 2; ++v) {
      double a, b;
      raw_pair(x[v], a, b);
      s = v ? (s + a) + b : a + b;
    }
    return s;
  }
};

template <typename S, int V, int DIM, bool GROUPED>
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
        Vec<S, V> x[4];
        double v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) x[k].load(row + (r + k) * nbp);
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = x[k].sum();
        if constexpr (!GROUPED) {  // any order: every row by its own S
#pragma unroll
          for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int ax = 0; ax < DIM; ++ax) acc[ax] = fma(Sd[3 * (r + k) + ax], v[k], acc[ax]);
          continue;
        }
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
struct SideDirs {
  WallDirs d[6];
};
template <typename S>
__global__ void __launch_bounds__(kFluxThreads) flux_faces_kernel(const S* I, const double* I0ref, const double* I0wall,
                                                                  const DevGeom* geoms, int geom, SideDirs wd,
                                                                  const double* Sd, int nd, int nbp, double* face_out,
                                                                  int max_faces) {
  __shared__ double sh[kFluxThreads];
  const DevGeom g = geoms[geom];
  const int side = blockIdx.y;
  const int nfaces = side < 2 ? g.ny * g.nz : (side < 4 ? g.nx * g.nz : g.nx * g.ny);
  for (int f = blockIdx.x; f < nfaces; f += gridDim.x) {
    const double t = face_flux(I, I0ref, I0wall, g, side, f, wd.d[side], Sd, nd, nbp, sh);
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
// reduced modes): one CTA of 8 warps per cell, a warp per row.  On the internal
// side a lane holds a pair of bands (16 bytes in FP64), on the caller's side the
// warp touches 32 consecutive doubles at a time (rows of nb doubles start at any
// multiple of 8 bytes), shuffles in between; four rows in flight.  The CTA walks
// the caller's order (row[d]: its internal row), whose rows share 32-byte sectors;
// internal rows are whole sectors and may be scattered.  Bound by HBM:
// 16 bytes per FP64 value.  A thread per band with 8-byte accesses on both sides
// took 494 us (out) on 96x64 x 400 x 55 values from ff pairs; 409 here, where their
// conversions issue most instructions, and 330 from doubles.
template <typename S>
__global__ void __launch_bounds__(256) unpack_kernel(const S* I, double* out, const double* I0ref, const int* rows,
                                                     long long ncells, int nd, int nb, int nbp) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int dlo = wid * nd / 8, dhi = (wid + 1) * nd / 8;
  for (long long P = blockIdx.x; P < ncells; P += gridDim.x) {
    const S* row = I + P * (long long)nd * nbp;
    double* o = out + P * nd * nb;
    for (int c = 0; c < nbp; c += 64) {  // 64 bands at a time
      const int b = c + 2 * lane;
      double r0 = 0.0, r1 = 0.0;
      if (sizeof(S) != 8 && b < nbp) {
        r0 = I0ref[b];
        r1 = I0ref[b + 1];
      }
      for (int d0 = dlo; d0 < dhi; d0 += 4) {
        typename RawPair<S>::R x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)  // lanes and rows past the end repeat the last one's
          x[u] = ld_raw(row + (long long)rows[min(d0 + u, dhi - 1)] * nbp + min(b, nbp - 2));
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (d0 + u >= dhi) break;
          double x0, x1;
          raw_pair(x[u], x0, x1);
          double* q = o + (long long)(d0 + u) * nb + c;
#pragma unroll
          for (int h = 0; h < 2; ++h) {  // elements 32 h + lane of the 64
            const int src = 16 * h + (lane >> 1);
            const double v0 = __shfl_sync(0xffffffffu, sizeof(S) != 8 ? x0 + r0 : x0, src);
            const double v1 = __shfl_sync(0xffffffffu, sizeof(S) != 8 ? x1 + r1 : x1, src);
            if (c + 32 * h + lane < nb) __stcs(q + 32 * h + lane, (lane & 1) ? v1 : v0);
          }
        }
      }
    }
  }
}

// Energies after a separate sweep (the sweep-ordered pass, the unstructured sweep):
// one CTA of 8 warps per cell.  Loads of 16 bytes, eight in
// flight; FP64: four, warp w sums the directions [w nd / 8, (w + 1) nd / 8), lanes over
// band pairs (whole warps on one direction, so the runs of the fixed-point sums
// close together: groups of 28 lanes took 406 us where this took 308 on 6144 cells
// x 400 x 55), their weights loaded with them: loaded behind them, each value's sum
// waited for its own (ten sweep-ordered iterations of 128x128 x 400 x 55 31.6 ms, 30.1
// so; of 6144 triangles 12.6 and 12.0); reduced storage: lanes over the V bands of a vector, 256 V / nbp
// groups.  The partials are added in order (deterministic) to G_b = sum_d w_d I_{d,b};
// warp 0 leaves kRedEntries partial energies in Ec for cells_kernel.  Bound by the
// loads' latency and HBM, 8 bytes per FP64 value.
// FP64: sums over a run of equal-weight directions are 64-bit fixed-point additions
// on the integer pipe (unit 2^(E-50) for the cell's I0 of exponent E; terms are cut
// to whole units, less than one each; a value up to 32 I0 adds at most 2^55, so a run of
// 256 cannot overflow), closed by one FP64 FMA (sum x w x unit).  Values beyond that range (or negative, NaN) take
// the FP64 FMA directly.
// Reduced storage (deviations from I0_b(T_ref)): each lane sums w_d x deviation in
// FP32, added to a double-float sum every 16 directions (FP64 conversions and adds
// there kept the FP64 pipe busy), and G_b gets W I0_b(T_ref).
constexpr int kRedThreads = 256;

struct FixedSum {
  unsigned long long f[2];
  double G[2];
  long long fsc[2], w;
  int fe0[2], n;
  __device__ explicit FixedSum(const double* i0) : f{0ull, 0ull}, G{0.0, 0.0}, w(0), n(0) {
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const int e0 = (int)((unsigned long long)__double_as_longlong(i0[v]) >> 52);
      const bool on = e0 >= 200 && e0 <= 1900;
      fe0[v] = on ? e0 + 4 : -1;
      fsc[v] = on ? (long long)(e0 - 1073) * (1LL << 52) : 0;
    }
  }
  __device__ void close() {
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      if (f[v] != 0ull) G[v] = fma(__ull2double_rn(f[v]), __longlong_as_double(w + fsc[v]), G[v]);
      f[v] = 0ull;
    }
    n = 0;
  }
  __device__ void add(double x0, double x1, double wd) {
    const long long wb = __double_as_longlong(wd);
    if (wb != w || n == 256) {
      close();
      w = wb;
    }
    ++n;
    const double xv[2] = {x0, x1};
    bool big = false;
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const unsigned long long rb = (unsigned long long)__double_as_longlong(xv[v]);
      const int e = (int)(rb >> 52);  // sign bit included: negative values take the FP64 path
      const unsigned long long m = ((rb & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull) << 2;
      const int sh = e == 0 ? 63 : min(fe0[v] - e, 63);  // zero (and subnormal) adds nothing
      f[v] += sh >= 0 ? (m >> sh) : 0ull;
      big |= sh < 0;
    }
    // rare: a value beyond the fixed-point range (a warp-uniform branch, so no
    // FP64 instruction is issued in the common case)
    if (__any_sync(__activemask(), big)) {
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        const int e = (int)((unsigned long long)__double_as_longlong(xv[v]) >> 52);
        if (e != 0 && fe0[v] - e < 0) G[v] = fma(wd, xv[v], G[v]);
      }
    }
  }
};

// Warp 0: the parts' band sums added in order, then kRedEntries partial energies of cell P.
template <bool DEV>
__device__ __forceinline__ void reduce_energies(const SweepArgs& a, const double* gpart, int parts, long long P) {
  const int nbo = a.th.nbo;
  double el = 0.0, ep = 0.0;
  for (int b = threadIdx.x; b < nbo; b += 32) {
    double G = gpart[b];
    for (int w = 1; w < parts; ++w) G += gpart[w * nbo + b];
    if constexpr (DEV) G = fma(a.Wtot, a.I0ref[b], G);  // the reference part, sum_d w_d I0_b(T_ref)
    el = fma(G, a.th.inv_v[b], el);
    ep = fma(G, a.th.binv_v[b], ep);
  }
  for (int o = 16; o >= kRedEntries; o >>= 1) {
    el += __shfl_xor_sync(0xffffffffu, el, o);
    ep += __shfl_xor_sync(0xffffffffu, ep, o);
  }
  if (threadIdx.x < kRedEntries) a.Ec[P * kRedEntries + threadIdx.x] = make_double2(el, ep);
}

template <typename S, int V>
__global__ void __launch_bounds__(kRedThreads, 4) gs_reduce_kernel(SweepArgs a, long long ncells) {
  extern __shared__ double gpart[];  // [parts][nbo]
  constexpr bool kWarps = sizeof(S) == 8;
  const int nbo = a.th.nbo, nd = a.nd, lpc = nbo / V, parts = kWarps ? kRedThreads / 32 : kRedThreads / lpc;
  const int part = threadIdx.x / (kWarps ? 32 : lpc), first = threadIdx.x - part * (kWarps ? 32 : lpc);
  const int d0 = (int)((long long)part * nd / parts), d1 = (int)((long long)(part + 1) * nd / parts);
  for (long long P = blockIdx.x; P < ncells; P += gridDim.x) {
    for (int lp = first; part < parts && lp < lpc; lp += kWarps ? 32 : lpc) {
      const int b0 = V * lp;
      const S* row = reinterpret_cast<const S*>(a.Iout) + P * (long long)nd * nbo + b0;
      double* g = gpart + part * nbo + b0;
      if constexpr (kWarps) {
        FixedSum sum(a.I0cell + P * nbo + b0);
        auto batch = [&](auto n, int d) {
          constexpr int N = decltype(n)::value;
          double2 x[N];
          double w[N];
#pragma unroll
          for (int u = 0; u < N; ++u) x[u] = __ldcs(reinterpret_cast<const double2*>(row + (long long)(d + u) * nbo));
#pragma unroll
          for (int u = 0; u < N; ++u) w[u] = __ldg(a.wdir + d + u);
#pragma unroll
          for (int u = 0; u < N; ++u) sum.add(x[u].x, x[u].y, w[u]);
        };
        int d = d0;
        for (; d + 4 <= d1; d += 4) batch(std::integral_constant<int, 4>{}, d);
        for (; d < d1; ++d) batch(std::integral_constant<int, 1>{}, d);
        sum.close();
        g[0] = sum.G[0];
        g[1] = sum.G[1];
      } else {
        ff::P2 G[V / 2];
#pragma unroll
        for (int v = 0; v < V / 2; ++v) G[v] = ff::zero();
        for (int d = d0; d < d1; d += 16) {
          float acc[V];
#pragma unroll
          for (int v = 0; v < V; ++v) acc[v] = 0.f;
#pragma unroll
          for (int h = 0; h < 16; h += 8) {  // eight loads in flight
            float x[8][V];
#pragma unroll
            for (int u = 0; u < 8; ++u)
              if (d + h + u < d1) Tr<S>::ld_stream(row + (long long)(d + h + u) * nbo, x[u]);
#pragma unroll
            for (int u = 0; u < 8; ++u)
              if (d + h + u < d1) {
                const float w = a.wdir32[d + h + u];
#pragma unroll
                for (int v = 0; v < V; ++v) acc[v] = fmaf(w, x[u][v], acc[v]);
              }
          }
#pragma unroll
          for (int v = 0; v < V / 2; ++v) ff::acc(G[v], ff::P2{ff::pack(acc[2 * v], acc[2 * v + 1]), 0ull});
        }
#pragma unroll
        for (int v = 0; v < V / 2; ++v) ff::to_doubles(ff::norm(G[v]), g[2 * v], g[2 * v + 1]);
      }
    }
    __syncthreads();
    if (threadIdx.x < 32) reduce_energies<sizeof(S) != 8>(a, gpart, parts, P);
    __syncthreads();
  }
}

// FP64 values and their energies in one pass (REDUCE: a.Ec as gs_reduce_kernel leaves
// it, for the values as stored): a warp's lanes hold band pairs of one direction, the
// warps contiguous eighths of the caller's directions.  The sums are FP64 additions:
// the values need not be near I0(T_p), which the fixed-point sums of a step count on, and a
// reduced mode's deviations keep all their bits.  Bound by HBM, 16 bytes per FP64 value: the
// sums' two FMAs per lane and row hide behind the copies.  96x64 x 400 x 55, restore,
// T_L and read-out: 1459 us, 1540 with fixed-point sums here.
template <typename S, bool REDUCE>
__global__ void __launch_bounds__(256) pack_kernel(const double* in, S* I, const double* I0ref, const int* rows,
                                                   long long ncells, int nd, int nb, int nbp, SweepArgs a) {
  extern __shared__ double gpart[];  // REDUCE: [8][nbp]
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int dlo = wid * nd / 8, dhi = (wid + 1) * nd / 8;
  for (long long P = blockIdx.x; P < ncells; P += gridDim.x) {
    S* row = I + P * (long long)nd * nbp;
    const double* x = in + P * nd * nb;
    for (int c = 0; c < nbp; c += 64) {
      const int b = c + 2 * lane;
      double r0 = 0.0, r1 = 0.0, g0 = 0.0, g1 = 0.0;
      if (sizeof(S) != 8) {
        if (b < nb) r0 = I0ref[b];
        if (b + 1 < nb) r1 = I0ref[b + 1];
      }
      for (int d0 = dlo; d0 < dhi; d0 += 4) {
        double v[4][2];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int e = c + 32 * h + lane;
            v[u][h] = d0 + u < dhi && e < nb ? __ldcs(x + (long long)(d0 + u) * nb + e) : 0.0;
          }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (d0 + u >= dhi) break;
          // bands b, b + 1 = elements 2 lane, 2 lane + 1 of the 64: half lane >> 4, lanes 2 lane (+ 1) mod 32
          const int s0 = (2 * lane) & 31, r = rows[d0 + u];
          const double a0 = __shfl_sync(0xffffffffu, v[u][0], s0), a1 = __shfl_sync(0xffffffffu, v[u][0], s0 + 1);
          const double e0 = __shfl_sync(0xffffffffu, v[u][1], s0), e1 = __shfl_sync(0xffffffffu, v[u][1], s0 + 1);
          const double x0 = lane < 16 ? a0 : e0, x1 = lane < 16 ? a1 : e1;
          S* to = row + (long long)r * nbp + b;
          if (b < nbp) st_pair(to, x0 - r0, x1 - r1);
          if constexpr (REDUCE) {
            const double w = a.wdir[r];
            double y0 = x0, y1 = x1;
            if constexpr (sizeof(S) != 8) stored_pair<S>(x0 - r0, x1 - r1, y0, y1);
            g0 = fma(w, y0, g0);
            g1 = fma(w, y1, g1);
          }
        }
      }
      if constexpr (REDUCE) {
        if (b < nbp) {
          gpart[wid * nbp + b] = g0;
          gpart[wid * nbp + b + 1] = g1;
        }
      }
    }
    if constexpr (REDUCE) {
      __syncthreads();
      if (threadIdx.x < 32) reduce_energies<sizeof(S) != 8>(a, gpart, 8, P);
      __syncthreads();
    }
  }
}

// E_L of every cell from its partial energies (after a state restore).
__global__ void energy_L_kernel(const double2* Ec, double* EL, long long ncells) {
  for (long long P = blockIdx.x * (long long)blockDim.x + threadIdx.x; P < ncells; P += (long long)gridDim.x * blockDim.x) {
    double e = 0.0;
    for (int k = 0; k < kRedEntries; ++k) e += Ec[P * kRedEntries + k].x;
    EL[P] = e;
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
// 67x45 grid with 400 directions x 55 bands; this form takes 15 and 23 us.
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
    if constexpr (sizeof(S) != 8) num = fma((w.wd.sum_out - w.wd.sum_in) + (w.wd.sum_out_lo - w.wd.sum_in_lo), w.I0ref[b], num);
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
  auto go = [&](auto tag, auto vec) {
    using T = decltype(tag);
    constexpr int V = decltype(vec)::value;
    const size_t sm = (size_t)(sizeof(T) == 8 ? kRedThreads / 32 : kRedThreads / (a.th.nbo / V)) * a.th.nbo * sizeof(double);
    gs_reduce_kernel<T, V><<<grid, kRedThreads, sm, s>>>(a, ncells);
  };
  if (precision == 0) go(double{}, std::integral_constant<int, 2>{});
  else if (precision == 1) go(float{}, std::integral_constant<int, 4>{});
  else go(__nv_bfloat16{}, std::integral_constant<int, 8>{});
  return cudaGetLastError();
}

cudaError_t launch_refill(bool ff, void* I, const double* I0cell, long long ncells, int nd, int nbo, cudaStream_t s) {
  if (ff) refill_kernel<FFElem><<<cell_grid(ncells), 256, 0, s>>>((FFElem*)I, I0cell, ncells, nd, nbo);
  else refill_kernel<double><<<cell_grid(ncells), 256, 0, s>>>((double*)I, I0cell, ncells, nd, nbo);
  return cudaGetLastError();
}

cudaError_t launch_init_cells(int precision, bool ff, void* I, double* I0cell, double* J, double* Msum, double* MsumL, double* Tp,
                              double* Te, double* TL, double* EL, const double* Tcells, const double* I0ref,
                              long long cell0, int ncells, int nd, ThermoTables th, cudaStream_t s) {
  auto go = [&](auto tag) {
    using T = decltype(tag);
    init_cells_kernel<T><<<cell_grid(ncells), 256, th.nbp * sizeof(double), s>>>((T*)I, I0cell, J, Msum, MsumL, Tp, Te, TL, EL, Tcells,
                                                                                 I0ref, cell0, ncells, nd, th);
  };
  if (precision == 0 && ff) go(FFElem{});
  else if (precision == 0) go(double{});
  else if (precision == 1) go(float{});
  else go(__nv_bfloat16{});
  return cudaGetLastError();
}

cudaError_t launch_state_from_Tp(double* I0cell, double* J, double* Msum, double* MsumL, const double* Tp, double* Te,
                                 long long ncells, ThermoTables th, cudaStream_t s) {
  state_from_Tp_kernel<<<cell_grid(ncells), 64, th.nbp * sizeof(double), s>>>(I0cell, J, Msum, MsumL, Tp, Te, ncells,
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

cudaError_t launch_flux_cells(int precision, bool state_ff, bool grouped, const void* I, double* q, const double* S,
                              long long cell0, int ncells, int nd, int nbp, int dim, cudaStream_t s) {
  const int grid = cell_grid(ncells);
  auto go = [&](auto tag, auto vec) {
    using T = decltype(tag);
    constexpr int V = decltype(vec)::value;
    if (!grouped) flux_cells_kernel<T, V, 3, false><<<grid, 256, 0, s>>>((const T*)I, q, S, cell0, ncells, nd, nbp);
    else if (dim == 3) flux_cells_kernel<T, V, 3, true><<<grid, 256, 0, s>>>((const T*)I, q, S, cell0, ncells, nd, nbp);
    else flux_cells_kernel<T, V, 2, true><<<grid, 256, 0, s>>>((const T*)I, q, S, cell0, ncells, nd, nbp);
  };
  if (!grouped && dim != 3) return cudaErrorInvalidValue;
  if (precision == 0 && state_ff) go(FFElem{}, std::integral_constant<int, 2>{});
  else if (precision == 0) go(double{}, std::integral_constant<int, 2>{});
  else if (precision == 1) go(float{}, std::integral_constant<int, 4>{});
  else go(__nv_bfloat16{}, std::integral_constant<int, 8>{});
  return cudaGetLastError();
}

cudaError_t launch_flux_walls(int precision, bool state_ff, const void* I, const double* I0ref, const double* I0wall,
                              const DevGeom* geoms, int geom, const WallDirs* wall_dirs, const double* S, int nd, int nbp,
                              double* face_out, int max_faces, const int (&nfaces)[6], int nsides, double* out,
                              cudaStream_t s) {
  int most = 1;
  SideFaces nf{};
  for (int k = 0; k < nsides; ++k) {
    nf.n[k] = nfaces[k];
    most = std::max(most, nfaces[k]);
  }
  const dim3 grid(cell_grid(most), nsides);
  SideDirs wd;
  std::copy(wall_dirs, wall_dirs + 6, wd.d);
  auto go = [&](auto tag) {
    using T = decltype(tag);
    flux_faces_kernel<T><<<grid, kFluxThreads, 0, s>>>((const T*)I, I0ref, I0wall, geoms, geom, wd, S, nd, nbp, face_out,
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

cudaError_t launch_unpack(int precision, bool state_ff, const void* I, double* out, const double* I0ref, const int* rows,
                          long long ncells, int nd, int nb, int nbp, cudaStream_t s) {
  auto go = [&](auto tag) {
    using T = decltype(tag);
    unpack_kernel<T><<<cell_grid(ncells), 256, 0, s>>>((const T*)I, out, I0ref, rows, ncells, nd, nb, nbp);
  };
  if (precision == 0 && state_ff) go(FFElem{});
  else if (precision == 0) go(double{});
  else if (precision == 1) go(float{});
  else go(__nv_bfloat16{});
  return cudaGetLastError();
}

cudaError_t launch_pack(int precision, const double* in, void* I, const double* I0ref, const int* rows,
                        long long ncells, int nd, int nb, int nbp, const SweepArgs* energies, cudaStream_t s) {
  auto go = [&](auto tag) {
    using T = decltype(tag);
    if (energies)
      pack_kernel<T, true><<<cell_grid(ncells), 256, 8 * (size_t)nbp * sizeof(double), s>>>(in, (T*)I, I0ref, rows, ncells, nd, nb,
                                                                                          nbp, *energies);
    else
      pack_kernel<T, false><<<cell_grid(ncells), 256, 0, s>>>(in, (T*)I, I0ref, rows, ncells, nd, nb, nbp, SweepArgs{});
  };
  if (precision == 0) go(double{});
  else if (precision == 1) go(float{});
  else go(__nv_bfloat16{});
  return cudaGetLastError();
}

cudaError_t launch_energy_L(const double2* Ec, double* EL, long long ncells, cudaStream_t s) {
  energy_L_kernel<<<grid_for(ncells, 128), 128, 0, s>>>(Ec, EL, ncells);
  return cudaGetLastError();
}

}  // namespace bte
