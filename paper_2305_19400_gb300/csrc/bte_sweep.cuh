// bte_sweep.cuh -- the sweep kernel of one inner iteration, BF16 storage (sm_103a).
//
// sweep_kernel<DIM, MINB, EXPL>: a CTA owns a run of cells of one geometry; each
// cell is served by a team of lpc x dteam lanes.  Lane (q, l) holds 8 consecutive
// bands as one 16-byte vector and walks the directions d = q, q + dteam, ... (in
// the internal order, bte_tables.h); a team step so covers dteam consecutive
// rows of the cell, up to ~0.9 KB of contiguous memory per array.  For every
// (cell, direction, band) (Sec. 3.1, Eq. 5)
//   I^{k+1} = P I^n + Q (v_b sum_ax c_ax I_up,ax^k + beta_b I0^k)
// (implicit: point-Jacobi sweep of backward Euler; explicit: forward Euler with
// I^k = I^n) in FP32 on the stored deviation I - I0_b(T_ref): the update is affine
// with coefficients summing to one, so the deviation obeys the same update with
// I0 and wall ghosts shifted.  The upwind value is the neighbour cell on the side
// S_d comes from, or the Eq. 6 ghost at a wall (I0 of the wall face, or the
// cell's own value in the mirrored direction); isothermal ghosts are FP32
// deviations, read at use, which is why this storage keeps a kernel of its own
// beside the row sweeps of bte_rows.cuh.
// Each lane sums its part of G_b = sum_d w_d I^{k+1}_{d,b} in float partials flushed
// to FP64; at the end of an item the band owners add the dteam partials per band
// in a fixed order and write their bands' energies to Ec, from which cells_kernel
// (bte_cells.cu) solves T_p and refreshes I0.
// Memory: I^n is read once, I^{k+1} written once, and each I^k row read from
// DRAM once (adjacent cells, processed together, re-read it from L2).  Each
// thread copies the operands of its next directions into shared memory with
// cp.async kStages-1 steps before it uses them.  MINB is the launch-bounds
// minimum of resident CTAs per SM (a register cap).
#pragma once
#include <type_traits>

#include "bte_ff.cuh"
#include "bte_store.cuh"

namespace bte {
namespace sweep {

using S = __nv_bfloat16;
using T = Tr<S>;
constexpr int V = T::V;

// Per-cell addressing of one lane: its rows in I^n, I^k, I^{k+1} (band offset
// applied), the element strides to the x/y/z neighbours and which sides are
// walls, so a direction's upwind address is one select and one add.
struct CellAddr {
  const S* in;
  const S* ik;
  S* out;
  long long sx, sy, sz;
  int wall;      // bit 2*ax: low wall along ax, bit 2*ax+1: high wall
  int ci, cj, ck;
};

// Address of the upwind value along axis AX for direction row offset `off`
// (d * nbo): the neighbour's row or the Eq. 6 ghost of a wall side: I0 of the face
// (isothermal, or a refreshed diffuse value, as FP32 deviations), the side's
// per-direction ghost row (partially specular), or the cell's own value in the
// mirrored direction (specular).
template <int AX>
__device__ __forceinline__ const void* upwind_src(const SweepArgs& a, const DevGeom* gp, const CellAddr& c,
                                                  const int4 di, long long off, int b0) {
  const bool from_low = (di.x >> AX) & 1;
  const int side = 2 * AX + (from_low ? 0 : 1);
  if (!((c.wall >> side) & 1)) {
    const long long st = AX == 0 ? c.sx : (AX == 1 ? c.sy : c.sz);
    return c.ik + (from_low ? -st : st) + off;
  }
  const int nbp = a.th.nbo;
  const int bc = gp->bc[side];
  if (bc == 0 || bc == 3) {  // wall data stay in memory (L1): only wall cells get here
    const long long fl = AX == 0 ? c.cj + (long long)gp->ny * c.ck
                                 : (AX == 1 ? c.ci + (long long)gp->nx * c.ck : c.ci + (long long)gp->nx * c.cj);
    if (bc == 3) return reinterpret_cast<const S*>(gp->gdir[side]) + fl * ((long long)a.nd * nbp) + off + b0;
    return a.I0wall_dev + (gp->face0[side] + fl) * nbp + b0;
  }
  const int r = AX == 0 ? di.y : (AX == 1 ? di.z : di.w);
  return c.ik + (long long)r * nbp;
}

// Asynchronous global -> shared copy of one lane vector, L2 only.
__device__ __forceinline__ void cp_async(unsigned smem, const void* g) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Shared per-direction table of the current cell-size class.
struct DirSm {
  int4 info;     // up flags, rx, ry, rz
  float4 c;      // c_ax = |S_d,ax| / (w_d Delta_ax), their sum
  float w32;     // w_d rounded to float
  float pad[3];
};

// Staging ring: per thread and stage, 16 bytes per operand (I^n, the upwind value
// per axis).
constexpr int kStages = 4;
template <int DIM>
struct Ring {
  static constexpr int kOps = 1 + DIM;
};

// The end of an item: the lanes of a cell hold the partials G[v] of their
// directions; the band owners (dg == 0) add them in a fixed order to the
// W I0_b(T_ref) term of the deviation storage and write their energies to Ec.  With one
// direction per team step a lane's sums are complete and no barrier is needed;
// otherwise every thread calls it (two CTA barriers).
__device__ __forceinline__ void write_band_sums(const SweepArgs& a, double* gsm, bool active, int dg, int lane,
                                                long long P, double (&G)[V]) {
  const int lpc = a.lpc, b0 = V * lane;
  if (a.dteam > 1) {
#pragma unroll
    for (int v = 0; v < V; ++v) gsm[(size_t)threadIdx.x * V + v] = G[v];
    __syncthreads();
    if (dg == 0)
      for (int q = 1; q < a.dteam; ++q)
#pragma unroll
        for (int v = 0; v < V; ++v) G[v] += gsm[(size_t)(threadIdx.x + q * lpc) * V + v];
    __syncthreads();
  }
  if (dg == 0 && active) {
    double eL = 0.0, eP = 0.0;
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const double g = fma(a.Wtot, a.I0ref[b0 + v], G[v]);
      eL = fma(g, a.th.inv_v[b0 + v], eL);
      eP = fma(g, a.th.binv_v[b0 + v], eP);
    }
    a.Ec[P * lpc + lane] = make_double2(eL, eP);
  }
}

template <int DIM, int MINB, bool EXPL>
__global__ void __launch_bounds__(256, MINB) sweep_kernel(SweepArgs a) {
  extern __shared__ double sm[];
  __shared__ int cur_cls;
  const int lpc = a.lpc, nd = a.nd, nbp = a.th.nbo, dstep = a.dteam;
  const int team = lpc * dstep;                       // lanes per cell
  const int slot = threadIdx.x / team, tl = threadIdx.x - slot * team;
  const int dg = tl / lpc, lane = tl - dg * lpc;      // direction offset in a step, band vector
  DirSm* dsm = reinterpret_cast<DirSm*>(sm);          // [nd]
  double* gsm = sm + (sizeof(DirSm) / 8) * nd;        // [blockDim.x][V] per-lane band partials
  // staging ring of the far operands: [kStages][kOps][blockDim.x] x 16 bytes
  char* ring = reinterpret_cast<char*>(
      (reinterpret_cast<uintptr_t>(gsm + (size_t)V * blockDim.x) + 15) & ~static_cast<uintptr_t>(15));
  const S* __restrict__ In = reinterpret_cast<const S*>(a.In);
  const S* __restrict__ Ik = reinterpret_cast<const S*>(a.Ik);
  S* __restrict__ Io = reinterpret_cast<S*>(a.Iout);
  const long long row = (long long)nd * nbp;
  const int b0 = V * lane;
  if (threadIdx.x == 0) cur_cls = -1;
  float vb[V], bb[V];  // per-lane band constants
#pragma unroll
  for (int v = 0; v < V; ++v) {
    vb[v] = a.vb32[b0 + v];
    bb[v] = a.bb32[b0 + v];
  }
  // scalars of the scheme in both halves of a packed pair
  const ff::x2 dt2 = ff::pack(a.dt32, a.dt32), ndt2 = ff::pack(-a.dt32, -a.dt32), rdt2 = ff::pack(a.rdt32, a.rdt32),
               one2 = ff::pack(1.0f, 1.0f);
  __syncthreads();

  for (int item = blockIdx.x; item < a.nitems; item += gridDim.x) {
    const WorkItem wi = a.items[item];
    const DevGeom* gp = a.geoms + wi.geom;
    const int gnx = gp->nx, gny = gp->ny, gcls = gp->cls;
    const int gnz = DIM == 3 ? gp->nz : 1;
    if (gcls != cur_cls) {  // (block-uniform) direction table of this cell-size class
      __syncthreads();
      for (int d = threadIdx.x; d < nd; d += blockDim.x) {
        const DirInfo di = a.dirs[d];
        DirSm e;
        e.info = make_int4(di.up, di.rx, di.ry, di.rz);
        e.c = a.dirc[(size_t)gcls * nd + d];
        e.w32 = a.wdir32[d];
        dsm[d] = e;
      }
      if (threadIdx.x == 0) cur_cls = gcls;
      __syncthreads();
    }
    const bool active = slot < wi.cell_count;
    const int ci = wi.i0 + (active ? slot : 0), cj = wi.j, ck = wi.k;
    const long long P = gp->cell0 + wi.cell_begin + (active ? slot : 0);
    double G[V];
#pragma unroll
    for (int v = 0; v < V; ++v) G[v] = 0.0;

    if (active) {
      if (a.beta_exp != 0.0) {  // temperature-dependent relaxation: beta_b(T_p) = beta_b s
        const float bsc = (float)a.bscale[P];
#pragma unroll
        for (int v = 0; v < V; ++v) bb[v] = a.bb32[b0 + v] * bsc;
      }
      float src[V];  // beta_b(T_p) * (I0 - I0ref)
#pragma unroll
      for (int v = 0; v < V; ++v) src[v] = bb[v] * (float)(a.I0cell[P * nbp + b0 + v] - a.I0ref[b0 + v]);
      CellAddr c;
      c.in = In + P * row + b0;
      c.ik = Ik + P * row + b0;
      c.out = Io + P * row + b0;
      c.sx = row;
      c.sy = (long long)gnx * row;
      c.sz = (long long)gnx * gny * row;
      c.ci = ci; c.cj = cj; c.ck = ck;
      c.wall = (ci == 0) | ((ci == gnx - 1) << 1) | ((cj == 0) << 2) | ((cj == gny - 1) << 3) |
               (DIM == 3 ? ((ck == 0) << 4) | ((ck == gnz - 1) << 5) : 0);
      float acc[V];  // FP32 partial band sums, flushed to G periodically
#pragma unroll
      for (int v = 0; v < V; ++v) acc[v] = 0.f;
      int nacc = 0;
      // This lane's directions are d_j = dg + j*dstep.  Their operands (I^n and the
      // upwind I^k or wall ghost per axis) are copied global -> shared kStages-1
      // directions ahead with cp.async; each thread waits only for its own copies.
      const int nsteps = dg < nd ? (nd - dg + dstep - 1) / dstep : 0;
      // ring slot (stage st, operand op) of this thread: 32-bit shared addresses
      const unsigned rb0 = (unsigned)__cvta_generic_to_shared(ring) + threadIdx.x * 16u;
      const unsigned ostr = blockDim.x * 16u, sstr = Ring<DIM>::kOps * ostr;
      const long long sx = c.sx, sy = c.sy, sz = c.sz;
      // The step loop is compiled twice, for interior cells (no wall logic at all)
      // and for wall cells (per-axis Eq. 6 ghosts; isothermal ghosts are read at use).
      auto run = [&](auto interior_tag) {
        constexpr bool kInterior = decltype(interior_tag)::value;
        // stage the operands of step j into the ring slot at shared address sb
        auto issue = [&](auto checked, int j, const unsigned sb) {
          if (!decltype(checked)::value || j < nsteps) {
            const int d = dg + j * dstep;
            const int off = d * nbp;
            cp_async(sb, c.in + off);
            if (kInterior) {  // the upwind rows are the neighbours'
              const int up = dsm[d].info.x;
              cp_async(sb + ostr, c.ik + off + ((up & 1) ? -sx : sx));
              cp_async(sb + 2 * ostr, c.ik + off + ((up & 2) ? -sy : sy));
              if (DIM == 3) cp_async(sb + 3 * ostr, c.ik + off + ((up & 4) ? -sz : sz));
            } else {
              const int4 di = dsm[d].info;
#pragma unroll
              for (int ax = 0; ax < DIM; ++ax) {
                const int side = 2 * ax + (((di.x >> ax) & 1) ? 0 : 1);
                if (((c.wall >> side) & 1) && gp->bc[side] == 0) continue;  // isothermal ghosts: read at use
                cp_async(sb + (1 + ax) * ostr, ax == 0 ? upwind_src<0>(a, gp, c, di, off, b0)
                                               : (ax == 1 ? upwind_src<1>(a, gp, c, di, off, b0)
                                                          : upwind_src<2>(a, gp, c, di, off, b0)));
              }
            }
          }
          cp_async_commit();
        };
        // Upwind operand of axis ax from its slot.  A cell on an isothermal wall
        // reads that wall's FP32 ghost deviations (8 floats, cached wall data)
        // straight from memory instead.
        auto read_up = [&](unsigned sb, int ax, const int4 di, const int off, float (&x)[V]) {
          if constexpr (!kInterior) {
            const int side = 2 * ax + (((di.x >> ax) & 1) ? 0 : 1);
            if (((c.wall >> side) & 1) && gp->bc[side] == 0) {
              const void* g = ax == 0 ? upwind_src<0>(a, gp, c, di, off, b0)
                            : (ax == 1 ? upwind_src<1>(a, gp, c, di, off, b0) : upwind_src<2>(a, gp, c, di, off, b0));
              ldgv<float, V>(reinterpret_cast<const float*>(g), x);
              return;
            }
          }
          T::lds(sb + (1 + ax) * ostr, x);
        };
#pragma unroll
        for (int j = 0; j < kStages - 1; ++j) issue(std::true_type{}, j, rb0 + (unsigned)j * sstr);
        auto step = [&](int j, const unsigned sb) {
          cp_async_wait<kStages - 1>();
          const int d = dg + j * dstep;
          const int off = d * nbp;
          const int4 di = dsm[d].info;
          float vn[V], ux[V], uy[V], uz[V];
          T::lds(sb, vn);
          read_up(sb, 0, di, off, ux);
          read_up(sb, 1, di, off, uy);
          if (DIM == 3) read_up(sb, 2, di, off, uz);
          float r[V];
          // P and Q from v_b, beta_b and sum_ax c_ax (no table loads):
          // implicit Q = 1/(1/dt + beta_b + v_b sum c), P = Q/dt; explicit P = 1 - dt(beta_b + v_b sum c), Q = dt.
          // Two bands per packed f32x2 instruction (each half rounds as the
          // scalar instruction would: the same values as band by band).
          const float4 cc = dsm[d].c;
          const ff::x2 ccw = ff::pack(cc.w, cc.w), ccx = ff::pack(cc.x, cc.x), ccy = ff::pack(cc.y, cc.y),
                       ccz = ff::pack(cc.z, cc.z);
#pragma unroll
          for (int q = 0; q < V / 2; ++q) {
            const int v = 2 * q;
            const ff::x2 vb2 = ff::pack(vb[v], vb[v + 1]);
            const ff::x2 rate = ff::fma(vb2, ccw, ff::pack(bb[v], bb[v + 1]));
            ff::x2 Pc, Qc;
            if constexpr (EXPL) {
              Qc = dt2;
              Pc = ff::fma(ndt2, rate, one2);
            } else {
              const ff::x2 den = ff::add(rdt2, rate);
              float q0, q1;
              asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(q0) : "f"(ff::lo_of(den)));
              asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(q1) : "f"(ff::hi_of(den)));
              Qc = ff::pack(q0, q1);
              Pc = ff::mul(Qc, rdt2);
            }
            ff::x2 f = ff::mul(ccx, ff::pack(ux[v], ux[v + 1]));
            f = ff::fma(ccy, ff::pack(uy[v], uy[v + 1]), f);
            if (DIM == 3) f = ff::fma(ccz, ff::pack(uz[v], uz[v + 1]), f);
            const ff::x2 t = ff::fma(vb2, f, ff::pack(src[v], src[v + 1]));
            const ff::x2 rr = ff::fma(Qc, t, ff::mul(Pc, ff::pack(vn[v], vn[v + 1])));
            r[v] = ff::lo_of(rr);
            r[v + 1] = ff::hi_of(rr);
          }
          // store the rounded values and sum exactly what was stored
          const uint4 w = make_uint4(T::pack2(r[0], r[1]), T::pack2(r[2], r[3]), T::pack2(r[4], r[5]), T::pack2(r[6], r[7]));
          __stcs(reinterpret_cast<uint4*>(c.out + off), w);
          T::unpack(w, r);
          const float wd = dsm[d].w32;
          const ff::x2 wd2 = ff::pack(wd, wd);
#pragma unroll
          for (int q = 0; q < V / 2; ++q) {
            const ff::x2 a2 = ff::fma(wd2, ff::pack(r[2 * q], r[2 * q + 1]), ff::pack(acc[2 * q], acc[2 * q + 1]));
            acc[2 * q] = ff::lo_of(a2);
            acc[2 * q + 1] = ff::hi_of(a2);
          }
          // FP32 partials go to FP64 every 64 directions (the storage's 2^-8
          // rounding dwarfs the float sum's)
          if (++nacc == 64) {
#pragma unroll
            for (int v = 0; v < V; ++v) { G[v] += (double)acc[v]; acc[v] = 0.f; }
            nacc = 0;
          }
        };
        // Every step but the last kStages - 1 stages a later direction (no bounds
        // test), step j + kStages - 1 into the slot step j - 1 has just read; the
        // last steps commit an empty group, so that the wait still finds its own.
        const int nmain = nsteps - (kStages - 1);
        const unsigned slast = rb0 + (unsigned)(kStages - 1) * sstr;
        unsigned sb = rb0, sprev = slast;
        int j = 0;
        for (; j < nmain; ++j) {
          issue(std::false_type{}, j + kStages - 1, sprev);
          step(j, sb);
          sprev = sb;
          sb = sb == slast ? rb0 : sb + sstr;
        }
        for (; j < nsteps; ++j) {
          cp_async_commit();
          step(j, sb);
          sb = sb == slast ? rb0 : sb + sstr;
        }
      };
      if (c.wall == 0) run(std::true_type{});
      else run(std::false_type{});
      cp_async_wait<0>();
#pragma unroll
      for (int v = 0; v < V; ++v) G[v] += (double)acc[v];
    }
    write_band_sums(a, gsm, active, dg, lane, P, G);
  }
}

template <int MINB, bool EXPL>
cudaError_t launch_minb(const SweepArgs& a, int dim, int threads, int grid, cudaStream_t s) {
  const size_t smem = sizeof(DirSm) * (size_t)a.nd + (size_t)V * threads * sizeof(double) + 16 +
                      (size_t)kStages * (1 + dim) * threads * 16;
  const cudaError_t e = raise_dynamic_smem(
      dim == 3 ? (const void*)sweep_kernel<3, MINB, EXPL> : (const void*)sweep_kernel<2, MINB, EXPL>, smem);
  if (e != cudaSuccess) return e;
  if (dim == 3) sweep_kernel<3, MINB, EXPL><<<grid, threads, smem, s>>>(a);
  else sweep_kernel<2, MINB, EXPL><<<grid, threads, smem, s>>>(a);
  return cudaGetLastError();
}

// variant: 1 -> at least 2 resident CTAs per SM (<= 128 registers), 2 -> 3 CTAs (<= 80 registers)
inline cudaError_t launch(int variant, const SweepArgs& a, int dim, int threads, int grid, cudaStream_t s) {
  if (a.explicit_scheme)
    return variant >= 2 ? launch_minb<3, true>(a, dim, threads, grid, s) : launch_minb<2, true>(a, dim, threads, grid, s);
  return variant >= 2 ? launch_minb<3, false>(a, dim, threads, grid, s) : launch_minb<2, false>(a, dim, threads, grid, s);
}

}  // namespace sweep
}  // namespace bte
