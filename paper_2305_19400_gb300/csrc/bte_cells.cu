// bte_cells.cu -- the per-cell step after a sweep (sm_103a): energies from the
// sweep's band sums, T_p solve, I0 refresh (Sec. 2.2, 3.2).
//
// The sweeps (bte_rows.cuh, bte_sweep.cuh, the sweep-ordered pass and the
// unstructured sweep with gs_reduce_kernel) write G_b = sum_d w_d I_{d,b} of
// every cell to Gc[cell][team][band]; one launch of cells_kernel then serves every
// cell.  Keeping this out of the sweeps leaves them without a CTA barrier, a
// shuffle tree or a serial solve between two cells' streaming: on the paper's
// device (20 directions per cell) the fused epilogue took over half of a sweep.
#include <algorithm>

#include "bte_mlp.cuh"
#include "bte_solve.cuh"

namespace bte {

namespace {

// Eight lanes per cell, 16 cells per CTA pass; a CTA's cells lie gridDim.x
// apart, so that the cells of a hot spot, which leave their models' trust
// radius together, spread over the clusters.
//  mode 0  E_L, E_p from Gc, solve
//  mode 1  E_L, E_p from Gc to Epart (band-range handle, before the exchange)
//  mode 2  E_L, E_p from Epart, solve (after the exchange)
// Phase 1: the cell's sums (lanes over bands, a three-step shuffle tree), the
// root of its cached cubic model, I0 refresh inside the trust radius; other
// cells go to the CTA's own part of the queue a.fix.  Bound by the FP64 pipe
// (73 cycles per warp instruction and SM sub-partition, measured): per four
// cells of 56 bands 28 FMAs and adds of the sums, 14 of the trees and the
// solve, 21 of the refresh; a warp per cell would issue 32 for one.
// Phase 2: the queued cells, exactly (FP64 quadrature, Halley, bisection
// fallback), each by the whole cluster (exact_solve_cluster spreads an
// evaluation's bands over the cluster's SMs; with a handful of such cells the
// solve's latency is what the step waits for).  The start is the model root,
// or when there is none the previous T_p (plain mode) or the learned guess
// (net A, then surrogate Newton steps on net B, by warp 0 of each CTA: the
// same value everywhere); each evaluation becomes the cell's cached model.
constexpr int kCellThreads = 128;
constexpr int kCellCluster = 4;
constexpr int kCellLanes = 8;
constexpr int kCellSlots = kCellThreads / kCellLanes;

template <bool LEARNED>
__global__ void __cluster_dims__(kCellCluster, 1, 1) __launch_bounds__(kCellThreads, 6)
    cells_kernel(SweepArgs a, long long ncells, int mode, MLPView m) {
  extern __shared__ double fsm[];  // exact_solve_cluster scratch, T0, then the learned-mode buffers
  __shared__ int queued;           // this CTA's entries in a.fix
  __shared__ unsigned nsolve, nbad;
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int nbo = a.th.nbo, nbp = a.th.nbp;
  const int slot = threadIdx.x / kCellLanes, sub = threadIdx.x % kCellLanes;
  if (threadIdx.x == 0) { queued = 0; nsolve = 0; nbad = 0; }
  __syncthreads();
  const long long per_cta = (ncells + gridDim.x - 1) / gridDim.x;  // entries of one CTA's part of the queue
  for (long long k0 = 0; k0 < per_cta; k0 += kCellSlots) {
    const long long P = blockIdx.x + (long long)gridDim.x * (k0 + slot);
    const bool on = P < ncells;
    if (!__any_sync(0xffffffffu, on)) continue;
    double EL = 0.0, Ep = 0.0;
    if (mode == 2) {
      if (on) {
        EL = a.Epart[2 * P];
        Ep = a.Epart[2 * P + 1];
      }
    } else {
      if (on) {
        const double* G = a.Gc + P * a.gsplit * nbo;
        for (int b = sub; b < nbo; b += kCellLanes) {
          double g = G[b];
          for (int q = 1; q < a.gsplit; ++q) g += G[q * nbo + b];
          EL = fma(g, a.th.inv_v[b], EL);
          Ep = fma(g, a.th.binv_v[b], Ep);
        }
      }
#pragma unroll
      for (int o = kCellLanes / 2; o > 0; o >>= 1) {
        EL += __shfl_xor_sync(0xffffffffu, EL, o);
        Ep += __shfl_xor_sync(0xffffffffu, Ep, o);
      }
    }
    if (!on) continue;  // no barrier or shuffle below in this loop
    if (mode == 1) {
      if (sub == 0) {
        a.Epart[2 * P] = EL;
        a.Epart[2 * P + 1] = Ep;
      }
      continue;
    }
    if (sub == 0) a.EL[P] = EL;
    if (!isfinite(EL) || !isfinite(Ep)) {
      if (sub == 0) atomicAdd(&nbad, 1u);
      continue;
    }
    if (!a.solve_tp) continue;  // every beta_b is zero: only E_L is kept
    // root of (F - E_p) + F1 d + F2 d^2 / 2 + F3 d^3 / 6 nearest 0; F .. F3: the
    // model's sums sum_b a_p,b J_k,b, kept with J
    const double* M = a.Msum + 4 * P;
    const double Te = a.Teval[P];
    const double delta = model_step(M[0] - Ep, M[1], M[2], M[3]);
    const double Tn = Te + delta;
    if (isfinite(Tn) && fabs(delta) <= a.trust_rel * Tn) {
      if (sub == 0) {
        a.Tp[P] = Tn;
        if (a.beta_exp != 0.0) a.bscale[P] = pow(Tn / a.beta_Tref, a.beta_exp);
        atomicAdd(&nsolve, 1u);
      }
      const double* Jb = a.J + (P * 4) * nbp + a.th.band0;
      for (int b = sub; b < nbo; b += kCellLanes)
        a.I0cell[P * nbo + b] = b < a.th.nbr ? model_I0(Jb + b, nbp, delta) : 0.0;
    } else if (sub == 0) {
      atomicAdd(&nsolve, 1u);
      FixItem fi;
      fi.P = P;
      fi.Ep = Ep;
      fi.model = (isfinite(Tn) && Tn >= kTmin && Tn <= kTmax) ? 1 : 0;
      fi.T0 = fi.model ? Tn : a.Tp[P];
      fi.pad = 0;
      a.fix[blockIdx.x * per_cta + atomicAdd(&queued, 1)] = fi;
    }
  }
  if (mode == 1) return;
  __syncthreads();
  if (threadIdx.x == 0 && a.counters) {
    if (nsolve) atomicAdd(&a.counters->solves, (unsigned long long)nsolve);
    if (nbad) atomicAdd(&a.counters->nonfinite, (unsigned long long)nbad);
  }
  if (!a.solve_tp) return;
  cl.sync();  // every CTA's queue is complete

  const int rank = (int)cl.block_rank(), nr = (int)cl.num_blocks();
  const int own0 = rank * nbp / nr, own1 = (rank + 1) * nbp / nr;  // bands whose model row this CTA writes
  double* solve_sm = fsm;
  double* t0_sm = fsm + cta_solve_smem_doubles(nbp, a.th.ng, nr);
  [[maybe_unused]] float* ybuf = reinterpret_cast<float*>(t0_sm + 2);
  [[maybe_unused]] float* hbuf = ybuf + 2 * nbp;
  unsigned long long evals = 0, fb = 0, bad = 0;
  unsigned par = 0;  // evaluations of this cluster so far (the solve's buffer parity)
  for (int r = 0; r < nr; ++r) {  // the same items, in the same order, in every CTA of the cluster
    const int n = *cl.map_shared_rank(&queued, (unsigned)r);
    const FixItem* q = a.fix + (blockIdx.x - rank + r) * per_cta;
    for (int w = 0; w < n; ++w) {
      const FixItem it = q[w];
      const long long P = it.P;
      // learned mode: the networks' guess starts the cells that have no usable
      // root of their cached model (a cold or far-off start); a model root, when
      // there is one, is the closer start (measured: twice the evaluations from
      // the networks' guess on the learned 3-D workload)
      double T0 = it.T0;
      if constexpr (LEARNED) {
        if (!it.model) {  // uniform over the cluster (one item)
          if (threadIdx.x < 32) {
            const double g = mlp_guess_T(m, a.th.a_p, it.Ep, 2, ybuf, hbuf);
            if (threadIdx.x == 0) t0_sm[0] = g;
          }
          __syncthreads();
          T0 = t0_sm[0];
        }
      }
      const SolveResult s = exact_solve_cluster(a.th, it.Ep, T0, a.trust_rel, a.maxit, a.J + (P * 4) * nbp, solve_sm, par);
      evals += s.evals;
      fb += s.fallback;
      bad += s.bad;
      __syncthreads();  // this CTA's model rows, written by the solve, before its I0 refresh reads them
      // I0 refresh of the stored bands whose model rows this CTA wrote, at s.Te
      const int s0 = max(own0 - a.th.band0, 0), s1 = min(own1 - a.th.band0, nbo);
      for (int b = s0 + (int)threadIdx.x; b < s1; b += blockDim.x)
        a.I0cell[P * nbo + b] = b < a.th.nbr ? model_I0(a.J + (P * 4) * nbp + a.th.band0 + b, nbp, s.delta) : 0.0;
      if (rank == 0 && threadIdx.x == 0) {
        a.Teval[P] = s.Te;
        a.Tp[P] = s.Te + s.delta;
        if (a.beta_exp != 0.0) a.bscale[P] = pow((s.Te + s.delta) / a.beta_Tref, a.beta_exp);
        for (int k = 0; k < 4; ++k) a.Msum[4 * P + k] = s.M[k];  // the model just written to J
      }
      __syncthreads();  // t0_sm and the solve scratch are reused by the next item
    }
  }
  cl.sync();  // no CTA leaves while another may still read its shared memory
  if (rank == 0 && threadIdx.x == 0 && a.counters) {
    if (evals) atomicAdd(&a.counters->evals, evals);
    if (fb) atomicAdd(&a.counters->fallbacks, fb);
    if (bad) atomicAdd(&a.counters->nonfinite, bad);
  }
}

}  // namespace

// 76 clusters of kCellCluster CTAs at least (two CTAs per SM), eight per SM at
// most: a CTA pass holds 16 cells, and small grids spread over all SMs.
long long cells_queue_entries(long long ncells) {
  const long long g = cells_grid(ncells);
  return g * ((ncells + g - 1) / g);
}

int cells_grid(long long ncells) {
  const long long g = std::max<long long>(2 * 152, std::min<long long>(8 * 152, (ncells + kCellSlots - 1) / kCellSlots));
  return (int)((g + kCellCluster - 1) / kCellCluster * kCellCluster);
}

cudaError_t launch_cells(const SweepArgs& a, long long ncells, int mode, const MLPView* mlp, cudaStream_t s) {
  const size_t sm = mode == 1 ? 0
                              : (cta_solve_smem_doubles(a.th.nbp, a.th.ng, kCellCluster) + 2) * sizeof(double) +
                                    (mlp ? (2 * (size_t)a.th.nbp + 4 * kHidden) * sizeof(float) : 0);
  MLPView m{};
  if (mlp) m = *mlp;
  if (mlp) cells_kernel<true><<<cells_grid(ncells), kCellThreads, sm, s>>>(a, ncells, mode, m);
  else cells_kernel<false><<<cells_grid(ncells), kCellThreads, sm, s>>>(a, ncells, mode, m);
  return cudaGetLastError();
}

}  // namespace bte
