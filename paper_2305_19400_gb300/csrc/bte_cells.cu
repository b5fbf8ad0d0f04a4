// bte_cells.cu -- the per-cell step after a sweep (sm_103a): energies from the
// sweep's sums, T_p solve, I0 refresh (Sec. 2.2, 3.2), and T_L on request.
//
// The sweeps (bte_rows.cuh, bte_sweep.cuh, the sweep-ordered pass and the
// unstructured sweep with gs_reduce_kernel) write partial energies
// (sum_b G_b / v_b, sum_b beta_b G_b / v_b), G_b = sum_d w_d I_{d,b}, of every cell to
// Ec[cell][a.ne]; one launch of cells_kernel then serves every cell.  Keeping this
// out of the sweeps leaves them without a CTA barrier, a shuffle tree or a serial
// solve between two cells' streaming: on the paper's device (20 directions per
// cell) the fused epilogue took over half of a sweep.
#include <algorithm>
#include <type_traits>

#include "bte_mlp.cuh"
#include "bte_pdl.cuh"
#include "bte_solve.cuh"

namespace bte {

namespace {

// Eight lanes per cell, 16 cells per CTA pass; a CTA's cells lie gridDim.x
// apart and the number of clusters is a prime, so that the cells of a hot wall
// (a row or a column of the grid), which leave their models' trust radius
// together, spread over all clusters.
enum { kSolve = 0, kPartial = 1, kFromPartial = 2, kLattice = 3 };
//  kSolve        E_L, E_p from Ec, T_p
//  kPartial      E_L, E_p from Ec to Epart (band-range handle, before the exchange)
//  kFromPartial  E_L, E_p from Epart, T_p (after the exchange)
//  kLattice      T_L from E_L (on request; the cells' models stay as they are)
// Phase 1: the cell's sums (a three-step shuffle tree), the root of its cached
// cubic model, I0 refresh inside the trust radius; other cells go to the CTA's
// own part of the queue a.fix.  Bound by the FP64 pipe (73 cycles per warp
// instruction and SM sub-partition, measured): per four cells of 56 bands on the
// paper's device 7 adds of the partial energies, 6 of the tree, 7 of the solve and
// 21 FMAs of the refresh; a warp per cell would issue 30 for one.
// Phase 2: the queued cells, exactly (FP64 quadrature, Halley, bisection
// fallback): one or two in a cluster each by the whole cluster (an evaluation's
// bands spread over its SMs; the solve's latency is what the step then waits
// for), more of them each by its own CTA, which repeats no sums (in a transient
// every cell is queued and the FP64 pipe is the bound).  The start is the model root,
// or when there is none the previous T_p (plain mode) or the learned guess
// (net A, then surrogate Newton steps on net B, by warp 0 of each CTA: the
// same value everywhere); each evaluation becomes the cell's cached model.
constexpr int kCellThreads = 128;
constexpr int kCellCluster = 8;
constexpr int kCellLanes = 8;
constexpr int kCoopCells = 2;  // exact solves of a cluster up to which it works together on each
constexpr int kCellSlots = kCellThreads / kCellLanes;

template <bool LEARNED>
__global__ void __cluster_dims__(kCellCluster, 1, 1) __launch_bounds__(kCellThreads, 6)
    cells_kernel(SweepArgs a, long long ncells, int mode, MLPView m) {
  extern __shared__ double fsm[];  // exact_solve_cluster scratch, T0, then the learned-mode buffers
  __shared__ int queued;           // this CTA's entries in a.fix
  __shared__ int counts[kCellCluster];  // every CTA's of the cluster
  __shared__ unsigned nsolve, nbad;
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int nbo = a.th.nbo, nbp = a.th.nbp;
  const int slot = threadIdx.x / kCellLanes, sub = threadIdx.x % kCellLanes;
  const bool lattice = mode == kLattice;
  const float trust = (float)a.trust_rel, T_knee = (float)a.th.T_knee;
  const bool solves = mode != kPartial && (lattice || a.solve_tp);
  if (solves) asm volatile("barrier.cluster.arrive;" ::: "memory");  // awaited before the first remote access
  if (threadIdx.x == 0) { queued = 0; nsolve = 0; nbad = 0; }
  __syncthreads();
  pdl_wait();
  const long long per_cta = (ncells + gridDim.x - 1) / gridDim.x;  // entries of one CTA's part of the queue
  for (long long k0 = 0; k0 < per_cta; k0 += kCellSlots) {
    const long long P = blockIdx.x + (long long)gridDim.x * (k0 + slot);
    const bool on = P < ncells;
    if (!__any_sync(0xffffffffu, on)) continue;
    double EL = 0.0, Ep = 0.0, M[4] = {0.0, 0.0, 0.0, 0.0}, Te = 0.0;
    if (on && mode != kPartial) {  // the model's sums: loads in flight beside the energies'
      const double2* Mp = reinterpret_cast<const double2*>((lattice ? a.MsumL : a.Msum) + 4 * P);
      const double2 m0 = Mp[0], m1 = Mp[1];
      M[0] = m0.x; M[1] = m0.y; M[2] = m1.x; M[3] = m1.y;
      Te = a.Teval[P];
    }
    if (lattice) {
      if (on) EL = Ep = a.EL[P];
    } else if (mode == kFromPartial) {
      if (on) {
        EL = a.Epart[2 * P];
        Ep = a.Epart[2 * P + 1];
      }
    } else {
      if (on) {
        const double2* E = a.Ec + P * a.ne;
        int e = sub;
        for (; e + 3 * kCellLanes < a.ne; e += 4 * kCellLanes) {
          double2 x[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) x[u] = E[e + u * kCellLanes];
#pragma unroll
          for (int u = 0; u < 4; ++u) { EL += x[u].x; Ep += x[u].y; }
        }
        double2 x[3];
#pragma unroll
        for (int u = 0; u < 3; ++u) x[u] = e + u * kCellLanes < a.ne ? E[e + u * kCellLanes] : make_double2(0.0, 0.0);
#pragma unroll
        for (int u = 0; u < 3; ++u)
          if (e + u * kCellLanes < a.ne) { EL += x[u].x; Ep += x[u].y; }
      }
#pragma unroll
      for (int o = kCellLanes / 2; o > 0; o >>= 1) {
        EL += __shfl_xor_sync(0xffffffffu, EL, o);
        Ep += __shfl_xor_sync(0xffffffffu, Ep, o);
      }
    }
    if (!on) continue;  // no barrier or shuffle below in this loop
    if (mode == kPartial) {
      if (sub == 0) {
        a.Epart[2 * P] = EL;
        a.Epart[2 * P + 1] = Ep;
      }
      continue;
    }
    if (sub == 0 && !lattice) a.EL[P] = EL;
    if (!finite(EL) || !finite(Ep)) {
      if (sub == 0) {
        atomicAdd(&nbad, 1u);
        if (lattice) a.TL[P] = EL;
      }
      continue;
    }
    if (!lattice && !a.solve_tp) continue;  // every beta_b is zero: only E_L is kept
    // root of M_0 - E + M_1 d + M_2 d^2 + M_3 d^3 nearest 0
    const double delta = model_step(M[0] - Ep, M[1], M[2], M[3]);
    const double Tn = Te + delta;
    if (in_trust(delta, Tn, trust, T_knee)) {
      if (lattice) {
        if (sub == 0) a.TL[P] = Tn;
        continue;
      }
      if (sub == 0) {
        a.Tp[P] = Tn;
        if (a.beta_exp != 0.0) a.bscale[P] = pow(Tn / a.beta_Tref, a.beta_exp);
        atomicAdd(&nsolve, 1u);
      }
      const double* Jb = a.J + (P * 4) * nbp + a.th.band0;
#pragma unroll 4
      for (int b = sub; b < nbo; b += kCellLanes)
        a.I0cell[P * nbo + b] = b < a.th.nbr ? model_I0(Jb + b, nbp, delta) : 0.0;
    } else if (sub == 0) {
      atomicAdd(&nsolve, 1u);
      FixItem fi;
      fi.P = P;
      fi.Ep = Ep;
      fi.model = (finite(Tn) && Tn >= kTmin && Tn <= kTmax) ? 1 : 0;
      fi.T0 = fi.model ? Tn : (lattice ? a.Tguess[P] : a.Tp[P]);
      fi.pad = 0;
      a.fix[blockIdx.x * per_cta + atomicAdd(&queued, 1)] = fi;
    }
  }
  if (mode == kPartial) return;
  __syncthreads();
  if (threadIdx.x == 0 && a.counters) {
    if (nsolve && !lattice) atomicAdd(&a.counters->solves, (unsigned long long)nsolve);
    if (nbad) atomicAdd(&a.counters->nonfinite, (unsigned long long)nbad);
  }
  if (!solves) return;
  // Every CTA's count goes to all of the cluster, so that a cluster without queued
  // cells (the common case) ends at one barrier: counts read from the other CTAs
  // needed a second one before any could leave (400 cells: a step of 10 sweeps 198 us,
  // 176 so; 14400 cells: 10 steps 1105 and 1073).
  const int rank = (int)cl.block_rank(), nr = (int)cl.num_blocks();
  asm volatile("barrier.cluster.wait;" ::: "memory");  // every CTA runs
  if ((int)threadIdx.x < nr) *cl.map_shared_rank(&counts[rank], threadIdx.x) = queued;
  cl.sync();  // every CTA's queue and count are complete
  int total = 0;
  for (int r = 0; r < nr; ++r) total += counts[r];
  if (total == 0) return;

  double* solve_sm = fsm;
  double* t0_sm = fsm + cta_solve_smem_doubles(nbp, a.th.ng, 1);
  [[maybe_unused]] float* ybuf = reinterpret_cast<float*>(t0_sm + 2);
  [[maybe_unused]] float* hbuf = ybuf + 2 * nbp;
  unsigned long long evals = 0, fb = 0, bad = 0;
  unsigned par = 0;  // evaluations of this cluster so far (the solve's buffer parity)
  auto solve = [&](auto coop, const FixItem& it) {
    constexpr bool COOP = decltype(coop)::value;
    const long long P = it.P;
    // learned mode: the networks' guess starts the cells that have no usable
    // root of their cached model (a cold or far-off start); a model root, when
    // there is one, is the closer start (measured: twice the evaluations from
    // the networks' guess on the learned 3-D workload)
    double T0 = it.T0;
    if constexpr (LEARNED) {
      if (!it.model && !lattice) {  // uniform over the CTAs that solve the item
        if (threadIdx.x < 32) {
          const double g = mlp_guess_T(m, a.th.a_p, it.Ep, 2, ybuf, hbuf);
          if (threadIdx.x == 0) t0_sm[0] = g;
        }
        __syncthreads();
        T0 = t0_sm[0];
      }
    }
    double* Jrow = lattice ? nullptr : a.J + (P * 4) * nbp;
    const SolveResult s = exact_solve_cluster<COOP>(a.th, lattice ? a.th.a_L : a.th.a_p, it.Ep, T0, a.trust_rel, a.maxit,
                                                    Jrow, solve_sm, par);
    if (!COOP || rank == 0) {
      evals += s.evals;
      fb += s.fallback;
      bad += s.bad;
    }
    __syncthreads();  // this CTA's model rows, written by the solve, before its I0 refresh reads them
    const bool owner = (!COOP || rank == 0) && threadIdx.x == 0;
    if (lattice) {
      if (owner) a.TL[P] = s.Te + s.delta;
    } else {
      // I0 refresh of the stored bands whose model rows this CTA wrote, at s.Te
      const int own0 = COOP ? rank * nbp / nr : 0, own1 = COOP ? (rank + 1) * nbp / nr : nbp;
      const int s0 = max(own0 - a.th.band0, 0), s1 = min(own1 - a.th.band0, nbo);
      for (int b = s0 + (int)threadIdx.x; b < s1; b += blockDim.x)
        a.I0cell[P * nbo + b] = b < a.th.nbr ? model_I0(Jrow + a.th.band0 + b, nbp, s.delta) : 0.0;
      if (owner) {
        a.Teval[P] = s.Te;
        a.Tp[P] = s.Te + s.delta;
        if (a.beta_exp != 0.0) a.bscale[P] = pow((s.Te + s.delta) / a.beta_Tref, a.beta_exp);
        for (int k = 0; k < 4; ++k) {  // the model just written to J
          a.Msum[4 * P + k] = s.M[k];
          a.MsumL[4 * P + k] = s.ML[k];
        }
      }
    }
    __syncthreads();  // t0_sm and the solve scratch are reused by the next item
  };
  if (total <= kCoopCells) {
    for (int r = 0; r < nr; ++r)  // the same items, in the same order, in every CTA of the cluster
      for (int w = 0; w < counts[r]; ++w) solve(std::true_type{}, a.fix[(blockIdx.x - rank + r) * per_cta + w]);
    cl.sync();  // no CTA leaves while another may still read its shared memory
  } else {
    for (int w = 0; w < queued; ++w) solve(std::false_type{}, a.fix[blockIdx.x * per_cta + w]);
  }
  if (threadIdx.x == 0 && a.counters) {
    if (evals && !lattice) atomicAdd(&a.counters->evals, evals);
    if (fb) atomicAdd(&a.counters->fallbacks, fb);
    if (bad) atomicAdd(&a.counters->nonfinite, bad);
  }
}

}  // namespace

long long cells_queue_entries(long long ncells) {
  const long long g = cells_grid(ncells);
  return g * ((ncells + g - 1) / g);
}

// A prime number of clusters of eight CTAs: about two CTAs per SM at least (small
// grids spread over all SMs) and no more than are resident at once (six per SM at
// 80 registers; 1016 CTAs left a second wave of 104, 37 us for 14400 cells where
// one wave takes half), between them as many as hold one pass of 16 cells each.
int cells_grid(long long ncells) {
  const long long want = (ncells + kCellSlots * kCellCluster - 1) / (kCellSlots * kCellCluster);
  for (int c : {41, 61, 79, 97})
    if (want <= c) return c * kCellCluster;
  return 113 * kCellCluster;
}

cudaError_t launch_cells(const SweepArgs& a, long long ncells, int mode, const MLPView* mlp, long long before,
                         cudaStream_t s) {
  const size_t sm = mode == kPartial ? 0
                              : (cta_solve_smem_doubles(a.th.nbp, a.th.ng, 1) + 2) * sizeof(double) +
                                    (mlp ? (2 * (size_t)a.th.nbp + 4 * kHidden) * sizeof(float) : 0);
  MLPView m{};
  if (mlp) m = *mlp;
  // Launched early behind a sweep of at most eight warps per SM: the launch and the
  // prologue are then hidden (ten inner iterations of 400 cells x 16 x 4, 60 CTAs of a warp, 221
  // -> 199 us; of 992 cells x 20 x 55, 124 CTAs of seven warps, 227 -> 224; six of 960 cells x
  // 120 x 27 in FP32, 480 CTAs of a warp, 235 -> 224).  Behind more of them the early CTAs crowd
  // into the slots that are left on some SMs (992 cells x 400 x 55, 248 CTAs of seven
  // warps, 1133 -> 1142 us, 3015 cells 2 % and 14400 cells 2.5 % slower).
  const bool early = before <= 152 * 256;
  return launch_pdl(early, mlp ? cells_kernel<true> : cells_kernel<false>, cells_grid(ncells), kCellThreads, sm, s, a, ncells,
                    mode, m);
}

}  // namespace bte
