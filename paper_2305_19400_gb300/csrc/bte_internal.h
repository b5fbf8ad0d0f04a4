// bte_internal.h -- definitions shared by the library's own translation units.
//
// Device data layout (all in one workspace, see bte_capi.cu):
//   I buffers      3 x [cell][dir][nbp]      storage type per precision mode
//                                            (FP32/BF16 store I - I0_b(T_ref))
//   I0cell         [cell][nbp]  double        I0_b(T_p) of every cell
//   J, Teval       [cell][4][nbp], [cell]     cached quadrature model per cell
//   Tp, TL, EL     [cell]       double        temperatures, lattice energy
//   I0wall         [wall face][nbp] double    Eq. 6 ghost for isothermal faces
//   coef           [class][5][dir][nbp] double  sweep coefficients (A_n, A_x, A_y, A_z, A_s)
//   node_c, node_C [nbp][ng]    double        Gauss nodes: hbar*omega/kB and weights
//   per-band / per-direction / per-geometry tables, work list, counters.
// dir is the internal direction order (internal_order, bte_tables.h); the
// caller's order appears only in what crosses the C ABI.
// nbp is nb rounded up to a multiple of 8, so one (cell, dir) row is a whole
// number of 16-byte vectors in every precision.  Padding bands carry zero
// coefficients and stay zero.
#pragma once
#include <cuda_runtime.h>
#include <cstddef>
#include <cstdint>

struct bte_ctx;

namespace bte {

constexpr double kHbar = 1.054571817e-34;  // J s (CODATA 2018)
constexpr double kBoltz = 1.380649e-23;    // J/K (CODATA 2018, exact)
constexpr double kPi = 3.14159265358979323846;
constexpr int kMaxGauss = 32;
constexpr int kMaxBands = 256;
constexpr double kTmin = 1.0, kTmax = 5000.0;  // bracket of the temperature solves

enum Side { XLO = 0, XHI = 1, YLO = 2, YHI = 3, ZLO = 4, ZHI = 5 };

// One geometry as the kernels see it.
struct DevGeom {
  int nx, ny, nz, dim;
  long long cell0;        // global index of the first cell
  long long face0[6];     // first global wall-face row of each side (isothermal sides)
  int bc[6];              // 0 ghost row (isothermal, diffuse), 1 mirror, 3 per-direction ghost rows
  int cls;                // coefficient-table class (cells with equal dx, dy, dz)
  int pad;
  const void* gdir[6];    // bc 3 (partially specular): [side face][dir][nbo] ghosts, storage type
};

// A run of consecutive cells of one geometry processed by one CTA.
struct WorkItem {
  int geom;
  int cell_begin;  // local cell index of (i0, j, k)
  int cell_count;  // cells along x
  int i0, j, k;
};

// Sweep-ordered (Gauss-Seidel) pass: one unit = the directions dir0 .. dir0+ndc-1
// of the octant list (all with the same upwind sides) over one geometry.
struct GsUnit {
  int geom;
  int dir0;  // first entry in SweepArgs::gs_dirs
  int ndc;   // directions in this unit (<= SweepArgs::gs_ndc)
  int pad;
};

// Per direction: bit a of `up` set when S_{d,a} > 0 (upwind neighbour on the low
// side along axis a); mirror directions across x, y, z walls.
struct DirInfo {
  int up;
  int rx, ry, rz;
};

// The directions of one wall side: those leaving through it (S_d . n_out > 0),
// then the rest, and the sums of |S_d,ax| over the leaving and the entering ones, each
// with the rounding error of its double: a wall's net flux is a small difference of
// these sums' multiples.
struct WallDirs {
  const int* out;   // [nout]
  const int* rest;  // [nd - nout]
  int nout;
  double sum_out, sum_in, sum_out_lo, sum_in_lo;
};

// A cell whose temperature its cached model could not settle.
struct FixItem {
  long long P;  // global cell
  double Ep;    // right-hand side of the T_p equation: sum_b beta_b G_b / v_b
  double T0;    // start temperature of the exact solve
  int model;    // 1: T0 is the cached model's root (a warm start); 0: the previous T_p
  int pad;
};

// Counters written by the kernels (atomics), read back for bte_stats.
struct DevCounters {
  unsigned long long evals;
  unsigned long long solves;
  unsigned long long fallbacks;
  unsigned long long nonfinite;
};

struct ThermoTables {
  const double* node_c;   // [nbp][ng] hbar*omega_i/kB (K)
  const double* node_C;   // [nbp][ng] I0_b(T) = sum_i node_C / expm1(node_c / T)
  const double* a_p;      // [nbp] W beta_b / v_b  (T_p equation weights)
  const double* a_L;      // [nbp] W / v_b         (T_L equation weights)
  const double* inv_v;    // [nbo] 1/v_b of the stored bands (0 on padding)
  const double* binv_v;   // [nbo] beta_b/v_b of the stored bands (0 on padding)
  double T_knee;          // hbar omega_max / (32 k_B): the trust radius shrinks below (model_trust)
  int ng;
  int nbp;    // all bands, padded: width of node tables, J, a_p and a_L
  int nb;     // all bands
  int nbo;    // bands this handle stores (padded): width of I rows, I0cell, wall ghosts
  int nbr;    // bands this handle stores (real): stored band b < nbr is global band band0 + b
  int band0;  // global index of the first stored band (0 unless the handle owns a band range)
};

struct SweepArgs {
  const void* In;           // I^n   (storage type; deviation from I0ref in the reduced modes)
  const void* Ik;           // I^k   (== In for the explicit scheme)
  void* Iout;               // I^{k+1}
  void* Bout;               // FP64, bmode 1: receives B = A_n I^n (the inner-iteration invariant term)
  int bmode;                // FP64 implicit: 0 In is I^n; 1 In is I^n and B is written; 2 In holds B
  double* I0cell;           // [cell][nbp] in: I0^k, out: I0^{k+1}
  double* Tp;               // [cell] in/out
  double* Teval;            // [cell] evaluation point of the cached quadrature model
  double* J;                // [cell][4][nbp] Taylor coefficients of I0_b(T) at Teval, to third order
  double* Msum;             // [cell][4] sum_b a_p,b J_k,b: the T_p model's sums, kept with J
  double* MsumL;            // [cell][4] the same with the T_L weights
  double* EL;               // [cell] out
  double* TL;               // [cell] T_L (on request)
  const double* Tguess;     // [cell] its start where the model has no root
  const double* I0wall;     // [face][nbp] FP64 ghosts
  const void* I0wall_ff;    // [face][nbp] FP64 ghosts as ff pairs (bte_ff.cuh)
  const float* I0wall_dev;  // [face][nbp] FP32 ghosts minus I0ref (reduced modes)
  const double* I0ref;      // [nbp] I0_b(T_ref) (reduced modes)
  int ff;                   // FP64: 1 double-float arithmetic (every intensity buffer holds ff pairs), 0 IEEE
  // tables of the double-float sweep in the pair layout of bte_ff.cuh
  // (h_b, h_b+1, l_b, l_b+1 per two bands):
  const void* coef_R;       // [cls][nd][nbp] R = 1/(1/(v_b dt) + beta_b/v_b + sum_ax c_ax,d), then W = R/(v_b dt), per two bands
  const float* band_ff;     // [nbp] beta_b/v_b of the stored bands (0 on padding)
  const float* dirc_ff;     // [cls][nd][3][2] c_ax,d as (h, l)
  const void* coef;         // FP64: [cls][5][nd][nbp] A_n, A_x, A_y, A_z, A_s;
                            // reduced: [cls][2][nd][nbp] float P, Q with
                            // I' = P I^n + Q (v_b sum_ax c_ax I_up + beta_b dI0)
  const float4* dirc;       // reduced: [cls][nd] (c_x, c_y, c_z, sum), c_ax = |S_d,ax|/(w_d Delta_ax)
  const float* vb32;        // [nbp] v_b (reduced)
  const float* bb32;        // [nbp] beta_b (reduced)
  double2* Ec;              // [cell][ne] partial (E_L, E_p), written by the sweeps (one per lane), added by cells_kernel
  FixItem* fix;             // cells_kernel's queue of exact solves, a part per CTA
  const DirInfo* dirs;
  const double* wdir;       // [nd]
  const float* wdir32;      // [nd]
  const DevGeom* geoms;
  const WorkItem* items;
  int nitems;
  int nd;
  int lpc;                  // lanes per direction row = nbp / values per lane
  int dteam;                // directions one cell team covers per step (team = lpc * dteam lanes)
  int dir_group;            // rows that differ only in the signs of S: 4 (in-plane sets) or 8 (internal_order)
  int ne;                   // entries per cell in Ec
  int solve_tp;             // 0 when every beta_b == 0 (T_p then unused)
  double trust_rel;         // cached model accepted when |T - T_e| <= trust_rel * T (model_trust)
  int maxit;
  double Wtot;              // sum of direction weights
  int partial;              // 1: band-range handle; per-cell partial (E_L, E_p) go to Epart[cell][2]
  double* Epart;            //    and the solve runs after the caller's all-reduce
  double beta_exp;          // beta_b(T) = beta_b (T_p / beta_Tref)^beta_exp per cell (0: fixed tau)
  double beta_Tref;
  int explicit_scheme;      // reduced modes compute P, Q on the fly from these:
  float dt32, rdt32;        // dt and 1/dt
  DevCounters* counters;
  // sweep-ordered pass (scheme BTE_IMPLICIT_GS, FP64)
  const GsUnit* gs_units;
  const int* gs_dirs;       // direction indices grouped by octant
  int gs_nunits;
  int gs_ndc;               // directions per unit (the CTA layout)
  int gs_tx, gs_ty;         // cross-section of a column tile (2-D: gs_tx cells along x)
  double* bscale;           // [cell] beta_b(T_p)/beta_b (beta_exp != 0), kept current by cells_kernel
  ThermoTables th;
};

// Launchers (bte_kernels.cu).  precision: BTE_FP64 = 0, BTE_FP32 = 1, BTE_BF16 = 2.
int values_per_lane(int precision);
// Raises the dynamic shared memory limit of kernel func on the current device
// to at least bytes (no call below 48 KB).  The limit only grows, under a
// lock: handles on several host threads launch the same kernel with different
// needs, and a per-launch setting could lower another thread's limit between
// its own setting and its launch.
cudaError_t raise_dynamic_smem(const void* func, size_t bytes);
// grid <= 0 (FP64, FP32): as many CTAs as are resident
cudaError_t launch_sweep(int precision, int pd, const SweepArgs& a, int dim, int threads, int grid, cudaStream_t s);
cudaError_t launch_sweep_fp64(const SweepArgs& a, int dim, int threads, int grid, cudaStream_t s);
cudaError_t launch_sweep_fp32(const SweepArgs& a, int dim, int threads, int grid, cudaStream_t s);
cudaError_t launch_sweep_bf16(int pd, const SweepArgs& a, int dim, int threads, int grid, cudaStream_t s);
struct MLPView;
// per-cell step (bte_cells.cu): mode 0 energies from Ec and T_p, 1 energies from
// Ec to Epart, 2 T_p from Epart, 3 T_L from E_L
// before: threads of the kernel that runs before it, 0 where that one lets nothing start before its end
cudaError_t launch_cells(const SweepArgs& a, long long ncells, int mode, const MLPView* mlp, long long before,
                         cudaStream_t s);
int cells_grid(long long ncells);
long long cells_queue_entries(long long ncells);  // FixItems of a.fix
// sweep-ordered pass (bte_gs.cu) and its sums (bte_kernels.cu): the pass writes
// Iout, the reduction kRedEntries partial energies per cell to Ec
constexpr int kRedEntries = 8;
cudaError_t launch_gs_sweep(int precision, const SweepArgs& a, int dim, int threads, cudaStream_t s);
cudaError_t launch_gs_reduce(int precision, const SweepArgs& a, long long ncells, cudaStream_t s);
cudaError_t launch_beta_scale(double* out, const double* Tp, double Tref, double p, long long ncells, cudaStream_t s);
cudaError_t launch_diffuse_ghosts(int precision, const void* I, const double* I0ref, double* I0wall, float* I0wall_dev,
                                  const DevGeom* geoms, int geom, int side, const double* Sd, const WallDirs& wd, int nd,
                                  int nbp, int nfaces, cudaStream_t s);
// Partially specular side: per face, entering direction and band, p x the cell's
// mirrored value + (1 - p) x the diffuse value, into out [face][dir][nbp] (storage type).
cudaError_t launch_partial_ghosts(int precision, const void* I, const double* I0ref, const DevGeom* geoms, int geom,
                                  int side, const double* Sd, const WallDirs& wd, const DirInfo* dirs, int nd, int nbp,
                                  int nfaces, double p, void* out, cudaStream_t s);
// learned guess (bte_mlp.cu)
int mlp_param_total(int nb);
cudaError_t launch_mlp_norm(ThermoTables th, double T_lo, double T_hi, const double* I0ref, double* r_lo, double* r_hi,
                            double* E_lohi, cudaStream_t s);
cudaError_t launch_mlp_pairs(ThermoTables th, double T_lo, double T_hi, const double* I0ref, const double* r_lo,
                             const double* r_hi, const double* E_lohi, unsigned long long seed, int n, float* xA,
                             float* yA, float* yB, cudaStream_t s);
cudaError_t mlp_forward_backward(const float* p, int k, const float* X, int ldx, const float* Tg, int ldt, int B,
                                 float* grad, float* act, float* part, cudaStream_t s);
cudaError_t launch_adam(float* p, const float* g, float* m, float* v, int n, float lr, int step, cudaStream_t s);
cudaError_t launch_solve_batch(ThermoTables th, const double* Ep, const double* T0, int n, double trust_rel, int maxit,
                               const MLPView* mlp, double* Tout, int* evals, cudaStream_t s);
// ff: FP64 intensities as ff pairs
cudaError_t launch_init_cells(int precision, bool ff, void* I, double* I0cell, double* J, double* Msum, double* MsumL, double* Tp, double* Te,
                              double* TL, double* EL, const double* Tcells, const double* I0ref, long long cell0,
                              int ncells, int nd, ThermoTables th, cudaStream_t s);
cudaError_t launch_refill(bool ff, void* I, const double* I0cell, long long ncells, int nd, int nbo, cudaStream_t s);
cudaError_t launch_state_from_Tp(double* I0cell, double* J, double* Msum, double* MsumL, const double* Tp, double* Te, long long ncells,
                                 ThermoTables th, cudaStream_t s);
cudaError_t launch_wall_I0(double* I0wall, const double* Tfaces, long long nfaces, ThermoTables th, cudaStream_t s);
cudaError_t launch_wall_dev(float* out, const double* I0wall, const double* I0ref, long long nfaces, int nbp,
                            cudaStream_t s);
// state_ff: the FP64 intensities are ff pairs (bte_ff.cuh); grouped: rows in the internal order
cudaError_t launch_flux_cells(int precision, bool state_ff, bool grouped, const void* I, double* q, const double* S, long long cell0,
                              int ncells, int nd, int nbp, int dim, cudaStream_t s);
// every side of one geometry: face sums to face_out[side][max_faces], means to out[side]
cudaError_t launch_flux_walls(int precision, bool state_ff, const void* I, const double* I0ref, const double* I0wall,
                              const DevGeom* geoms, int geom, const WallDirs* wall_dirs, const double* S, int nd, int nbp,
                              double* face_out, int max_faces, const int (&nfaces)[6], int nsides, double* out,
                              cudaStream_t s);
// In place: npairs 16-byte ff pairs of two bands (bte_ff.cuh layout) -> two doubles each.
cudaError_t launch_ff_to_doubles(void* buf, long long npairs, cudaStream_t s);
// npairs x two doubles -> ff pairs (dst may be src)
cudaError_t launch_doubles_to_ff(const void* src, void* dst, long long npairs, cudaStream_t s);
// FP64 [cell][caller's d][nb] <-> internal rows; perm: the caller's index of every internal direction
cudaError_t launch_unpack(int precision, bool state_ff, const void* I, double* out, const double* I0ref, const int* rows,
                          long long ncells, int nd, int nb, int nbp, cudaStream_t s);
cudaError_t launch_pack(int precision, const double* in, void* I, const double* I0ref, const int* rows,
                        long long ncells, int nd, int nb, int nbp, const SweepArgs* energies, cudaStream_t s);
// E_L of every cell from its partial energies (launch_gs_reduce's or launch_pack's Ec)
cudaError_t launch_energy_L(const double2* Ec, double* EL, long long ncells, cudaStream_t s);

// Read-only view of one geometry's device state, for entry points that live
// outside bte_capi.cu (bte_noalloc.cu).  flux_view returns BTE_E_* codes.
struct FluxView {
  int precision;          // storage of I (BTE_FP64 = 0, BTE_FP32 = 1, BTE_BF16 = 2)
  const void* I;          // current intensity buffer (padded rows)
  bool state_ff;          // FP64: it holds ff pairs
  const double* I0wall;
  const DevGeom* geoms;
  WallDirs wall_dirs[6];
  const double* S;        // [nd][3]
  int nd, nbp, dim;
  int nfaces[6];          // faces per side (0 for sides beyond 2*dim)
  cudaStream_t stream;
  int dev;                // device that holds the handle's memory and stream
};
int flux_view(bte_ctx* h, int geom, FluxView* out);
int handle_device(bte_ctx* h);  // device that was current at bte_init_mesh
int set_handle_error(bte_ctx* h, int code, const char* fmt, ...);

}  // namespace bte
