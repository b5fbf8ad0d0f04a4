// bte_capi.cu -- the extern "C" entry points of libbte (declared in include/bte.h).
//
// A handle owns: the host copies of the direction and band tables, the
// per-geometry bookkeeping, and one device workspace (caller-bound or
// library-allocated) carved into the buffers listed in bte_internal.h.  Every
// kernel and copy goes to the stream given in bte_opts.
#include <algorithm>
#include <array>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <numeric>
#include <string>
#include <tuple>
#include <vector>

#include "../../include/bte.h"
#include "bte_internal.h"
#include "bte_mlp.cuh"
#include "bte_solve.cuh"
#include "bte_tables.h"

using namespace bte;

struct bte_ctx {
  std::string err;
  int dev = 0;
  cudaStream_t stream = nullptr;
  bte_opts opts{};
  // geometry
  std::vector<bte_geom> geoms;
  std::vector<long long> cell0;
  std::vector<long long> face0;  // [geom*6 + side]
  std::vector<int> cls;
  std::vector<std::tuple<int, double, double, double>> cls_key;
  long long ncells = 0, nfaces = 0;
  int max_side_faces = 0, max_geom_cells = 0;
  // directions
  int nd = 0;
  std::vector<double> S, w;
  std::vector<int> refl;
  std::vector<int> perm;       // the caller's index of every internal direction
  double Wtot = 0.0;
  double T_knee = 0.0;         // ThermoTables::T_knee
  // bands
  int nb = 0, nbp = 0, ng = 16;           // bands stored by this handle (padded: nbp)
  int nb_all = 0, nbp_all = 0, band0 = 0; // every band of the table; first stored band
  bte_allreduce_fn exchange = nullptr;    // band-range handles: sums per-cell partials over ranks
  void* exchange_user = nullptr;
  double* exchange_buf = nullptr;         // caller's device array for the partials (else Epart)
  int exchange_rc = 0;                    // last non-zero return of the exchange callback
  bool EL_partial = false;                // E_L not yet summed over the ranks (after bte_set_intensity)
  std::vector<double> wlo, whi, vg, beta, deg;
  bool solve_tp = false;
  // state
  bool bands_set = false;
  std::vector<std::array<int, 6>> bc_type;
  std::vector<std::array<bool, 6>> bc_set;
  std::vector<std::array<double, 6>> spec;   // specularity of partially specular sides
  std::vector<std::array<void*, 6>> gdir;    // their per-direction ghost rows (cudaMalloc, owned)
  std::vector<bool> init_set;
  bool TL_valid = false;
  // launch shape
  int lpc = 0, dteam = 1, cpb = 0, threads = 0, grid = 0, pd = 1;  // grid 0 (FP64, FP32): the resident CTAs
  int dir_group = 8;                                               // rows per block of the internal order
  // CUDA graphs of one time step, keyed by (scheme, ninner, starting buffer)
  struct GraphEntry {
    int scheme, ninner, cur_in, cur_out;
    bool ff_in;  // the state holds ff pairs
    cudaGraphExec_t exec;
  };
  std::vector<GraphEntry> graphs;
  cudaStream_t cap_stream = nullptr;
  std::string tune_report;
  std::vector<WorkItem> items;
  // sweep-ordered pass: directions grouped by octant, units, CTA layout and tiles
  std::vector<int> gs_dirs;
  std::vector<GsUnit> gs_units;
  int gs_ndc = 1, gs_tx = 128, gs_ty = 1, gs_threads = 0;
  std::string gs_tune_report;
  // device memory
  char* ws = nullptr;
  size_t ws_bytes = 0;
  bool ws_owned = false, mem_ready = false;
  char* Ibuf[3] = {nullptr, nullptr, nullptr};
  int cur = 0;
  // FP64 handles whose Jacobi steps run in double-float arithmetic keep the
  // current intensity buffer as ff pairs between such steps; steps of another
  // arithmetic convert it (ensure_state_doubles), a restored state is kept as doubles
  // until a double-float step (ensure_state_ff).  An initial state (initial: no geometry has
  // been stepped or restored since bte_set_initial) is I0cell in every direction and
  // written again from there, in either form: no rounding of one shows in the other
  bool state_ff = false, initial = false;
  double *I0cell = nullptr, *Tp = nullptr, *TL = nullptr, *EL = nullptr, *I0wall = nullptr;
  void* coef = nullptr;
  // FP64: tables of the factored double-float sweep (bte_rows.cuh)
  void* coef_R = nullptr;     // [cls][nd][nbp] R and W pairs
  float* dirc_ff = nullptr;   // [cls][nd][3][2]
  float* band_ff = nullptr;   // [nbp] beta_b/v_b pairs
  double *J = nullptr, *Teval = nullptr, *I0ref = nullptr, *scratch_pack = nullptr;
  double* Msum = nullptr;     // [cell][4] the T_p model's sums sum_b a_p,b J_k,b
  double* MsumL = nullptr;    // [cell][4] the same with the T_L weights
  double* I0ref_o = nullptr;  // I0_b(T_ref) of the stored bands (aliases I0ref unless a band range is set)
  double* Epart = nullptr;    // band-range handles: [ncells][2] partial (E_L, E_p) for the exchange
  float *I0wall_dev = nullptr, *wdir32 = nullptr, *vb32 = nullptr, *bb32 = nullptr;
  float4* dirc = nullptr;
  FixItem* fix = nullptr;
  double2* Ec = nullptr;      // [cell][entries] partial energies of the sweeps
  void* I0wall_ff = nullptr;  // FP64: [face][nbp] isothermal ghosts as ff pairs
  // learned guess: parameters of nets A and B, Adam state, normalisation
  float *mlp_p = nullptr, *mlp_g = nullptr, *mlp_m = nullptr, *mlp_v = nullptr;
  double *mlp_rlo = nullptr, *mlp_rhi = nullptr, *mlp_elohi = nullptr;
  bool mlp_trained = false;
  double mlp_Tlo = 0.0, mlp_Thi = 0.0, mlp_Elo = 0.0, mlp_Ehi = 0.0;
  long long pack_cells = 0;
  double *wdir = nullptr, *Sdev = nullptr, *node_c = nullptr, *node_C = nullptr, *a_p = nullptr, *a_L = nullptr;
  double *inv_v = nullptr, *binv_d = nullptr, *scratch_faces = nullptr, *scratch_T = nullptr, *scratch_out = nullptr;
  double* scratch_q = nullptr;
  std::vector<DevGeom> dgeoms;
  DirInfo* dirs_d = nullptr;
  int* rows_d = nullptr;
  int* wall_dirs_d = nullptr;   // [6][nd] per side: leaving directions, then the rest
  std::array<WallDirs, 6> wall_dirs{};
  DevGeom* geoms_d = nullptr;
  WorkItem* items_d = nullptr;
  DevCounters* counters = nullptr;
  GsUnit* gs_units_d = nullptr;
  int* gs_dirs_d = nullptr;
  double* bscale = nullptr;  // [cell] beta_b(T_p)/beta_b, kept current by cells_kernel once valid
  bool bscale_valid = false;
  // coefficient cache
  double coef_dt = -1.0;
  int coef_scheme = -1;
  std::vector<double> coef_host;
  std::vector<float> R_host, dirc_host, band_host;
  // per-launch timing of the sweeps (bte_set_sweep_timing): events around each
  // sweep of a step, recorded on the stream (captured into the step's graph)
  bool time_sweeps = false;
  std::vector<cudaEvent_t> tev;
  int tev_n = 0;  // sweeps the events of the last step cover
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;
};

namespace {

thread_local std::string g_init_err;

int fail(bte_ctx* h, int code, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  if (h) h->err = buf; else g_init_err = buf;
  return code;
}

#define CUDA_TRY(h, call)                                                                        \
  do {                                                                                           \
    cudaError_t e_ = (call);                                                                     \
    if (e_ != cudaSuccess) return fail((h), BTE_E_CUDA, "%s: %s", #call, cudaGetErrorString(e_)); \
  } while (0)

size_t elem_bytes(int precision) { return precision == BTE_FP64 ? 8 : (precision == BTE_FP32 ? 4 : 2); }

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

long long side_faces(const bte_geom& g, int side) {
  if (side < 2) return (long long)g.ny * g.nz;
  if (side < 4) return (long long)g.nx * g.nz;
  return (long long)g.nx * g.ny;
}

ThermoTables thermo(const bte_ctx* h) {
  ThermoTables t;
  t.node_c = h->node_c;
  t.node_C = h->node_C;
  t.a_p = h->a_p;
  t.a_L = h->a_L;
  t.inv_v = h->inv_v;
  t.binv_v = h->binv_d;
  t.T_knee = h->T_knee;
  t.ng = h->ng;
  t.nbp = h->nbp_all;
  t.nb = h->nb_all;
  t.nbo = h->nbp;
  t.nbr = h->nb;
  t.band0 = h->band0;
  return t;
}

// The same tables seen as a handle storing every band (for all-band outputs).
ThermoTables thermo_all(const bte_ctx* h) {
  ThermoTables t = thermo(h);
  t.nbo = h->nbp_all;
  t.nbr = h->nb_all;
  t.band0 = 0;
  return t;
}

// Teams a cell of the FP64 and FP32 sweeps may have (bte_rows.cuh): one on in-plane
// sets, two (FP32 also four) on polar x azimuthal ones; the BF16 sweep adds its
// teams' sums itself.
int max_teams(const bte_ctx* h) {
  if (h->opts.precision == BTE_BF16 || h->dir_group == 4) return 1;
  return h->opts.precision == BTE_FP64 ? 2 : 4;
}

// Workspace layout; with base == nullptr only the size is computed.
size_t carve(bte_ctx* h, char* base) {
  size_t off = 0;
  auto take = [&](size_t bytes) -> char* {
    char* p = base ? base + off : nullptr;
    off += align256(bytes);
    return p;
  };
  const size_t row = (size_t)h->nd * h->nbp;
  const size_t ibytes = (size_t)h->ncells * row * elem_bytes(h->opts.precision);
  for (int i = 0; i < 3; ++i) h->Ibuf[i] = take(ibytes);
  h->I0cell = (double*)take((size_t)h->ncells * h->nbp * 8);
  h->J = (double*)take((size_t)h->ncells * 4 * h->nbp_all * 8);
  h->Teval = (double*)take((size_t)h->ncells * 8);
  h->Msum = (double*)take((size_t)h->ncells * 4 * 8);
  h->MsumL = (double*)take((size_t)h->ncells * 4 * 8);
  h->I0ref = (double*)take((size_t)h->nbp_all * 8);
  const bool ranged = h->nb != h->nb_all;
  h->I0ref_o = ranged ? (double*)take((size_t)h->nbp * 8) : h->I0ref;
  h->Epart = ranged ? (double*)take((size_t)std::max(h->ncells, 1LL) * 2 * 8) : nullptr;
  h->I0wall_dev = (float*)take((size_t)std::max(h->nfaces, 1LL) * h->nbp * 4);
  h->wdir32 = (float*)take((size_t)h->nd * 4);
  h->Tp = (double*)take((size_t)h->ncells * 8);
  h->TL = (double*)take((size_t)h->ncells * 8);
  h->EL = (double*)take((size_t)h->ncells * 8);
  h->I0wall = (double*)take((size_t)std::max(h->nfaces, 1LL) * h->nbp * 8);
  h->coef = take((size_t)h->cls_key.size() * row * (h->opts.precision == BTE_FP64 ? 5 * 8 : 2 * 4));
  h->coef_R = h->opts.precision == BTE_FP64 ? take((size_t)h->cls_key.size() * row * 16) : nullptr;
  h->dirc_ff = h->opts.precision == BTE_FP64 ? (float*)take((size_t)h->cls_key.size() * h->nd * 6 * 4) : nullptr;
  h->band_ff = h->opts.precision == BTE_FP64 ? (float*)take((size_t)h->nbp * 2 * 4) : nullptr;
  h->dirc = (float4*)take((size_t)h->cls_key.size() * h->nd * sizeof(float4));
  h->vb32 = (float*)take((size_t)h->nbp * 4);
  h->bb32 = (float*)take((size_t)h->nbp * 4);
  h->fix = (FixItem*)take((size_t)cells_queue_entries(h->ncells) * sizeof(FixItem));
  h->Ec = (double2*)take((size_t)std::max(h->ncells, 1LL) *
                         std::max(kRedEntries, max_teams(h) * h->nbp / values_per_lane(h->opts.precision)) * 16);
  h->I0wall_ff = h->opts.precision == BTE_FP64 ? take((size_t)std::max(h->nfaces, 1LL) * h->nbp * 8) : nullptr;
  const size_t np = (size_t)mlp_param_total(h->nb_all);
  h->mlp_p = (float*)take(np * 4);
  h->mlp_g = (float*)take(np * 4);
  h->mlp_m = (float*)take(np * 4);
  h->mlp_v = (float*)take(np * 4);
  h->mlp_rlo = (double*)take((size_t)h->nbp_all * 8);
  h->mlp_rhi = (double*)take((size_t)h->nbp_all * 8);
  h->mlp_elohi = (double*)take(16);
  h->wdir = (double*)take((size_t)h->nd * 8);
  h->Sdev = (double*)take((size_t)h->nd * 3 * 8);
  h->dirs_d = (DirInfo*)take((size_t)h->nd * sizeof(DirInfo));
  h->wall_dirs_d = (int*)take((size_t)h->nd * 6 * 4);
  h->rows_d = (int*)take((size_t)h->nd * 4);
  h->node_c = (double*)take((size_t)h->nbp_all * h->ng * 8);
  h->node_C = (double*)take((size_t)h->nbp_all * h->ng * 8);
  h->a_p = (double*)take((size_t)h->nbp_all * 8);
  h->a_L = (double*)take((size_t)h->nbp_all * 8);
  h->inv_v = (double*)take((size_t)h->nbp * 8);   // stored bands
  h->binv_d = (double*)take((size_t)h->nbp * 8);
  h->geoms_d = (DevGeom*)take(h->geoms.size() * sizeof(DevGeom));
  h->items_d = (WorkItem*)take((size_t)std::max<long long>(h->ncells, 1) * sizeof(WorkItem));  // room for 1 cell per item
  h->counters = (DevCounters*)take(sizeof(DevCounters));
  h->gs_units_d = (GsUnit*)take(std::max<size_t>(h->geoms.size() * h->nd, 1) * sizeof(GsUnit));
  h->gs_dirs_d = (int*)take((size_t)h->nd * 4);
  h->bscale = (double*)take((size_t)std::max(h->ncells, 1LL) * 8);
  h->scratch_faces = (double*)take((size_t)std::max(h->max_side_faces, 1) * 6 * 8);
  h->scratch_T = (double*)take((size_t)std::max(h->max_side_faces, h->max_geom_cells) * 8);
  h->scratch_out = (double*)take(64);
  h->scratch_q = (double*)take((size_t)std::max(h->max_geom_cells, 1) * 3 * 8);
  // host <-> device staging of whole cell rows in the caller's order (64 MB at most)
  h->pack_cells = std::max(1LL, std::min<long long>(h->max_geom_cells, (64LL << 20) / ((long long)h->nd * h->nb * 8)));
  h->scratch_pack = (double*)take((size_t)h->pack_cells * h->nd * h->nb * 8);
  return off;
}

// Work list: runs of at most cpb consecutive cells along x.  2-D geometries are
// walked in strips of 64 columns, row by row within a strip, so the upwind
// row is at most 64 cells back (35 MB of the three intensity arrays in FP64
// at 400 x 56) and more of it is still in L2 (measured on the 128x128 FP64
// workload: 25.45 -> 24.58 ms per step against whole rows).  3-D
// geometries are walked in column blocks of bx x by cells marching in z, so
// the z-upwind plane of a block (bx*by cells back) is still in L2 when reused.
constexpr int kStrip2D = 64;
void build_items(bte_ctx* h, int cpb = 0, int dteam = 0) {
  h->lpc = h->nbp / values_per_lane(h->opts.precision);  // one vector of bands per lane
  const int rowb = h->nbp * (int)elem_bytes(h->opts.precision);
  if (dteam > 0) h->dteam = dteam;
  else if (h->opts.precision == BTE_BF16)  // ~896 contiguous bytes of a row, at least ~32 steps per lane
    h->dteam = std::max(1, std::min(std::min(896 / rowb, 256 / h->lpc), h->nd / 32));
  else  // IEEE sweeps share a block's coefficients over all of its rows: they wait for the FP64 pipe
    h->dteam = h->dir_group == 4 || (h->opts.precision == BTE_FP64 && (h->opts.fp64_strict || h->opts.beta_T_exp != 0.0)) ? 1 : 2;
  const int team = h->lpc * h->dteam;
  // default: the most cells whose CTA (at most 256 threads) is whole warps, else
  // the most that fit; small grids take fewer, so that every SM has two CTAs
  const int whole = 32 / std::gcd(team, 32);
  const int cpb_whole = (256 / team) / whole * whole;
  h->cpb = cpb > 0 ? cpb : (cpb_whole > 0 ? cpb_whole : std::max(1, 256 / team));
  if (cpb <= 0 && h->opts.precision != BTE_BF16)
    while (h->cpb > whole && h->ncells < 2LL * 152 * h->cpb) h->cpb -= whole;
  h->threads = h->cpb * team;
  h->items.clear();
  for (size_t gi = 0; gi < h->geoms.size(); ++gi) {
    const bte_geom& g = h->geoms[gi];
    if (g.nz == 1) {  // strips of kStrip2D columns, row by row within a strip
      const int bx = std::max(h->cpb, kStrip2D / h->cpb * h->cpb);
      for (int i0 = 0; i0 < g.nx; i0 += bx)
        for (int j = 0; j < g.ny; ++j)
          for (int i = i0; i < std::min(g.nx, i0 + bx); i += h->cpb)
            h->items.push_back(WorkItem{(int)gi, j * g.nx + i, std::min(h->cpb, std::min(g.nx, i0 + bx) - i), i, j, 0});
      continue;
    }
    // blocks of bx x by = 256 cells (bx a multiple of cpb, near square): the z
    // plane of a block stays in L2, and few upwind rows cross a block edge
    const int bx = std::max(h->cpb, 16 / h->cpb * h->cpb), by = std::max(1, 256 / bx);
    for (int j0 = 0; j0 < g.ny; j0 += by)
      for (int i0 = 0; i0 < g.nx; i0 += bx)
        for (int k = 0; k < g.nz; ++k)
          for (int j = j0; j < std::min(g.ny, j0 + by); ++j)
            for (int i = i0; i < std::min(g.nx, i0 + bx); i += h->cpb)
              h->items.push_back(
                  WorkItem{(int)gi, (k * g.ny + j) * g.nx + i, std::min(h->cpb, std::min(g.nx, i0 + bx) - i), i, j, k});
  }
  // One CTA per item, started in order: the cells in flight stay close together and
  // find their neighbours' rows in L2.  Resident CTAs that stride over the items drift
  // apart: 128x128 x 400 x 55 in FP64, a step's first iteration (I^n = I^k) 1372 us and 23.0
  // DRAM bytes an update against 1102 and 17.5, the others 1782 and 30.9 against 1430 and
  // 26.4; 32^3 in FP32 1450 and 2203 us against 1171 and 1584.  In-plane sets, whose items are
  // short and whose ring would drain, take the resident CTAs (120x120 x 20 x 55, first
  // and others: IEEE 146 and 115 us against 163 and 131, double-float 73 and 86 against 77
  // and 84).
  const bool persistent = h->opts.precision != BTE_BF16 && h->dir_group == 4;
  h->grid = persistent ? 0 : (int)std::min<size_t>(h->items.size(), 65535);
}

// Sweep-ordered pass.  Directions whose upwind sides agree (one octant) share
// a visiting order; a unit is up to ndc of them over one geometry, one CTA per
// unit.  2-D grids are walked in strips of tx columns, 3-D grids in tx x ty
// column tiles.  The CTA has lpc/2 lanes per (cell, direction) row (two FP64
// bands per lane) and as many cell slots as fit 256 threads.
void build_gs(bte_ctx* h, int ndc, int tx, int ty) {
  int dim = 2;
  for (auto& g : h->geoms) dim = std::max(dim, g.dim);
  const int noct = 1 << dim;
  h->gs_dirs.clear();
  h->gs_units.clear();
  std::vector<int> start(noct + 1, 0);
  for (int o = 0; o < noct; ++o) {
    start[o] = (int)h->gs_dirs.size();
    for (int d = 0; d < h->nd; ++d) {
      const int up = (h->S[3 * d] > 0) | ((h->S[3 * d + 1] > 0) << 1) | ((h->S[3 * d + 2] > 0) << 2);
      if ((up & (noct - 1)) == o) h->gs_dirs.push_back(d);
    }
  }
  start[noct] = (int)h->gs_dirs.size();
  const int lanes = h->nbp / values_per_lane(h->opts.precision);
  ndc = std::max(1, std::min(ndc, 256 / lanes));
  for (size_t gi = 0; gi < h->geoms.size(); ++gi)
    for (int o = 0; o < noct; ++o)
      for (int c = start[o]; c < start[o + 1]; c += ndc)
        h->gs_units.push_back(GsUnit{(int)gi, c, std::min(ndc, start[o + 1] - c), 0});
  h->gs_ndc = ndc;
  h->gs_tx = std::max(1, tx);
  h->gs_ty = std::max(1, ty);
  const int team = lanes * ndc;
  h->gs_threads = team * std::max(1, 256 / team);
}

int upload_gs(bte_ctx* h, cudaStream_t s) {
  CUDA_TRY(h, cudaMemcpyAsync(h->gs_dirs_d, h->gs_dirs.data(), h->gs_dirs.size() * 4, cudaMemcpyHostToDevice, s));
  CUDA_TRY(h, cudaMemcpyAsync(h->gs_units_d, h->gs_units.data(), h->gs_units.size() * sizeof(GsUnit),
                              cudaMemcpyHostToDevice, s));
  CUDA_TRY(h, cudaStreamSynchronize(s));
  return BTE_OK;
}

// Wall codes the kernels read: a diffuse side reads its (refreshed) ghost row
// like an isothermal one (0); a partially specular side its per-direction rows (3).
int dev_bc(int type) { return type == BTE_BC_DIFFUSE ? 0 : (type == BTE_BC_PARTIAL ? 3 : type); }

void drop_graphs(bte_ctx* h) {
  for (auto& e : h->graphs) cudaGraphExecDestroy(e.exec);
  h->graphs.clear();
}

int ensure_memory(bte_ctx* h) {
  if (h->mem_ready) return BTE_OK;
  if (!h->bands_set) return fail(h, BTE_E_STATE, "bte_set_bands must come first");
  const size_t need = carve(h, nullptr);
  if (!h->ws) {
    void* p = nullptr;
    cudaError_t e = cudaMalloc(&p, need);
    if (e != cudaSuccess) return fail(h, BTE_E_NOMEM, "cudaMalloc(%zu bytes): %s", need, cudaGetErrorString(e));
    h->ws = (char*)p;
    h->ws_bytes = need;
    h->ws_owned = true;
  }
  carve(h, h->ws);
  cudaStream_t s = h->stream;
  // I buffers start at zero so padding bands are zero everywhere.
  const size_t ibytes = (size_t)h->ncells * h->nd * h->nbp * elem_bytes(h->opts.precision);
  for (int i = 0; i < 3; ++i) CUDA_TRY(h, cudaMemsetAsync(h->Ibuf[i], 0, ibytes, s));
  CUDA_TRY(h, cudaMemsetAsync(h->I0wall, 0, (size_t)std::max(h->nfaces, 1LL) * h->nbp * 8, s));
  // direction tables
  std::vector<DirInfo> di(h->nd);
  for (int d = 0; d < h->nd; ++d) {
    di[d].up = (h->S[3 * d] > 0) | ((h->S[3 * d + 1] > 0) << 1) | ((h->S[3 * d + 2] > 0) << 2);
    di[d].rx = h->refl[d];
    di[d].ry = h->refl[h->nd + d];
    di[d].rz = h->refl[2 * h->nd + d];
  }
  CUDA_TRY(h, cudaMemcpyAsync(h->dirs_d, di.data(), di.size() * sizeof(DirInfo), cudaMemcpyHostToDevice, s));
  std::vector<int> wl((size_t)6 * h->nd);
  for (int side = 0; side < 6; ++side) {
    WallDirs& wd = h->wall_dirs[side];
    int* l = wl.data() + (size_t)side * h->nd;
    wd = WallDirs{h->wall_dirs_d + (size_t)side * h->nd, nullptr, 0, 0.0, 0.0, 0.0, 0.0};
    const auto add = [](double& s, double& lo, double x) {  // TwoSum
      const double t = s + x, v = t - s;
      lo += (s - (t - v)) + (x - v);
      s = t;
    };
    int nrest = 0;
    for (int d = 0; d < h->nd; ++d) {
      const double sn = (side & 1) ? h->S[3 * d + side / 2] : -h->S[3 * d + side / 2];
      if (sn > 0.0) { l[wd.nout++] = d; add(wd.sum_out, wd.sum_out_lo, sn); }
      else { l[h->nd - ++nrest] = d; add(wd.sum_in, wd.sum_in_lo, -sn); }
    }
    std::reverse(l + wd.nout, l + h->nd);
    wd.rest = wd.out + wd.nout;
  }
  std::vector<int> rows(h->perm.size());  // the internal row of each of the caller's directions
  for (size_t p = 0; p < rows.size(); ++p) rows[h->perm[p]] = (int)p;
  CUDA_TRY(h, cudaMemcpyAsync(h->rows_d, rows.data(), rows.size() * 4, cudaMemcpyHostToDevice, s));
  CUDA_TRY(h, cudaMemcpyAsync(h->wall_dirs_d, wl.data(), wl.size() * 4, cudaMemcpyHostToDevice, s));
  CUDA_TRY(h, cudaMemcpyAsync(h->wdir, h->w.data(), h->nd * 8, cudaMemcpyHostToDevice, s));
  CUDA_TRY(h, cudaMemcpyAsync(h->Sdev, h->S.data(), h->nd * 3 * 8, cudaMemcpyHostToDevice, s));
  // band tables
  std::vector<double> nc, nC, ap, aL, iv, be;
  build_thermo(h->nb_all, h->nbp_all, h->ng, h->wlo.data(), h->whi.data(), h->vg.data(), h->beta.data(),
               h->deg.data(), h->Wtot, nc, nC, ap, aL, iv, be);
  h->T_knee = model_knee(nc, h->nb_all, h->ng);
  CUDA_TRY(h, cudaMemcpyAsync(h->node_c, nc.data(), nc.size() * 8, cudaMemcpyHostToDevice, s));
  CUDA_TRY(h, cudaMemcpyAsync(h->node_C, nC.data(), nC.size() * 8, cudaMemcpyHostToDevice, s));
  CUDA_TRY(h, cudaMemcpyAsync(h->a_p, ap.data(), ap.size() * 8, cudaMemcpyHostToDevice, s));
  CUDA_TRY(h, cudaMemcpyAsync(h->a_L, aL.data(), aL.size() * 8, cudaMemcpyHostToDevice, s));
  {
    std::vector<double> iv_o(h->nbp, 0.0), bi_o(h->nbp, 0.0);  // stored bands, zero on padding
    for (int b = 0; b < h->nb; ++b) {
      iv_o[b] = iv[h->band0 + b];
      bi_o[b] = be[h->band0 + b] * iv_o[b];
    }
    CUDA_TRY(h, cudaMemcpyAsync(h->binv_d, bi_o.data(), bi_o.size() * 8, cudaMemcpyHostToDevice, s));
    CUDA_TRY(h, cudaMemcpyAsync(h->inv_v, iv_o.data(), iv_o.size() * 8, cudaMemcpyHostToDevice, s));
    CUDA_TRY(h, cudaStreamSynchronize(s));
  }
  {
    std::vector<float> v32(h->nbp, 0.f), b32(h->nbp, 0.f);  // stored bands
    for (int b = 0; b < h->nb; ++b) { v32[b] = (float)h->vg[h->band0 + b]; b32[b] = (float)h->beta[h->band0 + b]; }
    CUDA_TRY(h, cudaMemcpyAsync(h->vb32, v32.data(), v32.size() * 4, cudaMemcpyHostToDevice, s));
    CUDA_TRY(h, cudaMemcpyAsync(h->bb32, b32.data(), b32.size() * 4, cudaMemcpyHostToDevice, s));
    CUDA_TRY(h, cudaStreamSynchronize(s));
  }
  {
    std::vector<float> w32(h->w.begin(), h->w.end());
    CUDA_TRY(h, cudaMemcpyAsync(h->wdir32, w32.data(), w32.size() * 4, cudaMemcpyHostToDevice, s));
    // I0_b(T_ref): the reference the reduced-precision modes store deviations from
    const double tref = h->opts.T_ref;
    CUDA_TRY(h, cudaMemcpyAsync(h->scratch_T, &tref, 8, cudaMemcpyHostToDevice, s));
    CUDA_TRY(h, launch_wall_I0(h->I0ref, h->scratch_T, 1, thermo_all(h), s));
    if (h->I0ref_o != h->I0ref) {
      CUDA_TRY(h, cudaMemsetAsync(h->I0ref_o, 0, (size_t)h->nbp * 8, s));
      CUDA_TRY(h, cudaMemcpyAsync(h->I0ref_o, h->I0ref + h->band0, (size_t)h->nb * 8, cudaMemcpyDeviceToDevice, s));
    }
    CUDA_TRY(h, cudaMemsetAsync(h->I0wall_dev, 0, (size_t)std::max(h->nfaces, 1LL) * h->nbp * 4, s));
    CUDA_TRY(h, cudaStreamSynchronize(s));
  }
  // geometry + work list
  std::vector<DevGeom>& dg = h->dgeoms;
  dg.assign(h->geoms.size(), DevGeom{});
  for (size_t gi = 0; gi < h->geoms.size(); ++gi) {
    const bte_geom& g = h->geoms[gi];
    DevGeom& o = dg[gi];
    o.nx = g.nx; o.ny = g.ny; o.nz = g.nz; o.dim = g.dim;
    o.cell0 = h->cell0[gi];
    for (int s6 = 0; s6 < 6; ++s6) {
      o.face0[s6] = h->face0[gi * 6 + s6];
      o.bc[s6] = dev_bc(h->bc_type[gi][s6]);
      o.gdir[s6] = h->gdir[gi][s6];
    }
    o.cls = h->cls[gi];
    o.pad = 0;
  }
  CUDA_TRY(h, cudaMemcpyAsync(h->geoms_d, dg.data(), dg.size() * sizeof(DevGeom), cudaMemcpyHostToDevice, s));
  CUDA_TRY(h, cudaMemcpyAsync(h->items_d, h->items.data(), h->items.size() * sizeof(WorkItem), cudaMemcpyHostToDevice, s));
  CUDA_TRY(h, cudaMemsetAsync(h->counters, 0, sizeof(DevCounters), s));
  CUDA_TRY(h, cudaStreamSynchronize(s));
  {
    int dim = 2;
    for (auto& g : h->geoms) dim = std::max(dim, g.dim);
    build_gs(h, 1, dim == 3 ? 8 : 128, dim == 3 ? 8 : 1);
    const int rc = upload_gs(h, s);
    if (rc) return rc;
  }
  h->mem_ready = true;
  return BTE_OK;
}

int upload_geoms(bte_ctx* h) {
  std::vector<DevGeom>& dg = h->dgeoms;
  for (size_t gi = 0; gi < h->geoms.size(); ++gi)
    for (int s6 = 0; s6 < 6; ++s6) {
      dg[gi].bc[s6] = dev_bc(h->bc_type[gi][s6]);
      dg[gi].gdir[s6] = h->gdir[gi][s6];
    }
  drop_graphs(h);  // the launches of a step depend on the wall kinds
  CUDA_TRY(h, cudaMemcpyAsync(h->geoms_d, dg.data(), dg.size() * sizeof(DevGeom), cudaMemcpyHostToDevice, h->stream));
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  return BTE_OK;
}

int ensure_coef(bte_ctx* h, double dt, int scheme) {
  if (h->coef_dt == dt && h->coef_scheme == scheme) return BTE_OK;
  drop_graphs(h);  // captured launches carry dt in their arguments
  const size_t plane = (size_t)h->nd * h->nbp;
  const size_t ncls = h->cls_key.size();
  if (h->opts.precision == BTE_FP64) {
    h->coef_host.assign(5 * plane * ncls, 0.0);
    for (size_t c = 0; c < ncls; ++c) {
      const double delta[3] = {std::get<1>(h->cls_key[c]), std::get<2>(h->cls_key[c]), std::get<3>(h->cls_key[c])};
      build_coef(std::get<0>(h->cls_key[c]), delta, h->nd, h->S.data(), h->w.data(), h->nb, h->nbp,
                 h->vg.data() + h->band0, h->beta.data() + h->band0, dt, scheme == BTE_EXPLICIT,
                 h->coef_host.data() + c * 5 * plane);
    }
    CUDA_TRY(h, cudaMemcpyAsync(h->coef, h->coef_host.data(), h->coef_host.size() * 8, cudaMemcpyHostToDevice, h->stream));
    // the factored double-float tables (implicit update only)
    h->R_host.assign(4 * plane * ncls, 0.0f);
    h->dirc_host.assign(6 * (size_t)h->nd * ncls, 0.0f);
    h->band_host.assign(2 * (size_t)h->nbp, 0.0f);
    if (scheme != BTE_EXPLICIT)
      for (size_t c = 0; c < ncls; ++c) {
        const double delta[3] = {std::get<1>(h->cls_key[c]), std::get<2>(h->cls_key[c]), std::get<3>(h->cls_key[c])};
        build_ff_factored(std::get<0>(h->cls_key[c]), delta, h->nd, h->dir_group, h->S.data(), h->w.data(), h->nb, h->nbp,
                          h->vg.data() + h->band0, h->beta.data() + h->band0, dt, h->R_host.data() + c * 4 * plane,
                          h->dirc_host.data() + c * 6 * (size_t)h->nd, h->band_host.data());
      }
    CUDA_TRY(h, cudaMemcpyAsync(h->coef_R, h->R_host.data(), h->R_host.size() * 4, cudaMemcpyHostToDevice, h->stream));
    CUDA_TRY(h, cudaMemcpyAsync(h->dirc_ff, h->dirc_host.data(), h->dirc_host.size() * 4, cudaMemcpyHostToDevice, h->stream));
    CUDA_TRY(h, cudaMemcpyAsync(h->band_ff, h->band_host.data(), h->band_host.size() * 4, cudaMemcpyHostToDevice, h->stream));
  } else {
    std::vector<float> pq(2 * plane * ncls), dc(4 * (size_t)h->nd * ncls);
    for (size_t c = 0; c < ncls; ++c) {
      const double delta[3] = {std::get<1>(h->cls_key[c]), std::get<2>(h->cls_key[c]), std::get<3>(h->cls_key[c])};
      build_pq(std::get<0>(h->cls_key[c]), delta, h->nd, h->S.data(), h->w.data(), h->nb, h->nbp,
               h->vg.data() + h->band0, h->beta.data() + h->band0, dt, scheme == BTE_EXPLICIT,
               pq.data() + c * 2 * plane, pq.data() + c * 2 * plane + plane, dc.data() + c * 4 * h->nd);
    }
    CUDA_TRY(h, cudaMemcpyAsync(h->coef, pq.data(), pq.size() * 4, cudaMemcpyHostToDevice, h->stream));
    CUDA_TRY(h, cudaMemcpyAsync(h->dirc, dc.data(), dc.size() * 4, cudaMemcpyHostToDevice, h->stream));
    CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  }
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  h->coef_dt = dt;
  h->coef_scheme = scheme;
  return BTE_OK;
}

int check_geom(bte_ctx* h, int geom) {
  if (!h) return BTE_E_ARG;
  if (geom < 0 || geom >= (int)h->geoms.size()) return fail(h, BTE_E_ARG, "geometry index %d out of range", geom);
  return BTE_OK;
}

bool ready_to_step(bte_ctx* h, std::string& why) {
  for (size_t gi = 0; gi < h->geoms.size(); ++gi) {
    for (int s6 = 0; s6 < 2 * h->geoms[gi].dim; ++s6)
      if (!h->bc_set[gi][s6]) { why = "bte_set_bc missing for geometry " + std::to_string(gi) + " side " + std::to_string(s6); return false; }
    if (!h->init_set[gi]) { why = "bte_set_initial missing for geometry " + std::to_string(gi); return false; }
  }
  return true;
}

int copy_out(bte_ctx* h, double* out, const double* src, size_t n, int on_device) {
  CUDA_TRY(h, cudaMemcpyAsync(out, src, n * 8, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, h->stream));
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  return BTE_OK;
}

}  // namespace

namespace {

MLPView mlp_view(const bte_ctx* h) {
  MLPView m;
  m.A = h->mlp_p;
  m.B = h->mlp_p + mlp_param_count(1);
  m.nb = h->nb_all;
  m.T_lo = h->mlp_Tlo;
  m.T_hi = h->mlp_Thi;
  m.E_lo = h->mlp_Elo;
  m.E_hi = h->mlp_Ehi;
  m.r_lo = h->mlp_rlo;
  m.r_hi = h->mlp_rhi;
  m.I0ref = h->I0ref;
  return m;
}

SweepArgs sweep_args(bte_ctx* h) {
  SweepArgs a{};
  a.I0cell = h->I0cell;
  a.Tp = h->Tp;
  a.Teval = h->Teval;
  a.J = h->J;
  a.Msum = h->Msum;
  a.MsumL = h->MsumL;
  a.TL = h->TL;
  a.Tguess = h->solve_tp ? h->Tp : h->TL;  // or the previous T_L when T_p is not solved
  a.EL = h->EL;
  a.I0wall = h->I0wall;
  a.I0wall_dev = h->I0wall_dev;
  a.I0wall_ff = h->I0wall_ff;
  a.I0ref = h->I0ref_o;
  a.Epart = h->exchange_buf ? h->exchange_buf : h->Epart;
  a.partial = h->Epart ? 1 : 0;
  a.coef = h->coef;
  a.coef_R = h->coef_R;
  a.dirc_ff = h->dirc_ff;
  a.band_ff = h->band_ff;
  a.dirs = h->dirs_d;
  a.wdir = h->wdir;
  a.wdir32 = h->wdir32;
  a.Wtot = h->Wtot;
  a.geoms = h->geoms_d;
  a.items = h->items_d;
  a.nitems = (int)h->items.size();
  a.nd = h->nd;
  a.lpc = h->lpc;
  a.dteam = h->dteam;
  a.dir_group = h->dir_group;
  a.ne = h->lpc * (h->opts.precision == BTE_BF16 ? 1 : h->dteam);
  a.solve_tp = h->solve_tp ? 1 : 0;
  a.trust_rel = model_trust(h->opts.newton_rtol);
  a.maxit = h->opts.newton_maxit;
  a.counters = h->counters;
  a.explicit_scheme = h->coef_scheme == BTE_EXPLICIT ? 1 : 0;
  a.beta_exp = h->opts.beta_T_exp;
  a.beta_Tref = h->opts.T_ref;
  a.dt32 = (float)h->coef_dt;
  a.rdt32 = (float)(1.0 / h->coef_dt);
  a.dirc = h->dirc;
  a.vb32 = h->vb32;
  a.bb32 = h->bb32;
  a.fix = h->fix;
  a.Ec = h->Ec;
  a.gs_units = h->gs_units_d;
  a.gs_dirs = h->gs_dirs_d;
  a.gs_nunits = (int)h->gs_units.size();
  a.gs_ndc = h->gs_ndc;
  a.gs_tx = h->gs_tx;
  a.gs_ty = h->gs_ty;
  a.bscale = h->bscale;
  a.th = thermo(h);
  return a;
}

int ensure_TL(bte_ctx* h) {
  if (h->TL_valid) return BTE_OK;
  CUDA_TRY(h, launch_cells(sweep_args(h), h->ncells, 3, nullptr, 0, h->stream));
  h->TL_valid = true;
  return BTE_OK;
}

// Diffuse wall ghosts from intensity buffer I (before a sweep that reads I as
// its upwind field, and before wall fluxes).  *launches counts the kernels.
cudaError_t refresh_diffuse(bte_ctx* h, const void* I, cudaStream_t s, int* launches = nullptr) {
  for (size_t gi = 0; gi < h->geoms.size(); ++gi)
    for (int side = 0; side < 2 * h->geoms[gi].dim; ++side) {
      if (h->bc_type[gi][side] != BTE_BC_DIFFUSE) continue;
      const cudaError_t e = launch_diffuse_ghosts(
          h->opts.precision, I, h->I0ref_o, h->I0wall, h->opts.precision == BTE_FP64 ? nullptr : h->I0wall_dev,
          h->geoms_d, (int)gi, side, h->Sdev, h->wall_dirs[side], h->nd, h->nbp, (int)side_faces(h->geoms[gi], side), s);
      if (e != cudaSuccess) return e;
      if (launches) ++*launches;
    }
  return cudaSuccess;
}

// Per-direction ghost rows of the partially specular sides from intensity
// buffer I (before a sweep that reads I as its upwind field, and before wall
// fluxes).  *launches counts the kernels.
cudaError_t refresh_partial(bte_ctx* h, const void* I, cudaStream_t s, int* launches = nullptr) {
  for (size_t gi = 0; gi < h->geoms.size(); ++gi)
    for (int side = 0; side < 2 * h->geoms[gi].dim; ++side) {
      if (h->bc_type[gi][side] != BTE_BC_PARTIAL) continue;
      const cudaError_t e = launch_partial_ghosts(h->opts.precision, I, h->I0ref_o, h->geoms_d, (int)gi, side, h->Sdev,
                                                  h->wall_dirs[side], h->dirs_d, h->nd, h->nbp,
                                                  (int)side_faces(h->geoms[gi], side), h->spec[gi][side],
                                                  h->gdir[gi][side], s);
      if (e != cudaSuccess) return e;
      if (launches) ++*launches;
    }
  return cudaSuccess;
}

// Whether the FP64 Jacobi sweep of this handle runs in double-float arithmetic:
// FP64 storage without fp64_strict, fixed relaxation rates, and walls whose
// ghosts the sweep reads directly (isothermal faces and mirrors; diffuse and
// partially specular ghosts are refreshed between inner iterations by kernels
// that read the iterate as doubles).
bool ff_sweep(const bte_ctx* h) {
  if (h->opts.precision != BTE_FP64 || h->opts.fp64_strict || h->opts.beta_T_exp != 0.0) return false;
  for (size_t gi = 0; gi < h->geoms.size(); ++gi)
    for (int side = 0; side < 2 * h->geoms[gi].dim; ++side)
      if (h->bc_type[gi][side] == BTE_BC_DIFFUSE || h->bc_type[gi][side] == BTE_BC_PARTIAL) return false;
  return true;
}

// The current intensity buffer in the form the next step or call takes (in place):
// doubles, or ff pairs for the double-float sweep.
cudaError_t refill(bte_ctx* h, bool ff) {
  cudaError_t e = cudaSuccess;
  for (size_t gi = 0; gi < h->geoms.size() && e == cudaSuccess; ++gi) {
    if (!h->init_set[gi]) continue;
    const bte_geom& g = h->geoms[gi];
    e = launch_refill(ff, h->Ibuf[h->cur] + (size_t)h->cell0[gi] * h->nd * h->nbp * 8, h->I0cell + h->cell0[gi] * h->nbp,
                      (long long)g.nx * g.ny * g.nz, h->nd, h->nbp, h->stream);
  }
  return e;
}
cudaError_t ensure_state_doubles(bte_ctx* h) {
  if (!h->state_ff) return cudaSuccess;
  const cudaError_t e = h->initial ? refill(h, false)
                                   : launch_ff_to_doubles(h->Ibuf[h->cur], (long long)h->ncells * h->nd * h->nbp / 2, h->stream);
  if (e == cudaSuccess) h->state_ff = false;
  return e;
}
cudaError_t ensure_state_ff(bte_ctx* h) {
  if (h->state_ff) return cudaSuccess;
  const cudaError_t e = h->initial ? refill(h, true)
                                   : launch_doubles_to_ff(h->Ibuf[h->cur], h->Ibuf[h->cur],
                                                          (long long)h->ncells * h->nd * h->nbp / 2, h->stream);
  if (e == cudaSuccess) h->state_ff = true;
  return e;
}
// Reading calls return an initial state in full precision.
cudaError_t ensure_initial_doubles(bte_ctx* h) { return h->initial ? ensure_state_doubles(h) : cudaSuccess; }

// The ghosts of the diffuse and partially specular sides from the current state,
// before wall fluxes read them.  Their kernels read doubles, so a state that stands
// as ff pairs (set, or stepped under other wall kinds) is converted first; callers take
// the state's form afterwards.
cudaError_t refresh_ghosts(bte_ctx* h) {
  cudaError_t e = cudaSuccess;
  if (h->state_ff && !ff_sweep(h)) e = ensure_state_doubles(h);
  else e = ensure_initial_doubles(h);
  if (e == cudaSuccess) e = refresh_diffuse(h, h->Ibuf[h->cur], h->stream);
  if (e == cudaSuccess) e = refresh_partial(h, h->Ibuf[h->cur], h->stream);
  return e;
}

// A timing event on stream s: inside a stream capture it must become an event
// record node of the graph (cudaEventRecordExternal), so that every replay
// records it and the host can read it.
cudaError_t record_timing_event(cudaEvent_t ev, cudaStream_t s) {
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  cudaError_t e = cudaStreamIsCapturing(s, &st);
  if (e != cudaSuccess) return e;
  return cudaEventRecordWithFlags(ev, s, st == cudaStreamCaptureStatusActive ? cudaEventRecordExternal : cudaEventRecordDefault);
}

// One time step: ninner sweeps rotating the three intensity buffers from *cur.
// scheme BTE_IMPLICIT_GS runs the sweep-ordered pass and the per-cell step as
// two kernels and cells_kernel, the Jacobi sweep as one and cells_kernel.
cudaError_t enqueue_step(bte_ctx* h, SweepArgs a, int ninner, int scheme, cudaStream_t s, int* cur) {
  int dim = 2;
  for (auto& g : h->geoms) dim = std::max(dim, g.dim);
  const int n = *cur;
  int k = n;
  // double-float Jacobi sweeps read I^n in every inner iteration; FP64 implicit
  // steps in IEEE arithmetic keep B = A_n I^n, the same in every inner iteration,
  // in the third buffer: iteration 0 reads I^n and writes I^1 and B; iteration k
  // reads B and I^k and overwrites the buffer I^n (or I^{k-2}) was in.
  const bool use_ff = h->state_ff;  // bte_step has put the state in the form of this scheme
  const bool use_b = h->opts.precision == BTE_FP64 && !use_ff && !a.explicit_scheme && ninner >= 2;
  a.ff = use_ff ? 1 : 0;
  if (scheme == BTE_IMPLICIT_GS) a.ne = kRedEntries;
  // threads behind which cells_kernel may start: those of the row sweep (gs_reduce_kernel
  // and the BF16 sweep let nothing start before their end)
  const long long before =
      scheme == BTE_IMPLICIT_GS || h->opts.precision == BTE_BF16 ? 0 : (long long)a.nitems * h->threads;
  int z = -1;
  for (int it = 0; it < ninner; ++it) {
    int o = 0;
    a.bmode = 0;
    a.Bout = nullptr;
    if (use_b && it == 0) {
      while (o == n) ++o;
      z = 0;
      while (z == n || z == o) ++z;
      a.In = h->Ibuf[n];
      a.Bout = h->Ibuf[z];
      a.bmode = 1;
    } else if (use_b) {
      while (o == z || o == k) ++o;
      a.In = h->Ibuf[z];
      a.bmode = 2;
    } else {
      while (o == n || o == k) ++o;
      a.In = h->Ibuf[n];
    }
    a.Ik = h->Ibuf[k];
    a.Iout = h->Ibuf[o];
    cudaError_t e = refresh_diffuse(h, a.Ik, s);
    if (e == cudaSuccess) e = refresh_partial(h, a.Ik, s);
    const bool timed = h->time_sweeps && 2 * it + 1 < (int)h->tev.size();
    if (e == cudaSuccess && timed) e = record_timing_event(h->tev[2 * it], s);
    if (scheme == BTE_IMPLICIT_GS) {
      if (e == cudaSuccess && a.beta_exp != 0.0)
        e = launch_beta_scale(h->bscale, h->Tp, a.beta_Tref, a.beta_exp, h->ncells, s);
      if (e == cudaSuccess) e = launch_gs_sweep(h->opts.precision, a, dim, h->gs_threads, s);
      if (e == cudaSuccess) e = launch_gs_reduce(h->opts.precision, a, h->ncells, s);
    } else if (e == cudaSuccess) {
      e = launch_sweep(h->opts.precision, h->pd, a, dim, h->threads, h->grid, s);
    }
    if (e == cudaSuccess && timed) e = record_timing_event(h->tev[2 * it + 1], s);
    if (e == cudaSuccess && a.partial) {
      // band-range handle: the caller sums the per-cell (E_L, E_p) partials over
      // the ranks that hold the other bands, then every rank solves every cell
      e = launch_cells(a, h->ncells, 1, nullptr, before, s);
      if (e != cudaSuccess) return e;
      const int xr = h->exchange(a.Epart, 2 * h->ncells, (void*)s, h->exchange_user);
      if (xr != 0) {
        h->exchange_rc = xr;
        return cudaErrorUnknown;
      }
    }
    if (e == cudaSuccess) {
      const MLPView m = mlp_view(h);
      e = launch_cells(a, h->ncells, a.partial ? 2 : 0, h->opts.learned ? &m : nullptr, a.partial ? 256 * h->ncells : before, s);
    }
    if (e != cudaSuccess) return e;
    k = o;
  }
  *cur = k;
  return cudaSuccess;
}

}  // namespace

namespace bte {

cudaError_t raise_dynamic_smem(const void* func, size_t bytes) {
  if (bytes <= 48 * 1024) return cudaSuccess;
  static std::mutex mu;
  static std::map<std::pair<int, const void*>, size_t> granted;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  size_t& g = granted[{dev, func}];
  if (bytes <= g) return cudaSuccess;
  e = cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) g = bytes;
  return e;
}


int flux_view(bte_ctx* h, int geom, FluxView* out) {
  int rc = check_geom(h, geom);
  if (rc) return rc;
  if (!h->mem_ready || !h->init_set[geom]) return fail(h, BTE_E_STATE, "geometry %d has no state", geom);
  const bte_geom& g = h->geoms[geom];
  {  // kernel launches, no allocation
    const cudaError_t e = refresh_ghosts(h);
    if (e != cudaSuccess) return fail(h, BTE_E_CUDA, "diffuse wall ghosts: %s", cudaGetErrorString(e));
  }
  out->precision = h->opts.precision;
  out->I = h->Ibuf[h->cur];
  out->state_ff = h->state_ff;
  out->I0wall = h->I0wall;
  out->geoms = h->geoms_d;
  std::copy(h->wall_dirs.begin(), h->wall_dirs.end(), out->wall_dirs);
  out->S = h->Sdev;
  out->nd = h->nd;
  out->nbp = h->nbp;
  out->dim = g.dim;
  for (int s6 = 0; s6 < 6; ++s6) out->nfaces[s6] = s6 < 2 * g.dim ? (int)side_faces(g, s6) : 0;
  out->stream = h->stream;
  out->dev = h->dev;
  return BTE_OK;
}

int handle_device(bte_ctx* h) { return h->dev; }

int set_handle_error(bte_ctx* h, int code, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  if (h) h->err = buf;
  return code;
}

}  // namespace bte

extern "C" {

int bte_default_opts(bte_opts* o) {
  if (!o) return BTE_E_ARG;
  std::memset(o, 0, sizeof *o);
  o->dir_kind = BTE_DIRS_POLAR_AZIM;
  o->n_inplane = 16;
  o->n_polar = 20;
  o->n_azim = 20;
  o->precision = BTE_FP64;
  o->learned = 0;
  o->n_gauss = 16;
  o->newton_rtol = 1e-14;
  o->newton_maxit = 50;
  o->cuda_stream = nullptr;
  o->T_ref = 300.0;
  o->use_graph = 0;
  o->autotune = 0;
  o->beta_T_exp = 0.0;
  o->fp64_strict = 0;
  return BTE_OK;
}

int bte_init_mesh(bte_handle* out, int n_geom, const bte_geom* geoms, const bte_opts* opts) {
  if (!out) return fail(nullptr, BTE_E_ARG, "out is NULL");
  *out = nullptr;
  if (n_geom < 1 || !geoms) return fail(nullptr, BTE_E_ARG, "need n_geom >= 1 and a geometry array");
  bte_opts o;
  if (opts) o = *opts; else bte_default_opts(&o);
  if (o.precision != BTE_FP64 && o.precision != BTE_FP32 && o.precision != BTE_BF16)
    return fail(nullptr, BTE_E_ARG, "unknown precision %d", o.precision);
  if (!(o.T_ref >= kTmin && o.T_ref <= kTmax)) return fail(nullptr, BTE_E_ARG, "T_ref must lie in [1, 5000] K");
  if (!(std::fabs(o.beta_T_exp) <= 16.0)) return fail(nullptr, BTE_E_ARG, "beta_T_exp must lie in [-16, 16]");
  if (o.learned != 0 && o.learned != 1) return fail(nullptr, BTE_E_ARG, "learned must be 0 or 1");
  if (o.n_gauss < 1 || o.n_gauss > kMaxGauss) return fail(nullptr, BTE_E_ARG, "n_gauss must be in 1..%d", kMaxGauss);
  if (!(o.newton_rtol > 0 && o.newton_rtol < 1e-3) || o.newton_maxit < 1)
    return fail(nullptr, BTE_E_ARG, "newton_rtol must be in (0, 1e-3) and newton_maxit >= 1");
  long long total = 0;
  for (int i = 0; i < n_geom; ++i) {
    const bte_geom& g = geoms[i];
    if (!(g.dim == 2 || g.dim == 3) || g.nx < 1 || g.ny < 1 || g.nz < 1 || (g.dim == 2 && g.nz != 1))
      return fail(nullptr, BTE_E_ARG, "geometry %d: bad dim/size", i);
    if (g.dim != geoms[0].dim)  // one sweep launch serves every geometry of a handle
      return fail(nullptr, BTE_E_ARG, "geometry %d: every geometry of a handle must have the same dim", i);
    if (!(g.dx > 0 && g.dy > 0 && (g.dim == 2 || g.dz > 0))) return fail(nullptr, BTE_E_ARG, "geometry %d: cell sizes must be > 0", i);
    const long long nc = (long long)g.nx * g.ny * g.nz;
    if (nc > (1LL << 30)) return fail(nullptr, BTE_E_ARG, "geometry %d: too many cells", i);
    total += nc;
  }
  bte_ctx* h = new bte_ctx();
  h->opts = o;
  h->ng = o.n_gauss;
  h->stream = (cudaStream_t)o.cuda_stream;
  cudaGetDevice(&h->dev);
  int rc;
  if (o.dir_kind == BTE_DIRS_INPLANE) rc = build_dirs_inplane(o.n_inplane, h->S, h->w, h->refl);
  else if (o.dir_kind == BTE_DIRS_POLAR_AZIM) rc = build_dirs_polar_azim(o.n_polar, o.n_azim, h->S, h->w, h->refl);
  else rc = -1;
  if (rc != 0) {
    delete h;
    return fail(nullptr, BTE_E_ARG, "bad direction set (in-plane needs n %% 4 == 0; polar x azimuthal needs even n_polar and n_azim %% 4 == 0)");
  }
  h->dir_group = o.dir_kind == BTE_DIRS_INPLANE ? 4 : 8;
  h->perm = internal_order(h->S, h->w, h->refl, h->dir_group);
  h->nd = (int)h->w.size();
  if (h->nd > 2048) {  // the sweep keeps the direction table in shared memory
    delete h;
    return fail(nullptr, BTE_E_ARG, "at most 2048 directions");
  }
  for (double x : h->w) h->Wtot += x;
  h->geoms.assign(geoms, geoms + n_geom);
  h->ncells = total;
  long long c0 = 0, f0 = 0;
  std::map<std::tuple<int, double, double, double>, int> keys;
  for (int i = 0; i < n_geom; ++i) {
    bte_geom g = geoms[i];
    if (g.dim == 2) g.dz = g.dz > 0 ? g.dz : 1.0;
    h->geoms[i] = g;
    h->cell0.push_back(c0);
    const long long nc = (long long)g.nx * g.ny * g.nz;
    h->max_geom_cells = std::max<long long>(h->max_geom_cells, nc);
    c0 += nc;
    for (int s6 = 0; s6 < 6; ++s6) {
      h->face0.push_back(f0);
      if (s6 < 2 * g.dim) {
        f0 += side_faces(g, s6);
        h->max_side_faces = std::max<long long>(h->max_side_faces, side_faces(g, s6));
      }
    }
    auto key = std::make_tuple(g.dim, g.dx, g.dy, g.dim == 3 ? g.dz : 0.0);
    auto it = keys.find(key);
    if (it == keys.end()) {
      const int id = (int)h->cls_key.size();
      keys[key] = id;
      h->cls_key.push_back(key);
      h->cls.push_back(id);
    } else {
      h->cls.push_back(it->second);
    }
  }
  h->nfaces = f0;
  h->bc_type.assign(n_geom, {BTE_BC_SPECULAR, BTE_BC_SPECULAR, BTE_BC_SPECULAR, BTE_BC_SPECULAR, BTE_BC_SPECULAR, BTE_BC_SPECULAR});
  h->bc_set.assign(n_geom, {false, false, false, false, false, false});
  h->spec.assign(n_geom, {0, 0, 0, 0, 0, 0});
  h->gdir.assign(n_geom, {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr});
  h->init_set.assign(n_geom, false);
  if (cudaEventCreate(&h->ev0) != cudaSuccess || cudaEventCreate(&h->ev1) != cudaSuccess) {
    delete h;
    return fail(nullptr, BTE_E_CUDA, "cudaEventCreate failed");
  }
  *out = h;
  return BTE_OK;
}

int bte_set_bands(bte_handle h, int nb, const double* wlo, const double* whi, const double* vg, const double* beta,
                  const double* deg) {
  if (!h) return BTE_E_ARG;
  if (h->bands_set) return fail(h, BTE_E_STATE, "bands are already set");
  if (nb < 1 || nb > kMaxBands || !wlo || !whi || !vg || !beta || !deg)
    return fail(h, BTE_E_ARG, "need 1 <= nb <= %d and five band arrays", kMaxBands);
  for (int b = 0; b < nb; ++b) {
    if (!(std::isfinite(wlo[b]) && std::isfinite(whi[b]) && wlo[b] >= 0 && whi[b] > wlo[b]))
      return fail(h, BTE_E_ARG, "band %d: need 0 <= omega_lo < omega_hi", b);
    if (!(std::isfinite(vg[b]) && vg[b] > 0)) return fail(h, BTE_E_ARG, "band %d: vg must be > 0", b);
    if (!(std::isfinite(beta[b]) && beta[b] >= 0)) return fail(h, BTE_E_ARG, "band %d: beta must be >= 0", b);
    if (!(std::isfinite(deg[b]) && deg[b] > 0)) return fail(h, BTE_E_ARG, "band %d: degeneracy must be > 0", b);
  }
  h->nb = h->nb_all = nb;
  h->nbp = h->nbp_all = (nb + 7) / 8 * 8;
  h->band0 = 0;
  h->wlo.assign(wlo, wlo + nb);
  h->whi.assign(whi, whi + nb);
  h->vg.assign(vg, vg + nb);
  h->beta.assign(beta, beta + nb);
  h->deg.assign(deg, deg + nb);
  h->solve_tp = false;
  for (int b = 0; b < nb; ++b) h->solve_tp |= beta[b] > 0;
  build_items(h);
  h->bands_set = true;
  return BTE_OK;
}

int bte_set_band_range(bte_handle h, int band_lo, int band_hi) {
  if (!h) return BTE_E_ARG;
  if (!h->bands_set) return fail(h, BTE_E_STATE, "bte_set_bands must come before bte_set_band_range");
  if (h->mem_ready || h->ws) return fail(h, BTE_E_STATE, "bte_set_band_range must come before device memory is in use");
  if (!(0 <= band_lo && band_lo < band_hi && band_hi <= h->nb_all))
    return fail(h, BTE_E_ARG, "need 0 <= band_lo < band_hi <= %d", h->nb_all);
  h->band0 = band_lo;
  h->nb = band_hi - band_lo;
  h->nbp = (h->nb + 7) / 8 * 8;
  build_items(h);
  return BTE_OK;
}

int bte_set_exchange(bte_handle h, bte_allreduce_fn fn, void* user, double* dev_buf) {
  if (!h) return BTE_E_ARG;
  if (!fn) return fail(h, BTE_E_ARG, "fn is NULL");
  if (((uintptr_t)dev_buf) & 7) return fail(h, BTE_E_ARG, "dev_buf must be 8-byte aligned");
  h->exchange = fn;
  h->exchange_user = user;
  h->exchange_buf = dev_buf;
  return BTE_OK;
}

size_t bte_workspace_bytes(bte_handle h) {
  if (!h || !h->bands_set) return 0;
  bte_ctx tmp = *h;  // carve() writes pointers; keep h untouched
  return carve(&tmp, nullptr);
}

int bte_bind_workspace(bte_handle h, void* dev_ptr, size_t bytes) {
  if (!h) return BTE_E_ARG;
  if (!h->bands_set) return fail(h, BTE_E_STATE, "bte_set_bands must come before bte_bind_workspace");
  if (h->mem_ready || h->ws) return fail(h, BTE_E_STATE, "device memory is already in use");
  if (!dev_ptr) return fail(h, BTE_E_ARG, "dev_ptr is NULL");
  if (((uintptr_t)dev_ptr) & 255) return fail(h, BTE_E_ARG, "workspace must be 256-byte aligned");
  const size_t need = bte_workspace_bytes(h);
  if (bytes < need) return fail(h, BTE_E_NOMEM, "workspace of %zu bytes is smaller than the %zu needed", bytes, need);
  h->ws = (char*)dev_ptr;
  h->ws_bytes = bytes;
  h->ws_owned = false;
  return BTE_OK;
}

int bte_set_bc(bte_handle h, int geom, int side, int type, const double* T_faces, double T_uniform) {
  int rc = check_geom(h, geom);
  if (rc) return rc;
  if (!h->bands_set) return fail(h, BTE_E_STATE, "bte_set_bands must come before bte_set_bc");
  const bte_geom& g = h->geoms[geom];
  if (side < 0 || side >= 2 * g.dim) return fail(h, BTE_E_ARG, "side %d out of range for a %dD geometry", side, g.dim);
  if (type != BTE_BC_ISOTHERMAL && type != BTE_BC_SPECULAR && type != BTE_BC_DIFFUSE)
    return fail(h, BTE_E_ARG, "unknown wall type %d", type);
  const long long nf = side_faces(g, side);
  std::vector<double> T;
  if (type == BTE_BC_ISOTHERMAL) {
    T.assign(nf, T_uniform);
    if (T_faces) T.assign(T_faces, T_faces + nf);
    for (double t : T)
      if (!(t >= kTmin && t <= kTmax)) return fail(h, BTE_E_ARG, "wall temperature %g outside [1, 5000] K", t);
  }
  if ((rc = ensure_memory(h))) return rc;
  if (type == BTE_BC_ISOTHERMAL) {
    CUDA_TRY(h, cudaMemcpyAsync(h->scratch_T, T.data(), nf * 8, cudaMemcpyHostToDevice, h->stream));
    CUDA_TRY(h, launch_wall_I0(h->I0wall + h->face0[geom * 6 + side] * h->nbp, h->scratch_T, nf, thermo(h), h->stream));
    if (h->opts.precision == BTE_FP64)
      CUDA_TRY(h, launch_doubles_to_ff(h->I0wall + h->face0[geom * 6 + side] * h->nbp,
                                       (char*)h->I0wall_ff + h->face0[geom * 6 + side] * h->nbp * 8, nf * h->nbp / 2,
                                       h->stream));
    else
      CUDA_TRY(h, launch_wall_dev(h->I0wall_dev + h->face0[geom * 6 + side] * h->nbp,
                                  h->I0wall + h->face0[geom * 6 + side] * h->nbp, h->I0ref_o, nf, h->nbp,
                                  h->stream));
  }
  const bool changed = h->bc_type[geom][side] != type;
  h->bc_type[geom][side] = type;
  h->bc_set[geom][side] = true;
  if (changed && (rc = upload_geoms(h))) return rc;
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  return BTE_OK;
}

int bte_set_specularity(bte_handle h, int geom, int side, double p) {
  int rc = check_geom(h, geom);
  if (rc) return rc;
  if (!h->bands_set) return fail(h, BTE_E_STATE, "bte_set_bands must come before bte_set_specularity");
  const bte_geom& g = h->geoms[geom];
  if (side < 0 || side >= 2 * g.dim) return fail(h, BTE_E_ARG, "side %d out of range for a %dD geometry", side, g.dim);
  if (!(p >= 0.0 && p <= 1.0)) return fail(h, BTE_E_ARG, "specularity must lie in [0, 1]");
  if ((rc = ensure_memory(h))) return rc;
  if (!h->gdir[geom][side]) {
    const size_t bytes = (size_t)side_faces(g, side) * h->nd * h->nbp * elem_bytes(h->opts.precision);
    void* q = nullptr;
    const cudaError_t e = cudaMalloc(&q, bytes);
    if (e != cudaSuccess) return fail(h, BTE_E_NOMEM, "cudaMalloc(%zu bytes): %s", bytes, cudaGetErrorString(e));
    h->gdir[geom][side] = q;
  }
  h->spec[geom][side] = p;
  h->bc_type[geom][side] = BTE_BC_PARTIAL;
  h->bc_set[geom][side] = true;
  return upload_geoms(h);
}

int bte_set_initial(bte_handle h, int geom, const double* T_cells, double T_uniform) {
  int rc = check_geom(h, geom);
  if (rc) return rc;
  if (!h->bands_set) return fail(h, BTE_E_STATE, "bte_set_bands must come before bte_set_initial");
  const bte_geom& g = h->geoms[geom];
  const long long nc = (long long)g.nx * g.ny * g.nz;
  std::vector<double> T(nc, T_uniform);
  if (T_cells) T.assign(T_cells, T_cells + nc);
  for (double t : T)
    if (!(t >= kTmin && t <= kTmax)) return fail(h, BTE_E_ARG, "initial temperature %g outside [1, 5000] K", t);
  if ((rc = ensure_memory(h))) return rc;
  // the first geometry set, or a lone one set again, starts in the form of the handle's
  // default sweep (as far as its walls are known); beside geometries that have been
  // stepped or restored an initial state is written in doubles
  bool others = false;
  for (size_t gi = 0; gi < h->geoms.size(); ++gi) others |= (int)gi != geom && h->init_set[gi];
  if (!others) {
    h->initial = true;
    h->state_ff = ff_sweep(h);
  }
  if (!h->initial) CUDA_TRY(h, ensure_state_doubles(h));
  CUDA_TRY(h, cudaMemcpyAsync(h->scratch_T, T.data(), nc * 8, cudaMemcpyHostToDevice, h->stream));
  CUDA_TRY(h, launch_init_cells(h->opts.precision, h->state_ff, h->Ibuf[h->cur], h->I0cell, h->J, h->Msum, h->MsumL, h->Tp, h->Teval, h->TL, h->EL,
                                h->scratch_T, h->I0ref_o, h->cell0[geom], (int)nc, h->nd, thermo(h), h->stream));
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  h->init_set[geom] = true;
  h->bscale_valid = false;
  h->TL_valid = false;  // T_L is recomputed from E_L on request
  return BTE_OK;
}

int bte_step(bte_handle h, double dt, int nsteps, int ninner, int scheme, bte_stats* stats) {
  if (!h) return BTE_E_ARG;
  std::string why;
  if (!h->mem_ready || !ready_to_step(h, why)) return fail(h, BTE_E_STATE, "not ready to step: %s", why.empty() ? "no state" : why.c_str());
  if (!(dt > 0 && std::isfinite(dt))) return fail(h, BTE_E_ARG, "dt must be > 0");
  if (nsteps < 0) return fail(h, BTE_E_ARG, "nsteps must be >= 0");
  if (scheme != BTE_IMPLICIT_JACOBI && scheme != BTE_EXPLICIT && scheme != BTE_IMPLICIT_GS)
    return fail(h, BTE_E_ARG, "unknown scheme %d", scheme);
  if (scheme == BTE_EXPLICIT) ninner = 1;
  if (ninner < 1) return fail(h, BTE_E_ARG, "ninner must be >= 1");
  const int cscheme = scheme == BTE_EXPLICIT ? BTE_EXPLICIT : BTE_IMPLICIT_JACOBI;  // coefficient set
  int rc = ensure_coef(h, dt, cscheme);
  if (rc) return rc;
  if (h->opts.learned && !h->mlp_trained) return fail(h, BTE_E_STATE, "learned mode needs bte_train_mlp first");
  if (h->opts.autotune && (scheme == BTE_IMPLICIT_GS ? h->gs_tune_report.empty() : h->tune_report.empty())) {
    if ((rc = bte_autotune(h, dt, scheme, nullptr, 0)) != BTE_OK) return rc;
  }
  cudaStream_t s = h->stream;
  if (stats) {
    CUDA_TRY(h, cudaMemsetAsync(h->counters, 0, sizeof(DevCounters), s));
    CUDA_TRY(h, cudaEventRecord(h->ev0, s));
  }
  SweepArgs a = sweep_args(h);
  int launches = 0;
  const bool ranged = h->Epart != nullptr;
  if (ranged && !h->exchange) return fail(h, BTE_E_STATE, "a band-range handle needs bte_set_exchange before stepping");
  h->exchange_rc = 0;
  const bool ff_step = h->opts.precision == BTE_FP64 && scheme == BTE_IMPLICIT_JACOBI && ff_sweep(h);
  if (nsteps > 0) {
    CUDA_TRY(h, ff_step ? ensure_state_ff(h) : ensure_state_doubles(h));
    h->initial = false;
  }
  if (h->opts.beta_T_exp != 0.0 && !h->bscale_valid && nsteps > 0) {  // later changes of T_p come from cells_kernel
    CUDA_TRY(h, launch_beta_scale(h->bscale, h->Tp, h->opts.T_ref, h->opts.beta_T_exp, h->ncells, s));
    h->bscale_valid = true;
  }
  if (h->time_sweeps && nsteps > 0) {
    if ((int)h->tev.size() < 2 * ninner) {  // events for every sweep of a step; graphs captured before lack them
      drop_graphs(h);
      while ((int)h->tev.size() < 2 * ninner) {
        cudaEvent_t ev = nullptr;
        CUDA_TRY(h, cudaEventCreate(&ev));
        h->tev.push_back(ev);
      }
    }
    h->tev_n = ninner;
  }
  for (int st = 0; st < nsteps; ++st) {
    if (h->opts.use_graph && !ranged) {  // the host-side exchange cannot sit inside a graph
      cudaGraphExec_t exec = nullptr;
      int cur_out = -1;
      for (auto& e : h->graphs)
        if (e.scheme == scheme && e.ninner == ninner && e.cur_in == h->cur && e.ff_in == h->state_ff) {
          exec = e.exec;
          cur_out = e.cur_out;
        }
      if (!exec) {
        if (!h->cap_stream) CUDA_TRY(h, cudaStreamCreateWithFlags(&h->cap_stream, cudaStreamNonBlocking));
        cudaGraph_t graph = nullptr;
        CUDA_TRY(h, cudaStreamBeginCapture(h->cap_stream, cudaStreamCaptureModeThreadLocal));
        int cur = h->cur;
        cudaError_t e = enqueue_step(h, a, ninner, scheme, h->cap_stream, &cur);
        cudaError_t e2 = cudaStreamEndCapture(h->cap_stream, &graph);
        if (e != cudaSuccess || e2 != cudaSuccess) {
          if (graph) cudaGraphDestroy(graph);
          return fail(h, BTE_E_CUDA, "graph capture: %s", cudaGetErrorString(e != cudaSuccess ? e : e2));
        }
        e = cudaGraphInstantiate(&exec, graph, 0);
        cudaGraphDestroy(graph);
        if (e != cudaSuccess) return fail(h, BTE_E_CUDA, "cudaGraphInstantiate: %s", cudaGetErrorString(e));
        h->graphs.push_back({scheme, ninner, h->cur, cur, h->state_ff, exec});
        cur_out = cur;
      }
      CUDA_TRY(h, cudaGraphLaunch(exec, s));
      h->cur = cur_out;
    } else {
      const cudaError_t e = enqueue_step(h, a, ninner, scheme, s, &h->cur);
      if (e != cudaSuccess && h->exchange_rc)
        return fail(h, BTE_E_EXCHANGE, "the exchange callback returned %d", h->exchange_rc);
      CUDA_TRY(h, e);
    }
    int ndiff = 0;  // ghost refresh launches: diffuse and partially specular sides
    for (auto& bt : h->bc_type)
      for (int t : bt) ndiff += t == BTE_BC_DIFFUSE || t == BTE_BC_PARTIAL;
    // sweep (sweep-ordered: pass + band sums, and the beta scale with tau(T)),
    // per-cell step (two launches around a band-range exchange), diffuse wall ghosts
    const int sweep_k = scheme == BTE_IMPLICIT_GS ? 2 + (h->opts.beta_T_exp != 0.0 ? 1 : 0) : 1;
    launches += ninner * (sweep_k + 1 + (ranged ? 1 : 0) + ndiff);
  }
  if (nsteps > 0) {
    h->TL_valid = false;
    h->EL_partial = false;
  }
  if (stats) {
    CUDA_TRY(h, cudaEventRecord(h->ev1, s));
    CUDA_TRY(h, cudaEventSynchronize(h->ev1));
    DevCounters c;
    CUDA_TRY(h, cudaMemcpy(&c, h->counters, sizeof c, cudaMemcpyDeviceToHost));
    float ms = 0.f;
    CUDA_TRY(h, cudaEventElapsedTime(&ms, h->ev0, h->ev1));
    stats->updates = (long long)h->ncells * h->nd * h->nb * (long long)ninner * nsteps;
    stats->solve_evals = (long long)c.evals;
    stats->solves = (long long)c.solves;
    stats->fallbacks = (long long)c.fallbacks;
    stats->nonfinite = (long long)c.nonfinite;
    stats->launches = launches;
    stats->gpu_ms = ms;
    if (c.nonfinite) return fail(h, BTE_E_NONFINITE, "%llu cells had a non-finite energy or no temperature in [1, 5000] K", (unsigned long long)c.nonfinite);
    if (c.fallbacks) return BTE_W_FALLBACK;
  }
  return BTE_OK;
}

namespace {

void copy_report(const std::string& r, char* report, size_t report_len) {
  if (report && report_len) {
    std::strncpy(report, r.c_str(), report_len - 1);
    report[report_len - 1] = 0;
  }
}

// Sweep-ordered pass: directions per CTA x column-tile size, timed on a spare buffer.
int autotune_gs(bte_ctx* h, char* report, size_t report_len) {
  cudaStream_t s = h->stream;
  int dim = 2;
  for (auto& g : h->geoms) dim = std::max(dim, g.dim);
  const int spare = (h->cur + 1) % 3;
  struct Cand { int ndc, tx, ty; float ms; };
  std::vector<Cand> tried;
  const int tiles2[3][2] = {{64, 1}, {128, 1}, {256, 1}};
  const int tiles3[3][2] = {{4, 4}, {8, 8}, {16, 16}};
  Cand best{h->gs_ndc, h->gs_tx, h->gs_ty, 1e30f};
  if (h->opts.beta_T_exp != 0.0)
    CUDA_TRY(h, launch_beta_scale(h->bscale, h->Tp, h->opts.T_ref, h->opts.beta_T_exp, h->ncells, s));
  for (int ndc = 1; ndc <= 2; ++ndc)
    for (int t = 0; t < 3; ++t) {
      const int tx = dim == 3 ? tiles3[t][0] : tiles2[t][0], ty = dim == 3 ? tiles3[t][1] : tiles2[t][1];
      build_gs(h, ndc, tx, ty);
      bool dup = false;
      for (auto& c : tried) dup |= c.ndc == h->gs_ndc && c.tx == tx && c.ty == ty;
      if (dup) continue;
      int rc = upload_gs(h, s);
      if (rc) return rc;
      SweepArgs a = sweep_args(h);
      a.bmode = 0;
      a.Bout = nullptr;
      a.In = a.Ik = h->Ibuf[h->cur];
      a.Iout = h->Ibuf[spare];
      CUDA_TRY(h, launch_gs_sweep(h->opts.precision, a, dim, h->gs_threads, s));
      CUDA_TRY(h, cudaEventRecord(h->ev0, s));
      for (int r = 0; r < 3; ++r) CUDA_TRY(h, launch_gs_sweep(h->opts.precision, a, dim, h->gs_threads, s));
      CUDA_TRY(h, cudaEventRecord(h->ev1, s));
      CUDA_TRY(h, cudaEventSynchronize(h->ev1));
      float ms = 0.f;
      CUDA_TRY(h, cudaEventElapsedTime(&ms, h->ev0, h->ev1));
      tried.push_back({h->gs_ndc, tx, ty, ms / 3.f});
      if (ms / 3.f < best.ms) best = tried.back();
    }
  build_gs(h, best.ndc, best.tx, best.ty);
  int rc = upload_gs(h, s);
  if (rc) return rc;
  drop_graphs(h);
  char buf[128];
  h->gs_tune_report = "directions_per_cta,tile_x,tile_y,threads,ms_per_pass\n";
  for (auto& c : tried) {
    const int lanes = h->nbp / values_per_lane(h->opts.precision);
    snprintf(buf, sizeof buf, "%d,%d,%d,%d,%.4f\n", c.ndc, c.tx, c.ty, lanes * c.ndc * std::max(1, 256 / (lanes * c.ndc)), c.ms);
    h->gs_tune_report += buf;
  }
  snprintf(buf, sizeof buf, "chosen,%d,%d,%d,%d\n", best.ndc, best.tx, best.ty, h->gs_threads);
  h->gs_tune_report += buf;
  copy_report(h->gs_tune_report, report, report_len);
  return BTE_OK;
}

}  // namespace

int bte_autotune(bte_handle h, double dt, int scheme, char* report, size_t report_len) {
  if (!h) return BTE_E_ARG;
  std::string why;
  if (!h->mem_ready || !ready_to_step(h, why)) return fail(h, BTE_E_STATE, "not ready to tune: %s", why.empty() ? "no state" : why.c_str());
  if (!(dt > 0 && std::isfinite(dt))) return fail(h, BTE_E_ARG, "dt must be > 0");
  if (scheme != BTE_IMPLICIT_JACOBI && scheme != BTE_EXPLICIT && scheme != BTE_IMPLICIT_GS)
    return fail(h, BTE_E_ARG, "unknown scheme %d", scheme);
  int rc = ensure_coef(h, dt, scheme == BTE_EXPLICIT ? BTE_EXPLICIT : BTE_IMPLICIT_JACOBI);
  if (rc) return rc;
  const bool ff = scheme == BTE_IMPLICIT_JACOBI && ff_sweep(h);
  if (!ff) CUDA_TRY(h, ensure_state_doubles(h));  // the form the timed sweeps read
  if (h->opts.beta_T_exp != 0.0 && !h->bscale_valid) {
    CUDA_TRY(h, launch_beta_scale(h->bscale, h->Tp, h->opts.T_ref, h->opts.beta_T_exp, h->ncells, h->stream));
    h->bscale_valid = true;
  }
  if (scheme == BTE_IMPLICIT_GS) return autotune_gs(h, report, report_len);
  cudaStream_t s = h->stream;
  int sms = 152;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->dev);
  const int spare = (h->cur + 1) % 3;  // timing launches write here; the state is untouched
  int src = h->cur;                    // and read it, or a copy as ff pairs of one held in doubles
  if (ff && !h->state_ff) {
    src = (h->cur + 2) % 3;
    CUDA_TRY(h, launch_doubles_to_ff(h->Ibuf[h->cur], h->Ibuf[src], (long long)h->ncells * h->nd * h->nbp / 2, s));
  }
  struct Cand { int cpb, dteam, grid, pd; float ms; };
  std::vector<Cand> tried;
  // directions per team step: the default and half of it (fewer lanes per
  // cell, longer items: the per-item epilogue is spread over more updates)
  build_items(h);
  const bool bf16 = h->opts.precision == BTE_BF16;
  std::vector<int> dteam_list = {h->dteam};
  if (h->dteam >= 2) dteam_list.push_back(h->dteam / 2);
  if (h->opts.precision == BTE_FP32 && max_teams(h) == 4 && 4 * h->lpc <= 256) dteam_list.push_back(4);
  const std::vector<int> pd_list = bf16 ? std::vector<int>{1, 2} : std::vector<int>{1};
  int best_cpb = h->cpb, best_dteam = h->dteam, best_grid = h->grid, best_pd = h->pd;
  float best_ms = 1e30f;
  int dim = 2;
  for (auto& g : h->geoms) dim = std::max(dim, g.dim);
  // candidates: cells per CTA about 128 or 256 threads, and every count up
  // to 256 threads whose CTA is whole warps (a partial warp still occupies
  // the FP64 pipe's issue slots of a full one); three grids; both register
  // variants
  for (int dteam : dteam_list) {
    const int team = h->lpc * dteam;
    std::vector<int> cpb_list = {std::max(1, 128 / team), std::max(1, 256 / team)};
    const int whole = 32 / std::gcd(team, 32);
    for (int c = whole; c * team <= 256; c += whole) cpb_list.push_back(c);
    for (int cpb : cpb_list) {
      build_items(h, cpb, dteam);
      const int nit = (int)h->items.size();
      std::vector<int> grids = {std::min(nit, 65535)};
      if (bf16) grids.insert(grids.end(), {std::min(nit, 2 * sms), std::min(nit, 4 * sms)});
      else grids.push_back(0);  // the resident CTAs
      for (int grid : grids)
        for (int pd : pd_list) {
          bool dup = false;
          for (auto& c : tried) dup |= c.cpb == cpb && c.dteam == dteam && c.grid == grid && c.pd == pd;
          if (!dup) tried.push_back({cpb, dteam, grid, pd, 1e30f});
        }
    }
  }
  // Two passes over all candidates, each timing enough launches to span about
  // 2 ms (at least 3) after one untimed launch; a candidate keeps its faster
  // pass, so that clock and cache drift over the tuning do not pick the shape.
  int reps = 3;
  for (int pass = 0; pass < 2; ++pass) {
    int cur_cpb = -1, cur_dteam = -1;
    for (auto& c : tried) {
      if (c.cpb != cur_cpb || c.dteam != cur_dteam) {
        build_items(h, c.cpb, c.dteam);
        CUDA_TRY(h, cudaMemcpyAsync(h->items_d, h->items.data(), h->items.size() * sizeof(WorkItem),
                                    cudaMemcpyHostToDevice, s));
        cur_cpb = c.cpb;
        cur_dteam = c.dteam;
      }
      SweepArgs a = sweep_args(h);
      a.counters = nullptr;
      a.In = a.Ik = h->Ibuf[src];
      a.Iout = h->Ibuf[spare];
      a.ff = ff ? 1 : 0;
      CUDA_TRY(h, launch_sweep(h->opts.precision, c.pd, a, dim, h->threads, c.grid, s));
      CUDA_TRY(h, cudaEventRecord(h->ev0, s));
      for (int r = 0; r < reps; ++r) CUDA_TRY(h, launch_sweep(h->opts.precision, c.pd, a, dim, h->threads, c.grid, s));
      CUDA_TRY(h, cudaEventRecord(h->ev1, s));
      CUDA_TRY(h, cudaEventSynchronize(h->ev1));
      float ms = 0.f;
      CUDA_TRY(h, cudaEventElapsedTime(&ms, h->ev0, h->ev1));
      ms /= (float)reps;
      if (pass == 0 && &c == &tried.front()) reps = std::min(30, std::max(3, (int)std::ceil(2.0f / std::max(ms, 1e-3f))));
      c.ms = std::min(c.ms, ms);
    }
  }
  for (auto& c : tried)
    if (c.ms < best_ms) { best_ms = c.ms; best_cpb = c.cpb; best_dteam = c.dteam; best_grid = c.grid; best_pd = c.pd; }
  build_items(h, best_cpb, best_dteam);
  h->grid = best_grid;
  h->pd = best_pd;
  CUDA_TRY(h, cudaMemcpyAsync(h->items_d, h->items.data(), h->items.size() * sizeof(WorkItem), cudaMemcpyHostToDevice, s));
  CUDA_TRY(h, cudaStreamSynchronize(s));
  drop_graphs(h);
  char buf[256];
  h->tune_report = "cells_per_cta,threads,grid,min_ctas_variant,ms_per_launch,directions_per_step\n";
  for (auto& c : tried) {
    snprintf(buf, sizeof buf, "%d,%d,%d,%d,%.4f,%d\n", c.cpb, c.cpb * h->lpc * c.dteam, c.grid, c.pd, c.ms, c.dteam);
    h->tune_report += buf;
  }
  snprintf(buf, sizeof buf, "chosen,%d,%d,%d,%d,%d\n", best_cpb, best_cpb * h->lpc * h->dteam, best_grid, best_pd,
           h->dteam);
  h->tune_report += buf;
  if (report && report_len) {
    std::strncpy(report, h->tune_report.c_str(), report_len - 1);
    report[report_len - 1] = 0;
  }
  return BTE_OK;
}

int bte_get_T(bte_handle h, int geom, int which, double* out, int on_device) {
  int rc = check_geom(h, geom);
  if (rc) return rc;
  if (!out) return fail(h, BTE_E_ARG, "out is NULL");
  if (!h->mem_ready || !h->init_set[geom]) return fail(h, BTE_E_STATE, "geometry %d has no state", geom);
  if (which != BTE_T_PSEUDO && which != BTE_T_LATTICE && which != BTE_E_LATTICE)
    return fail(h, BTE_E_ARG, "which must be BTE_T_PSEUDO, BTE_T_LATTICE or BTE_E_LATTICE");
  const bte_geom& g = h->geoms[geom];
  const size_t nc = (size_t)g.nx * g.ny * g.nz;
  const double* src;
  if (which == BTE_E_LATTICE) {
    if (h->EL_partial) return fail(h, BTE_E_STATE, "E_L of a band-range handle needs a step after bte_set_intensity");
    src = h->EL;
  } else if (which == BTE_T_PSEUDO && h->solve_tp) {
    src = h->Tp;
  } else {
    if (h->EL_partial) return fail(h, BTE_E_STATE, "T_L of a band-range handle needs a step after bte_set_intensity");
    if ((rc = ensure_TL(h))) return rc;
    src = h->TL;
  }
  return copy_out(h, out, src + h->cell0[geom], nc, on_device);
}

int bte_get_flux(bte_handle h, int geom, double* q_cells, double* q_walls, int on_device) {
  int rc = check_geom(h, geom);
  if (rc) return rc;
  if (!h->mem_ready || !h->init_set[geom]) return fail(h, BTE_E_STATE, "geometry %d has no state", geom);
  const bte_geom& g = h->geoms[geom];
  const int nc = g.nx * g.ny * g.nz;
  CUDA_TRY(h, ensure_initial_doubles(h));
  const void* I = h->Ibuf[h->cur];
  const int prec = h->opts.precision;
  cudaStream_t s = h->stream;
  if (q_cells) {
    double* q = on_device ? q_cells : h->scratch_q;
    CUDA_TRY(h, launch_flux_cells(prec, h->state_ff, true, I, q, h->Sdev, h->cell0[geom], nc, h->nd, h->nbp, g.dim, s));
    if (!on_device) CUDA_TRY(h, cudaMemcpyAsync(q_cells, q, (size_t)nc * g.dim * 8, cudaMemcpyDeviceToHost, s));
  }
  if (q_walls) {
    double res[6] = {0, 0, 0, 0, 0, 0};
    int nf[6] = {0, 0, 0, 0, 0, 0};
    for (int side = 0; side < 2 * g.dim; ++side) nf[side] = (int)side_faces(g, side);
    CUDA_TRY(h, refresh_ghosts(h));
    CUDA_TRY(h, launch_flux_walls(prec, h->state_ff, I, h->I0ref_o, h->I0wall, h->geoms_d, geom, h->wall_dirs.data(), h->Sdev, h->nd,
                                  h->nbp, h->scratch_faces, h->max_side_faces, nf, 2 * g.dim, h->scratch_out, s));
    CUDA_TRY(h, cudaMemcpyAsync(res, h->scratch_out, 2 * g.dim * 8, cudaMemcpyDeviceToHost, s));
    CUDA_TRY(h, cudaStreamSynchronize(s));
    if (on_device) CUDA_TRY(h, cudaMemcpy(q_walls, res, 2 * g.dim * 8, cudaMemcpyHostToDevice));
    else std::memcpy(q_walls, res, 2 * g.dim * 8);
  }
  CUDA_TRY(h, cudaStreamSynchronize(s));
  return BTE_OK;
}

int bte_get_intensity(bte_handle h, int geom, double* out, int on_device) {
  int rc = check_geom(h, geom);
  if (rc) return rc;
  if (!out) return fail(h, BTE_E_ARG, "out is NULL");
  if (!h->mem_ready || !h->init_set[geom]) return fail(h, BTE_E_STATE, "geometry %d has no state", geom);
  const bte_geom& g = h->geoms[geom];
  const long long nc = (long long)g.nx * g.ny * g.nz;
  const int prec = h->opts.precision;
  const size_t es = elem_bytes(prec);
  CUDA_TRY(h, ensure_initial_doubles(h));
  const char* I = h->Ibuf[h->cur] + (size_t)h->cell0[geom] * h->nd * h->nbp * es;
  for (long long c0 = 0; c0 < nc; c0 += on_device ? nc : h->pack_cells) {
    const long long n = on_device ? nc : std::min(h->pack_cells, nc - c0);
    double* dst = on_device ? out : h->scratch_pack;
    CUDA_TRY(h, launch_unpack(prec, h->state_ff, I + (size_t)c0 * h->nd * h->nbp * es, dst, h->I0ref_o, h->rows_d, n, h->nd,
                              h->nb, h->nbp, h->stream));
    if (!on_device)
      CUDA_TRY(h, cudaMemcpyAsync(out + (size_t)c0 * h->nd * h->nb, dst, (size_t)n * h->nd * h->nb * 8,
                                  cudaMemcpyDeviceToHost, h->stream));
  }
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  return BTE_OK;
}

int bte_set_intensity(bte_handle h, int geom, const double* in, const double* Tp_cells, int on_device) {
  int rc = check_geom(h, geom);
  if (rc) return rc;
  if (!in || !Tp_cells) return fail(h, BTE_E_ARG, "in and Tp_cells are required");
  if (!h->mem_ready || !h->init_set[geom]) return fail(h, BTE_E_STATE, "bte_set_initial must come first for geometry %d", geom);
  const bte_geom& g = h->geoms[geom];
  const long long nc = (long long)g.nx * g.ny * g.nz;
  const int prec = h->opts.precision;
  const size_t es = elem_bytes(prec);
  char* I = h->Ibuf[h->cur] + (size_t)h->cell0[geom] * h->nd * h->nbp * es;
  cudaStream_t s = h->stream;
  CUDA_TRY(h, cudaMemcpyAsync(h->Tp + h->cell0[geom], Tp_cells, nc * 8, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s));
  // a restored state is kept as given, in doubles, until a double-float step; a lone
  // geometry's is overwritten whole, and has no state when a call below fails half-way
  if (h->geoms.size() > 1) CUDA_TRY(h, ensure_state_doubles(h));
  else if (h->state_ff) h->init_set[geom] = h->state_ff = false;
  h->initial = false;
  CUDA_TRY(h, launch_state_from_Tp(h->I0cell + h->cell0[geom] * h->nbp, h->J + h->cell0[geom] * 4 * h->nbp_all,
                                   h->Msum + h->cell0[geom] * 4, h->MsumL + h->cell0[geom] * 4,
                                   h->Tp + h->cell0[geom], h->Teval + h->cell0[geom], nc, thermo(h), s));
  for (long long c0 = 0; c0 < nc; c0 += on_device ? nc : h->pack_cells) {
    const long long n = on_device ? nc : std::min(h->pack_cells, nc - c0);
    const double* src = in + (size_t)c0 * h->nd * h->nb;
    if (!on_device) {
      CUDA_TRY(h, cudaMemcpyAsync(h->scratch_pack, src, (size_t)n * h->nd * h->nb * 8, cudaMemcpyHostToDevice, s));
      src = h->scratch_pack;
    }
    char* dst = I + (size_t)c0 * h->nd * h->nbp * es;
    SweepArgs a = sweep_args(h);  // these cells' energies
    a.Iout = dst;
    a.I0cell = h->I0cell + (h->cell0[geom] + c0) * h->nbp;
    a.Ec = h->Ec + (h->cell0[geom] + c0) * kRedEntries;
    CUDA_TRY(h, launch_pack(prec, src, dst, h->I0ref_o, h->rows_d, n, h->nd, h->nb, h->nbp, h->Epart ? nullptr : &a, s));
    if (!on_device) CUDA_TRY(h, cudaStreamSynchronize(s));  // the caller's pageable memory and the staging buffer are reused
  }
  if (h->Epart) h->EL_partial = true;  // this handle holds only its bands' share of E_L until the next step's exchange
  else CUDA_TRY(h, launch_energy_L(h->Ec + h->cell0[geom] * kRedEntries, h->EL + h->cell0[geom], nc, s));
  CUDA_TRY(h, cudaStreamSynchronize(s));
  h->init_set[geom] = true;
  h->TL_valid = false;
  h->bscale_valid = false;
  return BTE_OK;
}

int bte_get_directions(bte_handle h, double* S, double* w, int* refl) {
  if (!h) return BTE_E_ARG;
  const int n = h->nd;
  for (int p = 0; p < n; ++p) {  // the caller's order
    const int d = h->perm[p];
    for (int c = 0; c < 3; ++c) {
      if (S) S[3 * d + c] = h->S[3 * p + c];
      if (refl) refl[c * n + d] = h->perm[h->refl[c * n + p]];
    }
    if (w) w[d] = h->w[p];
  }
  return h->nd;
}

// ---- learned guess ---------------------------------------------------------
namespace {

// Xavier-uniform weights and zero biases for one net (host SplitMix64 stream).
void mlp_init_host(std::vector<float>& p, int k, unsigned long long seed) {
  p.assign(mlp_param_count(k), 0.f);
  unsigned long long st = seed;
  auto next = [&]() {
    st += 0x9E3779B97F4A7C15ULL;
    unsigned long long z = st;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    z ^= z >> 31;
    return (double)(z >> 11) * (1.0 / 9007199254740992.0);
  };
  auto fill = [&](size_t off, int fan_in, int fan_out, int n) {
    const double a = std::sqrt(6.0 / (fan_in + fan_out));
    for (int i = 0; i < n; ++i) p[off + i] = (float)((2.0 * next() - 1.0) * a);
  };
  fill(0, 1, kHidden, kHidden);                                      // W1
  fill(2 * kHidden, kHidden, kHidden, kHidden * kHidden);           // W2
  fill(3 * kHidden + kHidden * kHidden, kHidden, k, k * kHidden);   // W3
}

int mlp_net_offset(const bte_ctx* h, int net, int* k) {
  *k = net == 0 ? 1 : h->nb_all;
  return net == 0 ? 0 : mlp_param_count(1);
}

}  // namespace

int bte_train_mlp(bte_handle h, long long n_pairs, double T_lo, double T_hi, int epochs, unsigned long long seed,
                  double* loss) {
  if (!h) return BTE_E_ARG;
  int rc = ensure_memory(h);
  if (rc) return rc;
  if (n_pairs < 1024 || n_pairs > (1LL << 26)) return fail(h, BTE_E_ARG, "n_pairs must lie in [1024, 2^26]");
  if (!(T_lo >= kTmin && T_hi <= kTmax && T_hi > T_lo + 1.0)) return fail(h, BTE_E_ARG, "need 1 <= T_lo < T_hi <= 5000 K");
  if (epochs < 1) return fail(h, BTE_E_ARG, "epochs must be >= 1");
  cudaStream_t s = h->stream;
  const int n = (int)n_pairs, nb = h->nb_all, B = 1024;
  // normalisation
  h->mlp_Tlo = T_lo;
  h->mlp_Thi = T_hi;
  CUDA_TRY(h, launch_mlp_norm(thermo(h), T_lo, T_hi, h->I0ref, h->mlp_rlo, h->mlp_rhi, h->mlp_elohi, s));
  double el[2];
  CUDA_TRY(h, cudaMemcpyAsync(el, h->mlp_elohi, 16, cudaMemcpyDeviceToHost, s));
  CUDA_TRY(h, cudaStreamSynchronize(s));
  h->mlp_Elo = el[0];
  h->mlp_Ehi = el[1];
  // temporary training buffers (stream-ordered allocation, freed before returning)
  const size_t pair_f = (size_t)n * (2 + nb), act_f = (size_t)(4 * kHidden + 2 * nb) * B, part_f = 8192;
  float* tmp = nullptr;
  CUDA_TRY(h, cudaMallocAsync((void**)&tmp, (pair_f + act_f + part_f) * 4, s));
  float* xA = tmp;
  float* yA = xA + n;
  float* yB = yA + n;
  float* act = yB + (size_t)nb * n;
  float* part = act + act_f;
  cudaError_t e = launch_mlp_pairs(thermo(h), T_lo, T_hi, h->I0ref, h->mlp_rlo, h->mlp_rhi, h->mlp_elohi, seed, n, xA,
                                   yA, yB, s);
  double losses[2] = {0.0, 0.0};
  for (int net = 0; net < 2 && e == cudaSuccess; ++net) {
    int k;
    const int off = mlp_net_offset(h, net, &k);
    const int np = mlp_param_count(k);
    std::vector<float> init;
    mlp_init_host(init, k, seed * 2654435761ULL + 17 + net);
    e = cudaMemcpyAsync(h->mlp_p + off, init.data(), np * 4, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(h->mlp_m + off, 0, np * 4, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(h->mlp_v + off, 0, np * 4, s);
    const float* X = net == 0 ? xA : yA;
    const float* Tg = net == 0 ? yA : yB;
    const int steps_per_epoch = std::max(1, n / B);
    int t = 0;
    for (int ep = 0; ep < epochs && e == cudaSuccess; ++ep) {
      const float lr = 2e-3f * std::pow(0.1f, (float)ep / (float)std::max(1, epochs - 1));  // decay to lr/10
      for (int st = 0; st < steps_per_epoch && e == cudaSuccess; ++st) {
        const int o = (int)(((long long)st * B + (long long)ep * 7919) % (n - B + 1));
        e = mlp_forward_backward(h->mlp_p + off, k, X + o, n, Tg + o, n, B, h->mlp_g + off, act, part, s);
        if (e == cudaSuccess) e = launch_adam(h->mlp_p + off, h->mlp_g + off, h->mlp_m + off, h->mlp_v + off, np, lr, ++t, s);
      }
    }
    // loss over the first min(n, 8192) pairs with the trained weights
    const int Bev = std::min(n, 8192);
    float* evact = nullptr;
    if (e == cudaSuccess) e = cudaMallocAsync((void**)&evact, ((size_t)(4 * kHidden + 2 * k) * Bev + 4 * (size_t)np) * 4, s);
    if (e == cudaSuccess)
      e = mlp_forward_backward(h->mlp_p + off, k, X, n, Tg, n, Bev, evact + (size_t)(4 * kHidden + 2 * k) * Bev,
                               evact, part, s);
    std::vector<float> hp((k * (size_t)Bev + 255) / 256);
    if (e == cudaSuccess) e = cudaMemcpyAsync(hp.data(), part, hp.size() * 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    for (float v : hp) losses[net] += v;
    if (evact) cudaFreeAsync(evact, s);
  }
  cudaFreeAsync(tmp, s);
  cudaError_t e2 = cudaStreamSynchronize(s);
  if (e != cudaSuccess || e2 != cudaSuccess)
    return fail(h, BTE_E_CUDA, "training: %s", cudaGetErrorString(e != cudaSuccess ? e : e2));
  h->mlp_trained = true;
  if (loss) {
    loss[0] = losses[0];
    loss[1] = losses[1];
  }
  return BTE_OK;
}

int bte_mlp_params(bte_handle h, int net, float* out, int n) {
  if (!h || (net != 0 && net != 1)) return BTE_E_ARG;
  int rc = ensure_memory(h);
  if (rc) return rc;
  int k;
  const int off = mlp_net_offset(h, net, &k);
  const int np = mlp_param_count(k);
  if (!out) return np;
  if (n < np) return fail(h, BTE_E_ARG, "need %d floats", np);
  CUDA_TRY(h, cudaMemcpy(out, h->mlp_p + off, np * 4, cudaMemcpyDeviceToHost));
  return np;
}

int bte_mlp_set_params(bte_handle h, int net, const float* in, int n) {
  if (!h || (net != 0 && net != 1) || !in) return BTE_E_ARG;
  int rc = ensure_memory(h);
  if (rc) return rc;
  int k;
  const int off = mlp_net_offset(h, net, &k);
  const int np = mlp_param_count(k);
  if (n != np) return fail(h, BTE_E_ARG, "net %d has %d parameters", net, np);
  CUDA_TRY(h, cudaMemcpy(h->mlp_p + off, in, np * 4, cudaMemcpyHostToDevice));
  return BTE_OK;
}

int bte_mlp_grad(bte_handle h, int net, const float* x, const float* y, int n, float* grad, double* loss) {
  if (!h || (net != 0 && net != 1) || !x || !y || !grad || n < 1 || n > 65536) return BTE_E_ARG;
  int rc = ensure_memory(h);
  if (rc) return rc;
  int k;
  const int off = mlp_net_offset(h, net, &k);
  const int np = mlp_param_count(k);
  cudaStream_t s = h->stream;
  const size_t act_f = (size_t)(4 * kHidden + 2 * k) * n, parts = ((size_t)k * n + 255) / 256;
  float* tmp = nullptr;
  CUDA_TRY(h, cudaMallocAsync((void**)&tmp, ((size_t)n + (size_t)k * n + act_f + parts + np) * 4, s));
  float* dx = tmp;
  float* dy = dx + n;
  float* act = dy + (size_t)k * n;
  float* part = act + act_f;
  float* g = part + parts;
  cudaError_t e = cudaMemcpyAsync(dx, x, (size_t)n * 4, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(dy, y, (size_t)k * n * 4, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = mlp_forward_backward(h->mlp_p + off, k, dx, n, dy, n, n, g, act, part, s);
  std::vector<float> hp(parts);
  if (e == cudaSuccess) e = cudaMemcpyAsync(grad, g, (size_t)np * 4, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(hp.data(), part, parts * 4, cudaMemcpyDeviceToHost, s);
  cudaFreeAsync(tmp, s);
  cudaError_t e2 = cudaStreamSynchronize(s);
  if (e != cudaSuccess || e2 != cudaSuccess) return fail(h, BTE_E_CUDA, "mlp grad: %s", cudaGetErrorString(e != cudaSuccess ? e : e2));
  if (loss) {
    double l = 0.0;
    for (float v : hp) l += v;
    *loss = l;
  }
  return BTE_OK;
}

int bte_solve_T(bte_handle h, const double* Ep, const double* T0, int n, int learned, double* T_out, int* evals) {
  if (!h || !Ep || !T_out || n < 1) return BTE_E_ARG;
  int rc = ensure_memory(h);
  if (rc) return rc;
  if (learned && !h->mlp_trained) return fail(h, BTE_E_STATE, "bte_train_mlp must come first");
  if (!h->solve_tp) return fail(h, BTE_E_STATE, "every beta_b is zero: the T_p equation is empty");
  cudaStream_t s = h->stream;
  double* tmp = nullptr;
  CUDA_TRY(h, cudaMallocAsync((void**)&tmp, (size_t)n * (3 * 8 + 4), s));
  double* dE = tmp;
  double* dT0 = dE + n;
  double* dT = dT0 + n;
  int* dev = (int*)(dT + n);
  cudaError_t e = cudaMemcpyAsync(dE, Ep, (size_t)n * 8, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess && T0) e = cudaMemcpyAsync(dT0, T0, (size_t)n * 8, cudaMemcpyHostToDevice, s);
  const MLPView m = mlp_view(h);
  if (e == cudaSuccess)
    e = launch_solve_batch(thermo(h), dE, T0 ? dT0 : nullptr, n, model_trust(h->opts.newton_rtol),
                           h->opts.newton_maxit, learned ? &m : nullptr, dT, dev, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(T_out, dT, (size_t)n * 8, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess && evals) e = cudaMemcpyAsync(evals, dev, (size_t)n * 4, cudaMemcpyDeviceToHost, s);
  cudaFreeAsync(tmp, s);
  cudaError_t e2 = cudaStreamSynchronize(s);
  if (e != cudaSuccess || e2 != cudaSuccess) return fail(h, BTE_E_CUDA, "solve: %s", cudaGetErrorString(e != cudaSuccess ? e : e2));
  return BTE_OK;
}

int bte_destroy(bte_handle h) {
  if (!h) return BTE_E_ARG;
  if (h->stream) cudaStreamSynchronize(h->stream);
  else cudaDeviceSynchronize();
  drop_graphs(h);
  if (h->cap_stream) cudaStreamDestroy(h->cap_stream);
  if (h->ws_owned && h->ws) cudaFree(h->ws);
  for (auto& sides : h->gdir)
    for (void* p : sides)
      if (p) cudaFree(p);
  if (h->ev0) cudaEventDestroy(h->ev0);
  if (h->ev1) cudaEventDestroy(h->ev1);
  for (cudaEvent_t ev : h->tev) cudaEventDestroy(ev);
  delete h;
  return BTE_OK;
}

int bte_set_sweep_timing(bte_handle h, int on) {
  if (!h) return BTE_E_ARG;
  if ((on != 0) != h->time_sweeps) drop_graphs(h);  // the step graphs gain or lose the event nodes
  h->time_sweeps = on != 0;
  h->tev_n = 0;
  return BTE_OK;
}

int bte_sweep_times(bte_handle h, float* ms, int n) {
  if (!h || (n > 0 && !ms)) return BTE_E_ARG;
  if (!h->time_sweeps || h->tev_n == 0) return fail(h, BTE_E_STATE, "no timed step since bte_set_sweep_timing");
  CUDA_TRY(h, cudaEventSynchronize(h->tev[2 * h->tev_n - 1]));
  for (int i = 0; i < n && i < h->tev_n; ++i) CUDA_TRY(h, cudaEventElapsedTime(ms + i, h->tev[2 * i], h->tev[2 * i + 1]));
  return h->tev_n;
}

const char* bte_last_error(bte_handle h) {
  if (!h) return g_init_err.c_str();
  return h->err.c_str();
}

}  // extern "C"
