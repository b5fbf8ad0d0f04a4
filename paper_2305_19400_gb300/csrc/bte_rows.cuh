// bte_rows.cuh -- the sweep of one inner iteration (sm_103a), FP64 and FP32
// storage: for every (cell, direction, band) (Sec. 3.1, Eq. 5)
//   I^{k+1} = [I^n/dt + beta_b I0_b^k + v_b sum_ax c_ax,d I_up,ax^k] / [1/dt + beta_b + v_b sum_ax c_ax,d],
//   c_ax,d = |S_ax,d| / (w_d Delta_ax),
// (implicit: point-Jacobi sweep of backward Euler) or the forward-Euler form of
// Eq. 3, and every lane's share of the cell's energies sum_b G_b / v_b and
// sum_b beta_b G_b / v_b, G_b = sum_d w_d I^{k+1}_{d,b}, to Ec, from which cells_kernel
// (bte_cells.cu) solves T_p and refreshes I0.  The upwind value is
// the neighbour cell's on the side S_d comes from, or the Eq. 6 ghost at a wall.
//
// Work layout.  A lane holds 16 bytes of one row, V consecutive bands, and a
// cell is served by DT teams of nbp/V lanes.  Rows stand in the internal
// direction order (bte_tables.h): blocks of 4 (in-plane sets) or 8 rows (polar x
// azimuthal) that differ only in the signs of S, so a block needs one set of
// coefficients.  Team dg takes row DT k + dg of a block in step k: a step reads
// DT consecutive rows per array (0.9 KB with 55 bands in FP64), and the RUN
// steps of a block share the coefficients, which so cost L2 traffic, shared
// memory and instructions once per RUN updates.
//
// Memory.  I^n is read once, I^{k+1} written once, and each I^k row read from
// DRAM once (neighbouring cells, processed together, read it from L2); L2 to SM
// traffic, 9 TB/s on the 128x128 FP64 workload with coefficients read per
// direction, bounds the sweeps more than DRAM.  Every thread copies the operands
// of its next kSlots - 1 steps into its own ring slots with cp.async.  The
// issuing side runs ahead across the items of a persistent CTA, so the ring
// never drains between two cells, and nothing in a CTA waits on another thread
// (no barrier, except to change the table of a cell-size class).
//
// Operand addresses are base + row x scale: a neighbour's row, a ghost row of
// the face (scale 0), a per-direction ghost row, or the cell's own mirrored row
// (r ^ 1, r ^ 3, r ^ 4: a constant shift of the base except in Map<1> and Map<3>), so wall
// cells run the same instructions as interior ones.
#pragma once
#include <algorithm>
#include <type_traits>

#include "bte_ff.cuh"
#include "bte_pdl.cuh"
#include "bte_quad.cuh"
#include "bte_store.cuh"

namespace bte {
namespace rows {

// MAP 1: in-plane sets (blocks of 4 rows, one team); 2 and 4: polar x azimuthal
// sets (blocks of 8 rows, two or four teams); 3: these with one team.
template <int MAP>
struct Map;
template <>
struct Map<3> {
  static constexpr int DT = 1, RUN = 8;
};
template <>
struct Map<1> {
  static constexpr int DT = 1, RUN = 4;
};
template <>
struct Map<2> {
  static constexpr int DT = 2, RUN = 4;
};
template <>
struct Map<4> {
  static constexpr int DT = 4, RUN = 2;
};

__device__ __forceinline__ void cp16(unsigned smem, const void* g) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ double2 ld2(const double* p) { return __ldg(reinterpret_cast<const double2*>(p)); }

// ------------------------------------------------------------------- modes
// FP64 storage in double-float arithmetic (bte_ff.cuh), implicit: divided
// through by v_b,
//   I' = W I^n + R (sum_ax c_ax u_ax + (beta_b/v_b) I0),
//   R = 1/(1/(v_b dt) + beta_b/v_b + sum_ax c_ax),  W = R/(v_b dt),
// beta_b/v_b and (beta_b/v_b) I0 in registers, c_ax of the block from shared memory, R
// and W of the block from their table one block ahead.  Forming W I^n in every iteration
// costs four packed operations more than reading a stored B, and saves the first
// iteration's write of B and its third buffer's traffic.  The tables come from the host
// in double-float form: R the pair nearest its value, and W = 1 - R (beta_b/v_b + sum c_ax)
// of that pair, formed in double-double (below 1/4 the pair nearest R/(v_b dt)), so that W +
// R (beta_b/v_b + sum c_ax) = 1 holds to 2^-49 W and a uniform equilibrium stays in place: after 4000 iterations at dt = 0.2
// ps 1e-14 rms from it, where R I^n/(v_b dt) from two products drifted by 1.2e-13 and W
// formed on the device by 1.1e-12.  I^n/(v_b dt), added to the upwind sum before one
// product with R, rounds alike in all directions of a cell near equilibrium (1.5e-15 of a
// uniform state's band in one update, here 0.4e-15).
// The direction sum adds a block's rows first, then the block to its run of equal
// weights, then the run times its weight to G: the rows of a block are close to equal, and
// adding equal pairs twenty in a row without renormalising leaves 1.5e-14 rms where blocks
// of four leave 2e-15, at the same number of operations.
// Bound by HBM (24 bytes an update) and L2 to SM traffic; of few directions by
// issue (0.51 of the slots at 16 warps per SM).  With coefficients read per
// direction and the cells' step in the same kernel: 128x128 x 400 x 55 1535 us an
// iteration, 23x18x13 867, 120x120 x 20 x 55 124; now 1410, 520 and 69, and 43, 30
// and 30 for the cells.
struct FF {
  using S = double;
  static constexpr int V = 2, kMinB = 2;
  static constexpr bool kStoreB = false, kFour = false;
  template <int DIM>
  static constexpr int slots = DIM == 2 ? 8 : 6;
  template <int DIM>
  struct Tab {
    ff::x2 ch[DIM], cl[DIM];  // c_ax high and low parts, each in both halves
    float w32, wlo;           // w_d as a double-float pair
    unsigned key;             // equal weights, equal keys (the runs of the direction sums)
    unsigned pad;
  };
  struct Lane {
    ff::P2 betav;
  };
  template <int DIM>
  struct Coef {
    ff::P2 R, W;
  };
  struct Cell {
    ff::P2 src;
  };
  struct Acc {
    ff::P2 B, S, G, w;  // sums of a block, of the run, of the closed runs; the run's weight
    unsigned key;
  };
  template <int DIM>
  __device__ static Tab<DIM> tab(const SweepArgs& a, int cls, int d) {
    Tab<DIM> e;
    e.w32 = a.wdir32[d];
    e.wlo = (float)(a.wdir[d] - (double)e.w32);
    e.key = __float_as_uint(e.w32) ^ __float_as_uint(e.wlo);
    e.pad = 0;
    const float* c = a.dirc_ff + ((size_t)cls * a.nd + d) * 6;
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
      e.ch[k] = ff::pack(c[2 * k], c[2 * k]);
      e.cl[k] = ff::pack(c[2 * k + 1], c[2 * k + 1]);
    }
    return e;
  }
  __device__ static Lane lane(const SweepArgs& a, int b0) {
    return Lane{ff::ldg(a.band_ff + 2 * b0)};
  }
  template <int DIM>
  __device__ static Coef<DIM> coef(const SweepArgs& a, int cls, int d, int b0) {
    const double* p = reinterpret_cast<const double*>(a.coef_R) + 2 * (((size_t)cls * a.nd + d) * a.th.nbo + b0);
    return Coef<DIM>{ff::ldg(p), ff::ldg(p + 2)};
  }
  __device__ static Cell cell(const SweepArgs&, const Lane& l, const double (&i0)[V], int, long long) {
    return Cell{ff::norm(ff::mul(l.betav, ff::from_doubles(i0[0], i0[1])))};
  }
  __device__ static Acc acc(const SweepArgs&, const Cell&) { return Acc{ff::zero(), ff::zero(), ff::zero(), ff::zero(), 0xffffffffu}; }
  template <int DIM>
  struct Block {
    ff::P2 c[DIM], R, W;
  };
  template <int DIM, int RUN>
  __device__ static Block<DIM> block(const SweepArgs&, const Lane&, const Cell&, const Coef<DIM>& cf, const Tab<DIM>& t,
                                     Acc& s) {
    ff::acc(s.S, s.B);
    if (t.key != s.key) {
      ff::acc(s.G, ff::mul(s.w, s.S));
      s.S = ff::zero();
      s.w = ff::P2{ff::pack(t.w32, t.w32), ff::pack(t.wlo, t.wlo)};
      s.key = t.key;
    }
    Block<DIM> b;
    b.R = cf.R;
    b.W = cf.W;
#pragma unroll
    for (int k = 0; k < DIM; ++k) b.c[k] = ff::P2{t.ch[k], t.cl[k]};
    return b;
  }
  template <int DIM, bool FIRST>
  __device__ static void step(const SweepArgs&, const Lane&, const Cell& c, const Block<DIM>& b, unsigned sb, unsigned ostr,
                              char* out, char*, bool on, Acc& s) {
    ff::P2 t = ff::mul(b.c[0], ff::lds(sb + ostr));
#pragma unroll
    for (int k = 1; k < DIM; ++k) t = ff::add(t, ff::mul(b.c[k], ff::lds(sb + (1 + k) * ostr)));
    const ff::P2 r = ff::norm(ff::add(ff::mul(b.W, ff::lds(sb)), ff::mul(b.R, ff::add(t, c.src))));
    if (on) ff::st_stream(out, r);
    if (FIRST) s.B = r;
    else ff::acc(s.B, r);
  }
  __device__ static void finish(const SweepArgs&, const Cell&, Acc& s, int, int, double (&G)[V]) {
    ff::acc(s.S, s.B);
    ff::acc(s.G, ff::mul(s.w, s.S));
    ff::to_doubles(ff::norm(s.G), G[0], G[1]);
  }
  __device__ static const void* wall_rows(const SweepArgs& a) { return a.I0wall_ff; }
};

// FP64 storage in IEEE arithmetic: I' = A_n I^n + A_x I_x + A_y I_y (+ A_z I_z) + A_s I0
// with coefficients already divided by the diagonal, one set per block.  BM:
// 0 I^n read; 1 B = A_n I^n (the same in all inner iterations of a step) also
// stored; 2 B read.  A_s I0 is formed once per block, so an update takes 3 FP64
// operations (2-D; 4 with BM 1), the bound of this form: 0.53e12 FP64 FMAs per
// second, measured.  TT: the relaxation rates depend on T, beta_b(T_p) = beta_b s;
// every coefficient takes the factor y = 1/(1 + (s - 1) A_s), A_s also s (explicit
// scheme: A_n + (1 - s) A_s and s A_s).  y is formed once per block too, by
// rcp_pos (an FP32 reciprocal and one third-order step inside its range, a division
// outside it: s runs to (T_p/T_ref)^16; a correctly rounded reciprocal per update took
// 1745 us on 64x48 cells x 400 x 55).
// The direction sum runs on the integer pipe: over a run of directions with the
// same weight each band adds I in 64-bit fixed point, unit 2^(E - 50) for the
// cell's I0 of exponent E, so a value up to 16 I0 adds at most 2^55 and a run of
// 256 cannot overflow; the run then enters G with one FP64 FMA (sum x w x unit).
// The additions are exact, the terms are cut to whole units: a value of I0's exponent
// loses two bits (3/4 unit at most, 2.2e-16 of it on average, always downwards), any other
// below 16 I0 less than one unit.  Values with a larger exponent (or negative, NaN)
// take the FP64 FMA directly.
// 64x48 x 400 x 55 with tau(T): 1745 -> 601 us; 120x120 x 20 x 55 explicit: 203 -> 107.
template <int BM, bool TT>
struct F64 {
  using S = double;
  static constexpr int V = 2, kMinB = 2;
  static constexpr bool kStoreB = BM == 1, kFour = false;
  template <int DIM>
  static constexpr int slots = DIM == 2 ? 8 : 6;
  template <int DIM>
  struct Tab {
    double w;
  };
  struct Lane {};
  template <int DIM>
  struct Coef {
    double2 An, Ax, Ay, Az, As;
  };
  struct Cell {
    double2 i0;  // I0, times s when TT
    double s;
    long long fsc[2];  // unit exponent shifted into a double's exponent field
    int fe0[2];        // largest exponent field summed in fixed point (-1: none)
  };
  struct Acc {
    unsigned long long f[2];
    double G[2];
    long long w;
    int n;
  };
  template <int DIM>
  struct Block {
    double2 An, Ax, Ay, Az, k, y;  // y: the factor of B (TT)
    double w;
  };
  template <int DIM>
  __device__ static Tab<DIM> tab(const SweepArgs& a, int, int d) { return Tab<DIM>{a.wdir[d]}; }
  __device__ static Lane lane(const SweepArgs&, int) { return Lane{}; }
  template <int DIM>
  __device__ static Coef<DIM> coef(const SweepArgs& a, int cls, int d, int b0) {
    const size_t plane = (size_t)a.nd * a.th.nbo;
    const double* p = reinterpret_cast<const double*>(a.coef) + (size_t)cls * 5 * plane + (size_t)d * a.th.nbo + b0;
    Coef<DIM> c{};
    if (BM != 2) c.An = ld2(p);
    c.Ax = ld2(p + plane);
    c.Ay = ld2(p + 2 * plane);
    if (DIM == 3) c.Az = ld2(p + 3 * plane);
    c.As = ld2(p + 4 * plane);
    return c;
  }
  __device__ static Cell cell(const SweepArgs& a, const Lane&, const double (&i0)[V], int, long long P) {
    Cell c;
    c.s = TT ? a.bscale[P] : 1.0;
    c.i0 = TT ? make_double2(c.s * i0[0], c.s * i0[1]) : make_double2(i0[0], i0[1]);
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const int e0 = (int)((unsigned long long)__double_as_longlong(i0[v]) >> 52);  // I0 >= 0
      const bool on = e0 >= 200 && e0 <= 1900;
      c.fe0[v] = on ? e0 + 4 : -1;
      c.fsc[v] = on ? (long long)(e0 - 1073) * (1LL << 52) : 0;
    }
    return c;
  }
  __device__ static Acc acc(const SweepArgs&, const Cell&) { return Acc{{0ull, 0ull}, {0.0, 0.0}, 0, 0}; }
  __device__ static void close_run(const Cell& c, Acc& s) {
#pragma unroll
    for (int v = 0; v < V; ++v) {
      if (s.f[v] != 0ull) s.G[v] = fma(__ull2double_rn(s.f[v]), __longlong_as_double(s.w + c.fsc[v]), s.G[v]);
      s.f[v] = 0ull;
    }
    s.n = 0;
  }
  __device__ static void yy(double2& x, double y0, double y1) {
    x.x *= y0;
    x.y *= y1;
  }
  template <int DIM, int RUN>
  __device__ static Block<DIM> block(const SweepArgs& a, const Lane&, const Cell& c, const Coef<DIM>& cf, const Tab<DIM>& t,
                                     Acc& s) {
    const long long wb = __double_as_longlong(t.w);
    if (wb != s.w || s.n + RUN > 256) {
      close_run(c, s);
      s.w = wb;
    }
    s.n += RUN;
    Block<DIM> b;
    b.w = t.w;
    b.y = make_double2(1.0, 1.0);
    b.An = cf.An;
    b.Ax = cf.Ax;
    b.Ay = cf.Ay;
    b.Az = cf.Az;
    b.k = make_double2(cf.As.x * c.i0.x, cf.As.y * c.i0.y);
    if constexpr (TT) {
      if (BM == 0 && a.explicit_scheme) {
        b.An = make_double2(fma(1.0 - c.s, cf.As.x, cf.An.x), fma(1.0 - c.s, cf.As.y, cf.An.y));
      } else {
        const double y0 = rcp_pos(fma(c.s - 1.0, cf.As.x, 1.0)), y1 = rcp_pos(fma(c.s - 1.0, cf.As.y, 1.0));
        yy(b.Ax, y0, y1);
        yy(b.Ay, y0, y1);
        if (DIM == 3) yy(b.Az, y0, y1);
        yy(b.k, y0, y1);
        if (BM == 0) yy(b.An, y0, y1);
        else b.y = make_double2(y0, y1);
      }
    }
    return b;
  }
  __device__ static double2 lds2(unsigned sa) {
    double2 x;
    asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(x.x), "=d"(x.y) : "r"(sa));
    return x;
  }
  template <int DIM, bool FIRST>
  __device__ static void step(const SweepArgs&, const Lane&, const Cell& c, const Block<DIM>& b, unsigned sb, unsigned ostr,
                              char* out, char* bout, bool on, Acc& s) {
    const double2 in = lds2(sb), ux = lds2(sb + ostr), uy = lds2(sb + 2 * ostr);
    double r[2];
    if constexpr (BM == 0) {
      r[0] = fma(b.An.x, in.x, b.k.x);
      r[1] = fma(b.An.y, in.y, b.k.y);
    } else {
      double2 B = in;
      if constexpr (BM == 1) {
        B = make_double2(b.An.x * in.x, b.An.y * in.y);
        if (on) __stcs(reinterpret_cast<double2*>(bout), B);
      }
      r[0] = TT ? fma(B.x, b.y.x, b.k.x) : B.x + b.k.x;
      r[1] = TT ? fma(B.y, b.y.y, b.k.y) : B.y + b.k.y;
    }
    r[0] = fma(b.Ax.x, ux.x, r[0]);
    r[1] = fma(b.Ax.y, ux.y, r[1]);
    r[0] = fma(b.Ay.x, uy.x, r[0]);
    r[1] = fma(b.Ay.y, uy.y, r[1]);
    if constexpr (DIM == 3) {
      const double2 uz = lds2(sb + 3 * ostr);
      r[0] = fma(b.Az.x, uz.x, r[0]);
      r[1] = fma(b.Az.y, uz.y, r[1]);
    }
    if (on) __stcs(reinterpret_cast<double2*>(out), make_double2(r[0], r[1]));
    bool big = false;
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const unsigned long long rb = (unsigned long long)__double_as_longlong(r[v]);
      const int e = (int)(rb >> 52);
      const unsigned long long m = ((rb & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull) << 2;
      const int sh = e == 0 ? 63 : min(c.fe0[v] - e, 63);  // zero (and subnormal) adds nothing
      s.f[v] += sh >= 0 ? (m >> sh) : 0ull;
      big |= sh < 0;
    }
    if (__any_sync(__activemask(), big)) {  // rare: a value beyond the fixed-point range
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const int e = (int)((unsigned long long)__double_as_longlong(r[v]) >> 52);
        if (e != 0 && c.fe0[v] - e < 0) s.G[v] = fma(b.w, r[v], s.G[v]);
      }
    }
  }
  __device__ static void finish(const SweepArgs&, const Cell& c, Acc& s, int, int, double (&G)[V]) {
    close_run(c, s);
    G[0] = s.G[0];
    G[1] = s.G[1];
  }
  __device__ static const void* wall_rows(const SweepArgs& a) { return a.I0wall; }
};

// FP32 storage of the deviation from I0_b(T_ref), FP32 arithmetic, two bands per
// packed instruction: I' = P I^n + Q (v_b sum_ax c_ax u_ax + beta_b (I0 - I0ref)) with
// Q = 1/(1/dt + beta_b + v_b sum c), P = Q/dt (explicit: Q = dt, P = 1 - dt (beta_b +
// v_b sum c)) formed once per block.  The update is affine with coefficients
// summing to one, so the deviation obeys the update of I with I0 and wall ghosts
// shifted.  The float sums of 16 directions go into a double-float sum.
// Bound by HBM, 12 bytes an update: 48x44x40 x 400 x 55 4040 us an iteration with the
// cells' step in the same kernel, 3904 (0.86 of HBM's rate) and 126 for the cells now.
template <bool EXPL>
struct F32 {
  using S = float;
  static constexpr int V = 4, kMinB = 2;
  static constexpr bool kStoreB = false, kFour = true;
  template <int DIM>
  static constexpr int slots = DIM == 2 ? 8 : 6;
  template <int DIM>
  struct Tab {
    float4 c;
    float w, pad[3];
  };
  struct Lane {
    ff::x2 vb[2], bb[2];
  };
  template <int DIM>
  struct Coef {};
  struct Cell {
    ff::x2 bb[2], src[2];
  };
  struct Acc {
    ff::x2 s[2];
    ff::P2 G[2];
    int n;
  };
  template <int DIM>
  struct Block {
    ff::x2 c[DIM], w, P[2], Q[2];
  };
  template <int DIM>
  __device__ static Tab<DIM> tab(const SweepArgs& a, int cls, int d) {
    return Tab<DIM>{a.dirc[(size_t)cls * a.nd + d], a.wdir32[d], {0.f, 0.f, 0.f}};
  }
  __device__ static Lane lane(const SweepArgs& a, int b0) {
    Lane l;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      l.vb[q] = ff::pack(a.vb32[b0 + 2 * q], a.vb32[b0 + 2 * q + 1]);
      l.bb[q] = ff::pack(a.bb32[b0 + 2 * q], a.bb32[b0 + 2 * q + 1]);
    }
    return l;
  }
  template <int DIM>
  __device__ static Coef<DIM> coef(const SweepArgs&, int, int, int) { return Coef<DIM>{}; }
  __device__ static Cell cell(const SweepArgs& a, const Lane& l, const double (&i0)[V], int b0, long long P) {
    Cell c;
    const float s = a.beta_exp != 0.0 ? (float)a.bscale[P] : 1.0f;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      c.bb[q] = ff::mul(l.bb[q], ff::pack(s, s));
      c.src[q] = ff::mul(c.bb[q], ff::pack((float)(i0[2 * q] - a.I0ref[b0 + 2 * q]),
                                           (float)(i0[2 * q + 1] - a.I0ref[b0 + 2 * q + 1])));
    }
    return c;
  }
  __device__ static Acc acc(const SweepArgs&, const Cell&) {
    return Acc{{0ull, 0ull}, {ff::zero(), ff::zero()}, 0};
  }
  template <int DIM, int RUN>
  __device__ static Block<DIM> block(const SweepArgs& a, const Lane& l, const Cell& c, const Coef<DIM>&, const Tab<DIM>& t,
                                     Acc& s) {
    if (s.n == 16) {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        ff::acc(s.G[q], ff::P2{s.s[q], 0ull});
        s.s[q] = 0ull;
      }
      s.n = 0;
    }
    s.n += RUN;
    Block<DIM> b;
    b.c[0] = ff::pack(t.c.x, t.c.x);
    b.c[1] = ff::pack(t.c.y, t.c.y);
    if constexpr (DIM == 3) b.c[2] = ff::pack(t.c.z, t.c.z);
    b.w = ff::pack(t.w, t.w);
    const ff::x2 sum = ff::pack(t.c.w, t.c.w), rdt = ff::pack(a.rdt32, a.rdt32);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const ff::x2 rate = ff::fma(l.vb[q], sum, c.bb[q]);
      if constexpr (EXPL) {
        b.Q[q] = ff::pack(a.dt32, a.dt32);
        b.P[q] = ff::fma(ff::pack(-a.dt32, -a.dt32), rate, ff::pack(1.0f, 1.0f));
      } else {
        const ff::x2 den = ff::add(rdt, rate);
        float q0, q1;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(q0) : "f"(ff::lo_of(den)));
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(q1) : "f"(ff::hi_of(den)));
        b.Q[q] = ff::pack(q0, q1);
        b.P[q] = ff::mul(b.Q[q], rdt);
      }
    }
    return b;
  }
  template <int DIM, bool FIRST>
  __device__ static void step(const SweepArgs&, const Lane& l, const Cell& c, const Block<DIM>& b, unsigned sb, unsigned ostr,
                              char* out, char*, bool on, Acc& s) {
    const ff::P2 in = ff::lds(sb);  // floats 0, 1 and 2, 3
    ff::P2 u = ff::lds(sb + ostr);
    ff::x2 f0 = ff::mul(b.c[0], u.h), f1 = ff::mul(b.c[0], u.l);
#pragma unroll
    for (int k = 1; k < DIM; ++k) {
      u = ff::lds(sb + (1 + k) * ostr);
      f0 = ff::fma(b.c[k], u.h, f0);
      f1 = ff::fma(b.c[k], u.l, f1);
    }
    const ff::P2 r{ff::fma(b.Q[0], ff::fma(l.vb[0], f0, c.src[0]), ff::mul(b.P[0], in.h)),
                   ff::fma(b.Q[1], ff::fma(l.vb[1], f1, c.src[1]), ff::mul(b.P[1], in.l))};
    if (on) ff::st_stream(out, r);
    s.s[0] = ff::fma(b.w, r.h, s.s[0]);
    s.s[1] = ff::fma(b.w, r.l, s.s[1]);
  }
  __device__ static void finish(const SweepArgs& a, const Cell&, Acc& s, int b0, int dg, double (&G)[V]) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      ff::acc(s.G[q], ff::P2{s.s[q], 0ull});
      ff::to_doubles(ff::norm(s.G[q]), G[2 * q], G[2 * q + 1]);
    }
    if (dg == 0)  // the reference part, sum_d w_d I0_b(T_ref)
#pragma unroll
      for (int v = 0; v < V; ++v) G[v] = fma(a.Wtot, a.I0ref[b0 + v], G[v]);
  }
  __device__ static const void* wall_rows(const SweepArgs& a) { return a.I0wall_dev; }
};

// ------------------------------------------------------------------ kernel
// One upwind operand of a cell: the row r of its source lies at base + r x scale
// (scale 0: one ghost row for every direction); mir: bytes of a row when the
// source is the cell's own mirrored row and the shift depends on the step
// (Map<1>, Map<3>; applied as shift x mir).
struct Src {
  const char* base;
  unsigned scale;
  int mir;
};

// A cell of the issuing side: base addresses of its operands for this lane.
template <int DIM>
struct Cursor {
  const char* in;
  Src x[2], y[2], z[2];
  int item, blk;
  unsigned r0;  // first row of this team in the current block
  bool on;
};

template <int DIM, int MAP, class M>
__global__ void __launch_bounds__(256, M::kMinB) rows_kernel(SweepArgs a) {
  using S = typename M::S;
  constexpr int V = M::V, DT = Map<MAP>::DT, RUN = Map<MAP>::RUN, ROWS = DT * RUN;
  constexpr int kOps = 1 + DIM, kSlots = M::template slots<DIM>, kAhead = kSlots - 1;
  extern __shared__ char sm[];
  pdl_trigger();
  const int nbp = a.th.nbo, nblk = a.nd / ROWS, lpc = nbp / V, team = lpc * DT;
  const int slot = threadIdx.x / team, tl = threadIdx.x - slot * team;
  const int dg = tl / lpc, b0 = V * (tl - dg * lpc);
  const unsigned rowB = nbp * (unsigned)sizeof(S);
  const long long cellB = (long long)a.nd * rowB;
  using Tab = typename M::template Tab<DIM>;
  Tab* tabs = reinterpret_cast<Tab*>(sm);
  const unsigned ostr = blockDim.x * 16u, sstr = kOps * ostr;
  const unsigned ring = ((unsigned)__cvta_generic_to_shared(tabs + nblk) + 15u & ~15u) + threadIdx.x * 16u;
  const unsigned rend = ring + kSlots * sstr;
  const typename M::Lane ln = M::lane(a, b0);

  Cursor<DIM> cu;
  // addresses of the cell of this thread's slot in an item (a slot beyond the
  // item's cells repeats its first cell and stores nothing)
  auto setup = [&](int item) {
    const WorkItem wi = a.items[item];
    const DevGeom* gp = a.geoms + wi.geom;
    const int sl = slot < wi.cell_count ? slot : 0;
    const int ci = wi.i0 + sl, cj = wi.j, ck = wi.k, nx = gp->nx, ny = gp->ny;
    const long long P = gp->cell0 + wi.cell_begin + sl;
    const char* ik = reinterpret_cast<const char*>(a.Ik) + P * cellB + b0 * sizeof(S);
    cu.in = reinterpret_cast<const char*>(a.In) + P * cellB + b0 * sizeof(S);
    auto src = [&](int ax, bool low, int c, int n, long long st, long long fl, int shift) -> Src {
      if (low ? c > 0 : c < n - 1) return Src{low ? ik - st : ik + st, rowB, 0};
      const int side = 2 * ax + (low ? 0 : 1), bc = gp->bc[side];
      if (bc == 1) return Src{ik + shift * (int)rowB, rowB, (int)rowB};
      if (bc == 3) return Src{reinterpret_cast<const char*>(gp->gdir[side]) + fl * cellB + b0 * sizeof(S), rowB, 0};
      return Src{reinterpret_cast<const char*>(M::wall_rows(a)) + ((gp->face0[side] + fl) * nbp + b0) * sizeof(S), 0u, 0};
    };
    const long long fx = cj + (long long)ny * ck, fy = ci + (long long)nx * ck, fz = ci + (long long)nx * cj;
    if constexpr (MAP == 1 || MAP == 3) {
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        cu.x[v] = src(0, v == 0, ci, nx, cellB, fx, 0);
        cu.y[v] = src(1, v == 0, cj, ny, cellB * nx, fy, 0);
        if (DIM == 3) {  // in-plane sets: S_z = 0 counts as from the high side, and mirrors onto itself
          cu.z[v] = src(2, MAP == 3 && v == 0, ck, gp->nz, cellB * nx * ny, fz, MAP == 3 ? (v ? -4 : 4) : 0);
          cu.z[v].mir = 0;
        }
      }
    } else if constexpr (MAP == 2) {
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        cu.x[v] = src(0, (dg == 0) == (v == 0), ci, nx, cellB, fx, dg ? -1 : 1);
        cu.y[v] = src(1, v == 0, cj, ny, cellB * nx, fy, (v ? -1 : 3) - 2 * dg);
        if (DIM == 3) cu.z[v] = src(2, v == 0, ck, gp->nz, cellB * nx * ny, fz, v ? -4 : 4);
      }
    } else {
      cu.x[0] = src(0, dg == 0 || dg == 3, ci, nx, cellB, fx, (dg ^ 1) - dg);
      cu.y[0] = src(1, dg < 2, cj, ny, cellB * nx, fy, 3 - 2 * dg);
      if (DIM == 3)
#pragma unroll
        for (int v = 0; v < 2; ++v) cu.z[v] = src(2, v == 0, ck, gp->nz, cellB * nx * ny, fz, v ? -4 : 4);
    }
    cu.item = item;
    cu.blk = 0;
    cu.r0 = dg;
  };
  auto next_block = [&]() {
    cu.r0 += ROWS;
    if (++cu.blk == nblk) {
      if (cu.item + (int)gridDim.x < a.nitems) setup(cu.item + gridDim.x);
      else cu.on = false;
    }
  };
  // stage step k of the cursor's block into the ring slot at si
  auto issue = [&](auto kc, unsigned si) {
    constexpr int k = decltype(kc)::value;
    if (cu.on) {
      const unsigned r = cu.r0 + DT * k;
      cp16(si, cu.in + (size_t)r * rowB);
      auto up = [&](const Src& s, int shift) -> const char* {
        const char* p = s.base + (size_t)r * s.scale;
        if constexpr (MAP == 1 || MAP == 3) p += shift * s.mir;
        return p;
      };
      constexpr bool one = MAP == 1 || MAP == 3;
      constexpr int q = k & 3;
      constexpr int vx = one ? (q == 1 || q == 2) : (MAP == 2 ? k & 1 : 0);
      constexpr int vy = one ? q >> 1 : (MAP == 2 ? k & 1 : 0);
      constexpr int vz = MAP == 1 ? 0 : (MAP == 3 ? k >> 2 : (MAP == 2 ? k >> 1 : k));
      cp16(si + ostr, up(cu.x[vx], k & 1 ? -1 : 1));
      cp16(si + 2 * ostr, up(cu.y[vy], 3 - 2 * q));
      if (DIM == 3) cp16(si + 3 * ostr, up(cu.z[vz], 0));
    }
    cp_commit();
  };

  int item = blockIdx.x;
  if (item >= a.nitems) return;
  cu.on = true;
  setup(item);
  // the consuming side's cell: address, table class, I0 (read one item ahead)
  long long P;
  int cls;
  bool act;
  double i0[V];
  auto meet = [&](int it, long long& p, int& c, bool& ac, double (&x)[V]) {
    const WorkItem wi = a.items[it];
    ac = slot < wi.cell_count;
    p = a.geoms[wi.geom].cell0 + wi.cell_begin + (ac ? slot : 0);
    c = a.geoms[wi.geom].cls;
#pragma unroll
    for (int v = 0; v < V; v += 2) {
      const double2 t = ld2(a.I0cell + p * nbp + b0 + v);
      x[v] = t.x;
      x[v + 1] = t.y;
    }
  };
  meet(item, P, cls, act, i0);
  unsigned si = ring, sb = ring;
  auto bump = [&](unsigned& s) {
    s += sstr;
    if (s == rend) s = ring;
  };
  auto prologue = [&](auto self, auto jc) -> void {
    constexpr int j = decltype(jc)::value;
    if constexpr (j < kAhead) {
      if (j > 0 && j % RUN == 0) next_block();
      issue(std::integral_constant<int, j % RUN>{}, si);
      bump(si);
      self(self, std::integral_constant<int, j + 1>{});
    }
  };
  prologue(prologue, std::integral_constant<int, 0>{});
  int cur_cls = -1;
  using Coef = typename M::template Coef<DIM>;
  Coef cf = M::template coef<DIM>(a, cls, 0, b0);
  for (;;) {
    if (cls != cur_cls) {  // (block-uniform) table of this cell-size class
      __syncthreads();
      for (int b = threadIdx.x; b < nblk; b += blockDim.x) tabs[b] = M::template tab<DIM>(a, cls, b * ROWS);
      __syncthreads();
      if (cur_cls >= 0) cf = M::template coef<DIM>(a, cls, 0, b0);
      cur_cls = cls;
    }
    const typename M::Cell cell = M::cell(a, ln, i0, b0, P);
    char* out = reinterpret_cast<char*>(a.Iout) + P * cellB + b0 * sizeof(S) + dg * rowB;
    char* bout = M::kStoreB ? reinterpret_cast<char*>(a.Bout) + P * cellB + b0 * sizeof(S) + dg * rowB : nullptr;
    const long long P0 = P;
    const bool act0 = act;
    const bool more = item + (int)gridDim.x < a.nitems;
    item += gridDim.x;
    if (more) meet(item, P, cls, act, i0);
    typename M::Acc acc = M::acc(a, cell);
    for (int blk = 0; blk < nblk; ++blk) {
      const Coef nx = M::template coef<DIM>(a, cur_cls, blk + 1 < nblk ? (blk + 1) * ROWS : 0, b0);
      const auto bk = M::template block<DIM, RUN>(a, ln, cell, cf, tabs[blk], acc);
      auto steps = [&](auto self, auto kc) -> void {
        constexpr int k = decltype(kc)::value;
        if constexpr (k < RUN) {
          constexpr int ck = (k + kAhead) % RUN;
          if (ck == 0) next_block();
          issue(std::integral_constant<int, ck>{}, si);
          bump(si);
          cp_wait<kAhead>();
          M::template step<DIM, k == 0>(a, ln, cell, bk, sb, ostr, out, bout, act0, acc);
          out += DT * rowB;
          if (M::kStoreB) bout += DT * rowB;
          bump(sb);
          self(self, std::integral_constant<int, k + 1>{});
        }
      };
      steps(steps, std::integral_constant<int, 0>{});
      cf = nx;
    }
    double G[V];
    M::finish(a, cell, acc, b0, dg, G);
    if (act0) {
      double eL = 0.0, eP = 0.0;
#pragma unroll
      for (int v = 0; v < V; v += 2) {
        const double2 iv = ld2(a.th.inv_v + b0 + v), bi = ld2(a.th.binv_v + b0 + v);
        eL = fma(G[v + 1], iv.y, fma(G[v], iv.x, eL));
        eP = fma(G[v + 1], bi.y, fma(G[v], bi.x, eP));
      }
      a.Ec[P0 * team + tl] = make_double2(eL, eP);
    }
    if (!more) break;
  }
  cp_wait<0>();
}

template <int DIM, int MAP, class M>
cudaError_t launch_one(const SweepArgs& a, int threads, int grid, cudaStream_t s) {
  const void* f = (const void*)rows_kernel<DIM, MAP, M>;
  const size_t smem = sizeof(typename M::template Tab<DIM>) * (size_t)(a.nd / (Map<MAP>::DT * Map<MAP>::RUN)) + 16 +
                      (size_t)M::template slots<DIM> * (1 + DIM) * threads * 16;
  cudaError_t e = raise_dynamic_smem(f, smem);
  if (e != cudaSuccess) return e;
  if (grid <= 0) {  // persistent: as many CTAs as are resident
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, threads, smem);
    if (e != cudaSuccess) return e;
    grid = std::min(a.nitems, std::max(1, per_sm) * 152);
  }
  rows_kernel<DIM, MAP, M><<<grid, threads, smem, s>>>(a);
  return cudaGetLastError();
}

// The map follows from the set and the directions per team step.
template <class M>
cudaError_t launch(const SweepArgs& a, int dim, int threads, int grid, cudaStream_t s) {
  if (a.dir_group == 4) {
    if (a.dteam != 1) return cudaErrorInvalidValue;
    return dim == 3 ? launch_one<3, 1, M>(a, threads, grid, s) : launch_one<2, 1, M>(a, threads, grid, s);
  }
  if (a.dteam == 1) return dim == 3 ? launch_one<3, 3, M>(a, threads, grid, s) : launch_one<2, 3, M>(a, threads, grid, s);
  if (a.dteam == 2) return dim == 3 ? launch_one<3, 2, M>(a, threads, grid, s) : launch_one<2, 2, M>(a, threads, grid, s);
  if constexpr (M::kFour) {
    if (a.dteam == 4) return dim == 3 ? launch_one<3, 4, M>(a, threads, grid, s) : launch_one<2, 4, M>(a, threads, grid, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace rows
}  // namespace bte
