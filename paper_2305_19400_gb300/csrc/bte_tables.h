// bte_tables.h -- host table builders (bte_tables.cpp).
#pragma once
#include <vector>

namespace bte {

void gauss_legendre(int n, double* x, double* w);
int build_dirs_inplane(int n, std::vector<double>& S, std::vector<double>& w, std::vector<int>& refl);
int build_dirs_polar_azim(int nt, int np, std::vector<double>& S, std::vector<double>& w, std::vector<int>& refl);
void build_thermo(int nb, int nbp, int ng, const double* wlo, const double* whi, const double* vg, const double* beta,
                  const double* deg, double Wtot, std::vector<double>& node_c, std::vector<double>& node_C,
                  std::vector<double>& a_p, std::vector<double>& a_L, std::vector<double>& inv_v,
                  std::vector<double>& beta_p);
// hbar omega_max / (32 k_B) of the nb bands, omega_max the highest node's.
double model_knee(const std::vector<double>& node_c, int nb, int ng);

void build_coef(int dim, const double delta[3], int nd, const double* S, const double* w, int nb, int nbp,
                const double* vg, const double* beta, double dt, int explicit_scheme, double* out);

// Tables of the factored double-float sweep (bte_rows.cuh) for one class,
// the implicit update divided through by v_b (v_b > 0 on every real band):
// I' = W I^n + R (sum_ax c_ax,d u_ax + (beta_b / v_b) I0),
// R = 1 / (1 / (v_b dt) + beta_b / v_b + sum_ax c_ax,d),  W = R / (v_b dt).
// dirc[nd][3][2] c_ax,d = |S_d,ax|/(w_d Delta_ax) as double-float pairs (h, l);
// band[nbp] beta_b/v_b in the pair layout of bte_ff.cuh (per two bands h_b, h_b+1,
// l_b, l_b+1; padding bands 0); RW[nd][nbp] the same, per two bands R's pairs, then W's.
// R is the double-float pair nearest the reciprocal of a denominator formed exactly
// (double-double) from the stored pairs themselves, W the pair nearest
// 1 - R (beta_b / v_b + sum c) of the stored R, so that a uniform field is a fixed point
// of the update to the pairs' resolution; below 1/4, where that difference would lose
// relative accuracy, the pair nearest R / (v_b dt).  Only the first of each group of directions
// (internal_order) is formed: its rows serve the group.
void build_ff_factored(int dim, const double delta[3], int nd, int group, const double* S, const double* w, int nb, int nbp,
                       const double* vg, const double* beta, double dt, float* RW, float* dirc, float* band);

void build_pq(int dim, const double delta[3], int nd, const double* S, const double* w, int nb, int nbp,
              const double* vg, const double* beta, double dt, int explicit_scheme, float* P, float* Q, float* dirc);

// Internal order of a direction set: the directions that differ only in the
// signs of S stand together, so that one set of sweep coefficients serves
// consecutive rows.  Groups of four (in-plane sets) by the signs of (S_x, S_y):
// (+,+), (-,+), (-,-), (+,-); of eight (polar x azimuthal sets): the four with
// S_z > 0, then their mirror images across z.  Row r of a group so reflects
// across x to r ^ 1, across y to r ^ 3, across z to r ^ 4.  Returns the
// caller's index of every internal direction and permutes S, w, refl in place.
std::vector<int> internal_order(std::vector<double>& S, std::vector<double>& w, std::vector<int>& refl, int group);

}  // namespace bte
