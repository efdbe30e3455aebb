// sph_fp64_tab.cuh -- the tables and stored rows the FP64 mode's kernels share
// (sph_fp64.cuh, sph_fp64_lines.cuh), as the host and the device see them.
#pragma once
#include <stddef.h>

namespace f64 {

// ------------------------------------------------------------------ tables
// Per centre (i, j).  "lap" weights: L0, L1 multiply (f_{m-1} - f_m) and
// (f_{m+1} - f_m) in the geometric Laplacian along a direction, G0, G1 the two
// faces' velocities in the d-part of div u.
enum {
  C_IR, C_HIR, C_QIR,                    // 1/r, 1/(2r), 1/(4r)
  C_MT, C_HMT, C_QMT,                    // 1/(r dtheta) and its half and quarter
  C_MP, C_HMP, C_QMP, C_MP2,             // 1/(r sin dphi), half, quarter, square
  C_G00, C_G01, C_G10, C_G11,            // divergence weights along r, theta (along phi: C_MP)
  C_E00, C_E01, C_E10, C_E11,            // divergence weights less the plain difference's (+-1/dr, +-C_MT)
  C_L00, C_L01, C_L10, C_L11,            // Laplacian weights along r, theta (along phi: C_MP2)
  C_COT, C_COT2, C_COTIR, C_HCOTIR,      // cot, 2 cot, cot/r, cot/(2r)
  C_IT,                                  // 1/(Rg T_ref)
  // rows of u_phi (its faces share the centres' i and j); the factor 1/rho =
  // 2 / (rho_0 + rho_1) enters as 1/(rho_0 + rho_1), the 2 is in the table
  P_WP, P_F, P_F2,                       // pressure gradient; normal row: off-diagonal, diagonal
  P_R0, P_R1, P_RS,                      // row along r
  P_T0, P_T1, P_TS,                      // row along theta
  P_V, P_D, P_UR, P_UT,                  // explicit viscous terms
  P_OC, P_OS,                            // Coriolis
  NC
};
// per r-face (i = 1..nr-1 used) and theta index
enum { R_WP, R_F0, R_F1, R_F2, R_T0, R_T1, R_TS, R_QT, R_P, R_P2, R_QP, R_QIR, R_V, R_Q0, R_Q1, R_OM, R_E, R_GE, NR };
// per radial index and theta-face (j = 1..nt-1 used)
enum { T_WP, T_HADV, T_F0, T_F1, T_F2, T_R0, T_R1, T_RS, T_P, T_P2, T_QP, T_HIR, T_C, T_V, T_D, T_D0, T_D1, T_UR, T_OM,
       NT };
// per centre and direction, for the assembly of the line rows: conduction
// weights of the T-row per unit beta (below, above, diagonal) and of the p-row
enum { S_K0, S_K1, S_KS, S_D0, S_D1, S_DS, NS };

struct Tabs {
  double *c, *r, *t, *s[3];
};
inline size_t tabs_doubles(int nr, int nt) {
  return (size_t)nr * nt * (NC + 3 * NS) + (size_t)(nr + 1) * nt * NR + (size_t)nr * (nt + 1) * NT;
}
inline Tabs tabs_of(double* p, int nr, int nt) {
  Tabs T;
  T.c = p; p += (size_t)nr * nt * NC;
  T.r = p; p += (size_t)(nr + 1) * nt * NR;
  T.t = p; p += (size_t)nr * (nt + 1) * NT;
  for (int d = 0; d < 3; d++) { T.s[d] = p; p += (size_t)nr * nt * NS; }
  return T;
}

// The line rows of D_r, D_theta, D_phi at Ubar that the right-hand side forms
// and the sweeps read (45 doubles a cell with beta from the coefficients):
//   c[d]: 5 planes over the centres: the advection weight, and the couplings of
//         the p- and T-row to u_d on the cell's two faces (p0, p1, T0, T1);
//   f[d]: 4 planes over the d-faces: the normal-velocity row (p, u below, u, u above);
//   s[c]: 6 planes over the c-faces: the rows of velocity component c along its
//         two transverse directions in increasing order (3 weights each).
struct Rows {
  double* c[3];
  double* f[3];
  double* s[3];
  long nc, nf[3];  // centres; faces of each kind
};
constexpr int ROWS_C = 5, ROWS_F = 4, ROWS_S = 6;
constexpr int ADJ_PLANES = 8;   // coefficient planes whose cotangents the adjoint accumulates
// slot of direction d among the transverse directions of component cc
__host__ __device__ constexpr int trans_slot(int cc, int d) { return d < cc ? d : d - 1; }

}  // namespace f64
