// sph_fp64_lines.cuh -- the line solves of the FP64 mode on the stored rows
// (sph_fp64.cuh): (I + h D_d) x = r on every line along d, or its transpose (the
// adjoint's), as (1/h I + D_d) x = r/h, so that no row is scaled.
//
// Block lines (p, T, u_d): 3x3-block Thomas from both ends of the line, the two
// sides meeting in the middle: two dependent chains of half the length.
//   top, cells 0 .. h-1 (h = ceil(N/2)):   S_m = B_m - A_m E_{m-1},
//     E_m = S_m^{-1} C_m,  g_m = S_m^{-1} (r_m - A_m g_{m-1}),  x_m = g_m - E_m x_{m+1};
//   bottom, cells N-1 .. h, the roles of A and C swapped.
// At the meeting cells (I - E_o E_p) x_o = g_o - E_o g_p with the partner's
// (E_p, g_p), then each side substitutes outwards.
// A cyclic line keeps its last cell X out: the N = n-1 other cells form a walled
// line whose first and last cells also couple to X (x = y - Z X, three more
// columns H carried through the elimination), and X's own row closes the ring.
//
// Two layouts (one FP64 instruction of a warp takes 64 cycles of its SM quarter
// however many lanes are active, so few lines must still fill every quarter):
//   * Many lines: one lane per line and side, the two sides in two warps of a
//     64-thread block (each with its own blocks' zeros skipped at compile time;
//     97 -> 85 FP64 instructions a cell against both sides in one warp).
//   * Few lines: a line and side takes 4 lanes (8 on a cyclic line), one per
//     column of [E | g | H]; the 3x3 inverse's rows are formed one per lane and
//     exchanged by shuffles.  About 40 FP64 instructions a cell and lane in
//     place of 95, at four times the warps.
// Measured, us per sweep, one lane per side with both sides' union of blocks ->
// these: 32^3 cells (1024 lines a direction, split) 92-101 -> 50-60; cyclic phi
// lines of 32 x 128 x 256 (4096 lines of 256 cells, split) 3930, one lane a line
// with the Woodbury correction, -> 1102.
#pragma once

#include "sph_blk3.cuh"

namespace f64 {

using namespace blk3;

// bits of a double that is zero, infinite or NaN (integer test: FP64 compares
// take the FP64 pipe)
__device__ __forceinline__ bool bad_pivot(double d) {
  const unsigned hi = (unsigned)__double2hiint(d) & 0x7fffffffu;
  return hi >= 0x7ff00000u || (hi | (unsigned)__double2loint(d)) == 0u;
}
// X = S^-1 (adjugate over determinant); a singular S gives NaN and the flag
__device__ __forceinline__ void inverse(const double* S, double* X, int* bad) {
  const double c00 = fma(S[4], S[8], -(S[5] * S[7])), c01 = fma(S[5], S[6], -(S[3] * S[8])),
               c02 = fma(S[3], S[7], -(S[4] * S[6]));
  const double det = fma(S[2], c02, fma(S[1], c01, S[0] * c00));
  double id;
  if (bad_pivot(det)) {
    *bad |= FLAG_SINGULAR;
    id = NAN;
  } else {
    id = 1.0 / det;
  }
  X[0] = c00 * id; X[3] = c01 * id; X[6] = c02 * id;
  X[1] = fma(S[2], S[7], -(S[1] * S[8])) * id;
  X[4] = fma(S[0], S[8], -(S[2] * S[6])) * id;
  X[7] = fma(S[1], S[6], -(S[0] * S[7])) * id;
  X[2] = fma(S[1], S[5], -(S[2] * S[4])) * id;
  X[5] = fma(S[2], S[3], -(S[0] * S[5])) * id;
  X[8] = fma(S[0], S[4], -(S[1] * S[3])) * id;
}

struct LineArgs {
  Geo<double> g;
  Rows rows;
  const double* beta;
  const double* tab;        // Tabs::s[d]
  double ih;                // 1/h, h = tau/2
  CF<double> rhs;
  MF<double> x;             // output increments (update = 0)
  int update;               // 1: uk = base + x
  int norms;                // accumulate the squares of x (update = 1)
  CF<double> base;
  MF<double> uk;
  double* scr;
  int scr_off[3], nl[3], a0[3], nb[3], b0[3];
  double* acc;
  int* flag;
};

template <int D> __device__ __forceinline__ int len(const Geo<double>& g) { return D == 0 ? g.nr : D == 1 ? g.nt : g.np; }

// flat indices of cell m of the line (a, b): centre, its face m + 1 (wrapping on
// a cyclic line), and the table row
template <int D, bool CYC>
__device__ __forceinline__ void cell_idx(const Geo<double>& g, int a, int b, int m, int& ic, int& fx, int& tb) {
  int i, j, k;
  line_pos(D, a, b, m, i, j, k);
  ic = IC(g, i, j, k);
  tb = (i * g.nt + j) * NS;
  fx = face_idx(g, D, D == 0 ? m + 1 : i, D == 1 ? m + 1 : j, D == 2 ? (CYC && m + 1 == g.np ? 0 : m + 1) : k);
}

// The raw values of blocks A, B, C of a cell, then the blocks (with the walls'
// folds): zero p- and T-gradient ghosts, the first face of a walled line is no
// unknown, and its last cell has no face m + 1 (identity row).
struct RawA { double adv, be, vp, vT, wu, K, Dc; };
struct RawB { double be, vp, vT, wp, wu, K, Dc; };
struct RawC { double adv, be, wp, wu, K, Dc; };

template <int D, bool CYC>
struct Cells {
  const LineArgs& S;
  int a, b, n;
  __device__ __forceinline__ Cells(const LineArgs& s, int a_, int b_) : S(s), a(a_), b(b_), n(len<D>(s.g)) {}
  __device__ __forceinline__ bool face(int m) const { return CYC || m < n - 1; }

  __device__ __forceinline__ void load(int m, RawA& r) const {
    int ic, fx, tb;
    cell_idx<D, CYC>(S.g, a, b, m, ic, fx, tb);
    const double* p = S.rows.c[D] + ic;
    const long nc = S.rows.nc;
    r.adv = p[0]; r.vp = p[nc]; r.vT = p[3 * nc];
    r.be = S.beta[ic];
    r.wu = face(m) ? S.rows.f[D][S.rows.nf[D] + fx] : 0.0;
    r.K = S.tab[tb + S_K0]; r.Dc = S.tab[tb + S_D0];
  }
  __device__ __forceinline__ void load(int m, RawB& r) const {
    int ic, fx, tb;
    cell_idx<D, CYC>(S.g, a, b, m, ic, fx, tb);
    const double* p = S.rows.c[D] + ic;
    const long nc = S.rows.nc, nf = S.rows.nf[D];
    r.vp = p[2 * nc]; r.vT = p[4 * nc];
    r.be = S.beta[ic];
    r.wp = face(m) ? S.rows.f[D][fx] : 0.0;
    r.wu = face(m) ? S.rows.f[D][2 * nf + fx] : 0.0;
    r.K = S.tab[tb + S_KS]; r.Dc = S.tab[tb + S_DS];
  }
  __device__ __forceinline__ void load(int m, RawC& r) const {
    int ic, fx, tb;
    cell_idx<D, CYC>(S.g, a, b, m, ic, fx, tb);
    const long nf = S.rows.nf[D];
    r.adv = S.rows.c[D][ic];
    r.be = S.beta[ic];
    r.wp = face(m) ? S.rows.f[D][fx] : 0.0;
    r.wu = face(m) ? S.rows.f[D][3 * nf + fx] : 0.0;
    r.K = S.tab[tb + S_K1]; r.Dc = S.tab[tb + S_D1];
  }
  __device__ __forceinline__ void form(const RawA& r, double* A) const {
    A[0] = -r.adv; A[1] = r.Dc; A[2] = r.vp;
    A[4] = fma(r.be, r.K, -r.adv); A[5] = r.vT;
    A[8] = r.wu;
  }
  __device__ __forceinline__ void form(const RawC& r, double* C) const {
    C[0] = r.adv; C[1] = r.Dc;
    C[4] = fma(r.be, r.K, r.adv);
    C[6] = r.wp; C[8] = r.wu;
  }
  // B of cell m; fold: the p- and T-columns of the block beyond the wall
  __device__ __forceinline__ void form(int m, const RawB& r, double* B) const {
    B[0] = S.ih; B[1] = r.Dc; B[2] = r.vp;
    B[4] = fma(r.be, r.K, S.ih); B[5] = r.vT;
    B[6] = -r.wp; B[8] = r.wu + S.ih;
    if (!CYC && (m == 0 || m == n - 1)) {
      if (m == 0) {
        RawA w;
        double A[9];
        load(m, w);
        form(w, A);
        B[0] += A[0]; B[1] += A[1]; B[4] += A[4];
      }
      if (m == n - 1) {
        RawC w;
        double C[9];
        load(m, w);
        form(w, C);
        B[0] += C[0]; B[1] += C[1]; B[4] += C[4];
        B[2] = 0.0; B[5] = 0.0;
      }
    }
  }
  // the right-hand side of cell m, unscaled (r[2] = 0 where it has no face)
  __device__ __forceinline__ void load_rhs(int m, double* r) const {
    int ic, fx, tb;
    cell_idx<D, CYC>(S.g, a, b, m, ic, fx, tb);
    r[0] = S.rhs.f[0][ic];
    r[1] = S.rhs.f[4][ic];
    r[2] = face(m) ? S.rhs.f[1 + D][fx] : 0.0;
  }
  __device__ __forceinline__ int wrap(int m) const { return m < 0 ? m + n : m >= n ? m - n : m; }
};

template <typename Acc>
__device__ __forceinline__ void emit(const LineArgs& S, int f, int idx, double v, Acc& ss, int* bad) {
  if (!S.update) {
    S.x.f[f][idx] = v;
    return;
  }
  if ((((unsigned)__double2hiint(v)) & 0x7ff00000u) == 0x7ff00000u) *bad |= FLAG_NONFINITE;
  S.uk.f[f][idx] = S.base.f[f][idx] + v;
  if (S.norms) ss.add(f, v);
}
__device__ __forceinline__ void emit_wall(const LineArgs& S, int f, int idx) {
  if (!S.update) S.x.f[f][idx] = 0.0;
  else S.uk.f[f][idx] = S.base.f[f][idx];
}
// x of cell m of a block line, and the wall faces next to a walled line's ends
template <int D, bool CYC, typename Acc>
__device__ __forceinline__ void emit_cell(const LineArgs& S, int a, int b, int m, const double* x, Acc& ss, int* bad) {
  int ic, fx, tb;
  cell_idx<D, CYC>(S.g, a, b, m, ic, fx, tb);
  emit(S, 0, ic, x[0], ss, bad);
  emit(S, 4, ic, x[1], ss, bad);
  if (CYC || m < len<D>(S.g) - 1) {
    emit(S, 1 + D, fx, x[2], ss, bad);
  } else {
    emit_wall(S, 1 + D, fx);
    int i, j, k;
    line_pos(D, a, b, 0, i, j, k);
    emit_wall(S, 1 + D, face_idx(S.g, D, i, j, k));
  }
}

// Elimination of one side of a block line (SIDE 0 from the first cell, 1 from the
// last) over cnt cells; writes (E, g[, H]) of every cell but the last to the
// scratch and leaves the last cell's.
template <int D, bool CYC, bool TR, int SIDE>
__device__ __forceinline__ void eliminate(const LineArgs& S, const Cells<D, CYC>& Z, int N, int cnt, int line, bool valid,
                                          double* E, double* g, double* H, int* bad) {
  // the block towards the eliminated cell (L) and towards the next (U): A and C
  // of the cell itself, or of the neighbours' transposes
  constexpr bool LA = SIDE == 0;       // L is A (of this row) from the top, C from the bottom
  constexpr unsigned ML = TR ? mt(LA ? M_C : M_A) : (LA ? M_A : M_C), MU = TR ? mt(LA ? M_A : M_C) : (LA ? M_C : M_A);
  const int nl = S.nl[0];
  constexpr int W = CYC ? 21 : 12;
  double* scr = S.scr + S.scr_off[0];
  RawA ra;
  RawB rb;
  RawC rc;
  double r[3];
  const int n = Z.n;
  // the cells whose A and C enter row m: m itself, or for the transpose A of
  // m + 1 and C of m - 1 (none past the ends of a walled line)
  auto fetch = [&](int m) {
    const int ma = TR ? m + 1 : m, mc = TR ? m - 1 : m;
    if (CYC || ma < n) Z.load(Z.wrap(ma), ra);
    if (CYC || mc >= 0) Z.load(Z.wrap(mc), rc);
    Z.load(m, rb);
    Z.load_rhs(m, r);
  };
  fetch(SIDE ? N - 1 : 0);
  for (int s = 0; s < cnt; s++) {
    const int m = SIDE ? N - 1 - s : s;
    double A[9], B[9], C[9], y[3];
    Z.form(ra, A);
    Z.form(rc, C);
    Z.form(m, rb, B);
#pragma unroll
    for (int q = 0; q < 3; q++) y[q] = r[q] * S.ih;
    if (s + 1 < cnt) fetch(SIDE ? m - 1 : m + 1);
    double Am[9], Cm[9], Bm[9];        // A, C, B of this row (transposed)
    if (TR) {
#pragma unroll
      for (int q = 0; q < 9; q++) {
        const int tq = (q % 3) * 3 + q / 3;
        Am[q] = C[tq]; Cm[q] = A[tq]; Bm[q] = B[tq];
      }
    } else {
#pragma unroll
      for (int q = 0; q < 9; q++) { Am[q] = A[q]; Cm[q] = C[q]; Bm[q] = B[q]; }
    }
    const double* L = LA ? Am : Cm;
    const double* U = LA ? Cm : Am;
    double Sm[9], Hs[9];
    constexpr unsigned MB = TR ? mt(M_B) : M_B;
#pragma unroll
    for (int q = 0; q < 9; q++) Sm[q] = (MB >> q & 1) ? Bm[q] : 0.0;
    if (s > 0) {
      sub_mul<ML, 3>(L, E, Sm);
      sub_mul<ML, 1>(L, g, y);
    }
    if (CYC) {
      if (s == 0) {
#pragma unroll
        for (int q = 0; q < 9; q++) Hs[q] = (ML >> q & 1) ? L[q] : 0.0;   // couples to X
      } else {
#pragma unroll
        for (int q = 0; q < 9; q++) Hs[q] = 0.0;
        sub_mul<ML, 3>(L, H, Hs);
      }
    }
    double Si[9];
    inverse(Sm, Si, bad);
    mul_sparse<MU>(Si, U, E);
    mv(Si, y, g);
    if (CYC) mul_sparse<0x1ff>(Si, Hs, H);
    if (s + 1 < cnt && valid) {
      double* sp = scr + m * W * nl + line;
#pragma unroll
      for (int q = 0; q < 9; q++) sp[q * nl] = E[q];
#pragma unroll
      for (int q = 0; q < 3; q++) sp[(9 + q) * nl] = g[q];
      if (CYC)
#pragma unroll
        for (int q = 0; q < 9; q++) sp[(12 + q) * nl] = H[q];
    }
  }
}

constexpr int NEX = 21;   // doubles a lane exchanges with the other side's warp

// One block line per lane; warp 0 of the block the top side, warp 1 the bottom.
template <int D, bool CYC, bool TR>
__device__ __forceinline__ void block_line(const LineArgs& S, double (*ex)[32], int line, bool valid, int a, int b,
                                           int side, SqSum<double>& ss, int* bad) {
  const Cells<D, CYC> Z(S, a, b);
  const int n = Z.n, N = CYC ? n - 1 : n, h = (N + 1) / 2, cnt = side ? N - h : h;
  const int nl = S.nl[0], lane = threadIdx.x & 31;
  constexpr int W = CYC ? 21 : 12;
  double* scr = S.scr + S.scr_off[0];
  double E[9], g[3], H[9];
  if (side == 0) eliminate<D, CYC, TR, 0>(S, Z, N, cnt, line, valid, E, g, H, bad);
  else eliminate<D, CYC, TR, 1>(S, Z, N, cnt, line, valid, E, g, H, bad);
  // the meeting cells (N >= 2: a cell on either side)
  {
    double* mine = &ex[side * NEX][lane];
#pragma unroll
    for (int q = 0; q < 9; q++) mine[q * 32] = E[q];
#pragma unroll
    for (int q = 0; q < 3; q++) mine[(9 + q) * 32] = g[q];
    if (CYC)
#pragma unroll
      for (int q = 0; q < 9; q++) mine[(12 + q) * 32] = H[q];
  }
  __syncthreads();
  double x[3], Zc[9];
  {
    const double* other = &ex[(1 - side) * NEX][lane];
    double M[9], Mi[9], v[3], Ep[9];
#pragma unroll
    for (int q = 0; q < 9; q++) { Ep[q] = other[q * 32]; M[q] = q % 4 == 0 ? 1.0 : 0.0; }
    sub_mul<0x1ff, 3>(E, Ep, M);
    double gp[3];
#pragma unroll
    for (int q = 0; q < 3; q++) { gp[q] = other[(9 + q) * 32]; v[q] = g[q]; }
    sub_mul<0x1ff, 1>(E, gp, v);
    inverse(M, Mi, bad);
    mv(Mi, v, x);
    if (CYC) {
      double Hp[9], Hv[9];
#pragma unroll
      for (int q = 0; q < 9; q++) { Hp[q] = other[(12 + q) * 32]; Hv[q] = H[q]; }
      sub_mul<0x1ff, 3>(E, Hp, Hv);
      mul_sparse<0x1ff>(Mi, Hv, Zc);
    }
  }
  // substitution outwards; the factors of the next cell out are loaded before
  // the current one is stored.  Cyclic lines keep y and Z in the factors' place.
  auto cell = [&](int s) { return side ? N - 1 - s : s; };
  double En[9], gn[3], Hn[9];
  auto fetch = [&](int s) {
    const double* sp = scr + cell(s) * W * nl + line;
#pragma unroll
    for (int q = 0; q < 9; q++) En[q] = sp[q * nl];
#pragma unroll
    for (int q = 0; q < 3; q++) gn[q] = sp[(9 + q) * nl];
    if (CYC)
#pragma unroll
      for (int q = 0; q < 9; q++) Hn[q] = sp[(12 + q) * nl];
  };
  if (cnt >= 2) fetch(cnt - 2);
  for (int s = cnt - 1; s >= 0; s--) {
    const int m = cell(s);
    if (s < cnt - 1) {
      double e[9], v[3], w[9];
#pragma unroll
      for (int q = 0; q < 9; q++) { e[q] = En[q]; if (CYC) w[q] = Hn[q]; }
#pragma unroll
      for (int q = 0; q < 3; q++) v[q] = gn[q];
      if (s >= 1) fetch(s - 1);
      sub_mul<0x1ff, 1>(e, x, v);
#pragma unroll
      for (int q = 0; q < 3; q++) x[q] = v[q];
      if (CYC) {
        sub_mul<0x1ff, 3>(e, Zc, w);
#pragma unroll
        for (int q = 0; q < 9; q++) Zc[q] = w[q];
      }
    }
    if (CYC) {
      if (valid) {
        double* sp = scr + m * W * nl + line;
#pragma unroll
        for (int q = 0; q < 9; q++) sp[q * nl] = Zc[q];
#pragma unroll
        for (int q = 0; q < 3; q++) sp[(9 + q) * nl] = x[q];
      }
    } else if (valid) {
      emit_cell<D, CYC>(S, a, b, m, x, ss, bad);
    }
  }
  if (CYC) {
    // the ring's last cell: (B - C Z_0 - A Z_{N-1}) X = r - C y_0 - A y_{N-1}
    // (the blocks of the transpose swap as in the elimination)
    __syncthreads();
    double* mine = &ex[side * NEX][lane];
#pragma unroll
    for (int q = 0; q < 9; q++) mine[q * 32] = Zc[q];
#pragma unroll
    for (int q = 0; q < 3; q++) mine[(9 + q) * 32] = x[q];
    __syncthreads();
    double A[9], B[9], C[9], X[3], v[3], r[3];
    {
      RawA ra;
      RawB rb;
      RawC rc;
      Z.load(TR ? 0 : n - 1, ra);
      Z.load(TR ? n - 2 : n - 1, rc);
      Z.load(n - 1, rb);
      Z.load_rhs(n - 1, r);
      double t[9];
      Z.form(ra, t);
      const double z = 0.0;
#pragma unroll
      for (int q = 0; q < 9; q++) {
        const double w = (M_A >> q & 1) ? t[q] : z;
        if (TR) C[(q % 3) * 3 + q / 3] = w; else A[q] = w;
      }
      Z.form(rc, t);
#pragma unroll
      for (int q = 0; q < 9; q++) {
        const double w = (M_C >> q & 1) ? t[q] : z;
        if (TR) A[(q % 3) * 3 + q / 3] = w; else C[q] = w;
      }
      Z.form(n - 1, rb, t);
#pragma unroll
      for (int q = 0; q < 9; q++) {
        const double w = (M_B >> q & 1) ? t[q] : z;
        B[TR ? (q % 3) * 3 + q / 3 : q] = w;
      }
    }
#pragma unroll
    for (int q = 0; q < 3; q++) v[q] = r[q] * S.ih;
    // y and Z of the line's first cell (the top side's) and its last (the bottom's)
    double Y[9], yv[3];
#pragma unroll
    for (int e = 0; e < 2; e++) {
      const double* src = &ex[e * NEX][lane];
#pragma unroll
      for (int q = 0; q < 9; q++) Y[q] = src[q * 32];
#pragma unroll
      for (int q = 0; q < 3; q++) yv[q] = src[(9 + q) * 32];
      sub_mul<0x1ff, 3>(e ? A : C, Y, B);
      sub_mul<0x1ff, 1>(e ? A : C, yv, v);
    }
    double Bi[9];
    inverse(B, Bi, bad);
    mv(Bi, v, X);
    if (valid) {
      for (int s = 0; s < cnt; s++) {
        const int m = cell(s);
        const double* sp = scr + m * W * nl + line;
        double e[9], v3[3];
#pragma unroll
        for (int q = 0; q < 9; q++) e[q] = sp[q * nl];
#pragma unroll
        for (int q = 0; q < 3; q++) v3[q] = sp[(9 + q) * nl];
        sub_mul<0x1ff, 1>(e, X, v3);
        emit_cell<D, CYC>(S, a, b, m, v3, ss, bad);
      }
      if (side == 0) emit_cell<D, CYC>(S, a, b, n - 1, X, ss, bad);
    }
  }
}

// ------------------------------------------------------------ scalar lines

// coefficients of row m of a transverse scalar line, (1/h I + D) scaled, with
// the no-slip folds of a walled line
template <int D, int CC, bool CYC>
struct SCells {
  const LineArgs& S;
  int a, b, n;
  __device__ __forceinline__ SCells(const LineArgs& s, int a_, int b_) : S(s), a(a_), b(b_), n(len<D>(s.g)) {}
  __device__ __forceinline__ int idx(int m) const {
    int i, j, k;
    line_pos(D, a, b, m, i, j, k);
    return face_idx(S.g, CC, i, j, k);
  }
  __device__ __forceinline__ const double* row(int m) const {
    return S.rows.s[CC] + 3 * trans_slot(CC, D) * S.rows.nf[CC] + idx(m);
  }
  __device__ __forceinline__ double w(int m, int q) const { return row(m)[q * S.rows.nf[CC]]; }
  __device__ __forceinline__ int wrap(int m) const { return m < 0 ? m + n : m >= n ? m - n : m; }
};

template <int D, int CC, typename Acc>
__device__ __forceinline__ void emit_scalar(const LineArgs& S, int a, int b, int m, double v, Acc& ss, int* bad) {
  const Geo<double>& g = S.g;
  int i, j, k;
  line_pos(D, a, b, m, i, j, k);
  emit(S, 1 + CC, face_idx(g, CC, i, j, k), v, ss, bad);
  const int lo = CC == 0 ? i == 1 : CC == 1 ? j == 1 : (k == 1 && !g.per);
  const int hi = CC == 0 ? i == g.nr - 1 : CC == 1 ? j == g.nt - 1 : (k == g.np - 1 && !g.per);
  if (lo) emit_wall(S, 1 + CC, face_idx(g, CC, CC == 0 ? 0 : i, CC == 1 ? 0 : j, CC == 2 ? 0 : k));
  if (hi) emit_wall(S, 1 + CC, face_idx(g, CC, CC == 0 ? g.nr : i, CC == 1 ? g.nt : j, CC == 2 ? g.np : k));
}

// One transverse scalar line, one lane per side, the same way.
template <int D, int KIND, bool CYC, bool TR>
__device__ __forceinline__ void scalar_line(const LineArgs& S, double (*ex)[32], int line, bool valid, int a, int b,
                                            int side, SqSum<double>& ss, int* bad) {
  constexpr int CC = trans_comp(D, KIND);
  const SCells<D, CC, CYC> Z(S, a, b);
  const int n = Z.n, N = CYC ? n - 1 : n, h = (N + 1) / 2, cnt = side ? N - h : h;
  const int nl = S.nl[KIND], lane = threadIdx.x & 31;
  double* scr = S.scr + S.scr_off[KIND];
  const double* rhs = S.rhs.f[1 + CC];
  auto cell = [&](int s) { return side ? N - 1 - s : s; };
  // the row (below, diagonal, above) of cell m; the transpose takes its
  // neighbours' weights towards it
  double wn[3], rn = 0.0;
  auto fetch = [&](int m) {
    wn[1] = Z.w(m, 1);
    wn[0] = TR ? (CYC || m > 0 ? Z.w(Z.wrap(m - 1), 2) : 0.0) : Z.w(m, 0);
    wn[2] = TR ? (CYC || m < n - 1 ? Z.w(Z.wrap(m + 1), 0) : 0.0) : Z.w(m, 2);
    rn = rhs[Z.idx(m)];
  };
  double e = 0.0, gy = 0.0, hz = 0.0;
  fetch(cell(0));
  for (int s = 0; s < cnt; s++) {
    const int m = cell(s);
    double am = wn[0], bm = wn[1] + S.ih, cm = wn[2], r = rn * S.ih;
    if (s + 1 < cnt) fetch(cell(s + 1));
    if (!CYC && m == 0) { bm -= TR ? Z.w(0, 0) : am; am = 0.0; }
    if (!CYC && m == n - 1) { bm -= TR ? Z.w(n - 1, 2) : cm; cm = 0.0; }
    const double lo = side ? cm : am, up = side ? am : cm;
    const double den = s ? fma(-lo, e, bm) : bm;
    if (bad_pivot(den)) *bad |= FLAG_SINGULAR;
    const double id = 1.0 / den;
    gy = (s ? fma(-lo, gy, r) : r) * id;
    if (CYC) hz = (s ? -lo * hz : lo) * id;
    e = up * id;
    if (s + 1 < cnt && valid) {
      double* sp = scr + m * 3 * nl + line;
      sp[0] = e;
      sp[nl] = gy;
      if (CYC) sp[2 * nl] = hz;
    }
  }
  {
    double* mine = &ex[side * NEX][lane];
    mine[0] = e; mine[32] = gy; mine[64] = hz;
  }
  __syncthreads();
  double x, z = 0.0;
  {
    const double* o = &ex[(1 - side) * NEX][lane];
    const double den = fma(-e, o[0], 1.0), id = 1.0 / den;
    if (bad_pivot(den)) *bad |= FLAG_SINGULAR;
    x = fma(-e, o[32], gy) * id;
    if (CYC) z = fma(-e, o[64], hz) * id;
  }
  double en = 0.0, gn = 0.0, hn = 0.0;
  auto fback = [&](int s) {
    const double* sp = scr + cell(s) * 3 * nl + line;
    en = sp[0]; gn = sp[nl];
    if (CYC) hn = sp[2 * nl];
  };
  if (cnt >= 2) fback(cnt - 2);
  for (int s = cnt - 1; s >= 0; s--) {
    const int m = cell(s);
    if (s < cnt - 1) {
      const double e_ = en, g_ = gn, h_ = hn;
      if (s >= 1) fback(s - 1);
      x = fma(-e_, x, g_);
      if (CYC) z = fma(-e_, z, h_);
    }
    if (CYC) {
      if (valid) { scr[m * 3 * nl + line] = z; scr[m * 3 * nl + nl + line] = x; }
    } else if (valid) {
      emit_scalar<D, CC>(S, a, b, m, x, ss, bad);
    }
  }
  if (CYC) {
    __syncthreads();
    double* mine = &ex[side * NEX][lane];
    mine[0] = z; mine[32] = x;
    __syncthreads();
    const double* o0 = &ex[0][lane];
    const double* o1 = &ex[NEX][lane];
    const double am = TR ? Z.w(n - 2, 2) : Z.w(n - 1, 0), cm = TR ? Z.w(0, 0) : Z.w(n - 1, 2);
    const double den = fma(-cm, o0[0], fma(-am, o1[0], Z.w(n - 1, 1) + S.ih));
    if (bad_pivot(den)) *bad |= FLAG_SINGULAR;
    const double X = fma(-cm, o0[32], fma(-am, o1[32], rhs[Z.idx(n - 1)] * S.ih)) * (1.0 / den);
    if (valid) {
      for (int s = 0; s < cnt; s++) {
        const int m = cell(s);
        const double* sp = scr + m * 3 * nl + line;
        emit_scalar<D, CC>(S, a, b, m, fma(-sp[0], X, sp[nl]), ss, bad);
      }
      if (side == 0) emit_scalar<D, CC>(S, a, b, n - 1, X, ss, bad);
    }
  }
}

__device__ __forceinline__ void add_norms(const LineArgs& S, const SqSum<double>& ss) {
  if (!S.update || !S.norms) return;
  for (int f = 0; f < 5; f++) {
    const double v = ss.warp_total(f);
    if ((threadIdx.x & 31) == 0 && v != 0.0) atomicAdd(S.acc + f, v);
  }
}

// ----------------------------------------------------- few lines: lane split

// this lane's value of element e of the blocks' column or of lane src's
__device__ __forceinline__ double get(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }

// Solve S w = u for the lane's own column, S's column r in lane g0 + r of the
// group (t there), u in every lane; w into v.  Lane r forms row r of the adjugate
// (the cross product of the other two columns).
__device__ __forceinline__ void split_solve(const double* t, const double* u, int g0, int q, double* v, int* bad) {
  const int r = q % 3, r1 = (r + 1) % 3, r2 = (r + 2) % 3;
  double p[3], s[3], row[3];
#pragma unroll
  for (int e = 0; e < 3; e++) { p[e] = get(t[e], g0 + r1); s[e] = get(t[e], g0 + r2); }
  row[0] = fma(p[1], s[2], -(p[2] * s[1]));
  row[1] = fma(p[2], s[0], -(p[0] * s[2]));
  row[2] = fma(p[0], s[1], -(p[1] * s[0]));
  double det = get(fma(t[2], row[2], fma(t[1], row[1], t[0] * row[0])), g0);
  double adj[9];
#pragma unroll
  for (int e = 0; e < 9; e++) adj[e] = get(row[e % 3], g0 + e / 3);
  double id;
  if (bad_pivot(det)) {
    *bad |= FLAG_SINGULAR;
    id = NAN;
  } else {
    id = 1.0 / det;
  }
  double w[3];
  mv(adj, u, w);
#pragma unroll
  for (int e = 0; e < 3; e++) v[e] = w[e] * id;
}

// A block line in the lanes [g0, g0 + LS) of a warp (top side) and those 16
// further on (bottom side); this lane is lane q of its side.  LS = 4: columns
// of E, then g; 8 (cyclic): E, g, the columns of H, one lane idle.
template <int D, bool CYC, bool TR>
__device__ __forceinline__ void block_line_split(const LineArgs& S, int line, bool valid, int a, int b, int side, int g0,
                                                 int q, SqSum<double>& ss, int* bad) {
  const Cells<D, CYC> Z(S, a, b);
  const int n = Z.n, N = CYC ? n - 1 : n, h = (N + 1) / 2, cnt = side ? N - h : h;
  const int nl = S.nl[0];
  constexpr int W = CYC ? 21 : 12, LS = CYC ? 8 : 4;
  double* scr = S.scr + S.scr_off[0];
  auto cell = [&](int s) { return side ? N - 1 - s : s; };
  RawA ra;
  RawB rb;
  RawC rc;
  double r[3];
  auto fetch = [&](int m) {
    const int ma = TR ? m + 1 : m, mc = TR ? m - 1 : m;
    if (CYC || ma < n) Z.load(Z.wrap(ma), ra);
    if (CYC || mc >= 0) Z.load(Z.wrap(mc), rc);
    Z.load(m, rb);
    Z.load_rhs(m, r);
  };
  // element (e) of the lane's column of a 3x3 block with nonzero entries MASK
  auto column = [&](const double* X, unsigned mask, int c, double* o) {
#pragma unroll
    for (int e = 0; e < 3; e++) {
      o[e] = 0.0;
#pragma unroll
      for (int z = 0; z < 3; z++)
        if ((mask >> (TR ? 3 * z + e : 3 * e + z) & 1) && c == z) o[e] = X[TR ? 3 * z + e : 3 * e + z];
    }
  };
  double v[3] = {0.0, 0.0, 0.0};
  // both sides run the same instructions for the same count (the longer, top
  // side's); a side that has finished repeats its last cell without a store
  // and keeps its factors
  fetch(cell(0));
  for (int s = 0; s < h; s++) {
    const bool live = s < cnt;
    const int m = cell(live ? s : cnt - 1);
    double A[9], B[9], C[9], t[3], u[3];
    Z.form(ra, A);
    Z.form(rc, C);
    Z.form(m, rb, B);
    double y[3];
#pragma unroll
    for (int e = 0; e < 3; e++) y[e] = r[e] * S.ih;
    if (s + 1 < cnt) fetch(cell(s + 1));
    // L and U of this row: A and C from the top, swapped from the bottom; the
    // transpose takes C^T and A^T
    constexpr unsigned MU2 = M_A | M_C;
    double L[9], U[9];
#pragma unroll
    for (int e = 0; e < 9; e++) {
      const double za = (M_A >> e & 1) ? A[e] : 0.0, zc = (M_C >> e & 1) ? C[e] : 0.0;
      L[e] = (side != 0) == TR ? za : zc;
      U[e] = (side != 0) == TR ? zc : za;
    }
    double bc[3], uc[3];
    column(B, M_B, q, bc);
    column(U, MU2, q, uc);
#pragma unroll
    for (int e = 0; e < 3; e++) t[e] = q < 3 ? bc[e] : q == 3 ? y[e] : 0.0;
    if (s > 0) {
#pragma unroll
      for (int e = 0; e < 3; e++)
#pragma unroll
        for (int z = 0; z < 3; z++)
          if (MU2 >> (TR ? 3 * z + e : 3 * e + z) & 1) t[e] = fma(-L[TR ? 3 * z + e : 3 * e + z], v[z], t[e]);
    } else if (CYC) {
      double lc[3];
      column(L, MU2, q - 4, lc);
#pragma unroll
      for (int e = 0; e < 3; e++) if (q > 3) t[e] = lc[e];
    }
#pragma unroll
    for (int e = 0; e < 3; e++) u[e] = q < 3 ? uc[e] : t[e];
    double w[3];
    int sing = 0;
    split_solve(t, u, g0, q, w, &sing);
    if (live) {
      *bad |= sing;
#pragma unroll
      for (int e = 0; e < 3; e++) v[e] = w[e];
    }
    if (s + 1 < cnt && valid && q < (CYC ? 7 : 4)) {
      double* sp = scr + m * W * nl + line;
#pragma unroll
      for (int e = 0; e < 3; e++) sp[(q < 3 ? 3 * e + q : q == 3 ? 9 + e : 12 + 3 * e + q - 4) * nl] = v[e];
    }
  }
  // the meeting cells: (I - E_o E_p) [x | Z] = [g_o | H_o] - E_o [g_p | H_p]
  double xv[3];
  {
    double t[3], Eo[9];
#pragma unroll
    for (int e = 0; e < 3; e++) {
      t[e] = q < 3 ? (e == q ? 1.0 : 0.0) : v[e];
#pragma unroll
      for (int z = 0; z < 3; z++) Eo[3 * e + z] = get(v[e], g0 + z);
    }
    double vp[3];
#pragma unroll
    for (int e = 0; e < 3; e++) vp[e] = __shfl_xor_sync(0xffffffffu, v[e], 16);
    sub_mul<0x1ff, 1>(Eo, vp, t);
    split_solve(t, t, g0, q, xv, bad);   // lanes 3 and up: x, the columns of Z
  }
  if (!CYC) {
    // substitution outwards: lane e < 3 takes unknown e
    double x[3];
#pragma unroll
    for (int e = 0; e < 3; e++) x[e] = get(xv[e], g0 + 3);
    const int e = q < 3 ? q : 2;
    double En[3], gn = 0.0;
    auto fb = [&](int s) {
      const double* sp = scr + cell(s) * W * nl + line;
#pragma unroll
      for (int z = 0; z < 3; z++) En[z] = sp[(3 * e + z) * nl];
      gn = sp[(9 + e) * nl];
    };
    __syncwarp();   // the factors were stored by the lanes of their columns
    if (cnt >= 2) fb(cnt - 2);
    for (int s = h - 1; s >= 0; s--) {
      const bool live = s < cnt;
      if (s < cnt - 1) {
        const double e0 = En[0], e1 = En[1], e2 = En[2], gg = gn;
        if (s >= 1) fb(s - 1);
        const double mine = fma(-e2, x[2], fma(-e1, x[1], fma(-e0, x[0], gg)));
        x[0] = e == 0 ? mine : x[0]; x[1] = e == 1 ? mine : x[1]; x[2] = e == 2 ? mine : x[2];
      }
      const double mine = e == 0 ? x[0] : e == 1 ? x[1] : x[2];
#pragma unroll
      for (int z = 0; z < 3; z++) x[z] = get(mine, g0 + z);
      if (live && valid && q < 3) {
        const int m = cell(s);
        int ic, fx, tb;
        cell_idx<D, CYC>(S.g, a, b, m, ic, fx, tb);
        if (e < 2) {
          emit(S, e == 0 ? 0 : 4, ic, mine, ss, bad);
        } else if (m < n - 1) {
          emit(S, 1 + D, fx, mine, ss, bad);
        } else {
          emit_wall(S, 1 + D, fx);
          int i, j, k;
          line_pos(D, a, b, 0, i, j, k);
          emit_wall(S, 1 + D, face_idx(S.g, D, i, j, k));
        }
      }
    }
    return;
  }
  // cyclic: y and the columns of Z outwards, one column per lane (3 and up),
  // kept in the factors' place (a slot is read and rewritten by one lane only)
  __syncwarp();
  for (int s = cnt - 1; s >= 0; s--) {
    double* sp = scr + cell(s) * W * nl + line;
    double E[9], nv[3];
    if (s < cnt - 1) {
#pragma unroll
      for (int e = 0; e < 9; e++) E[e] = sp[e * nl];
#pragma unroll
      for (int e = 0; e < 3; e++) nv[e] = sp[(q == 3 ? 9 + e : 12 + 3 * e + (q > 3 ? (q < 7 ? q - 4 : 2) : 0)) * nl];
      sub_mul<0x1ff, 1>(E, xv, nv);
#pragma unroll
      for (int e = 0; e < 3; e++) xv[e] = nv[e];
    }
    if (valid && q >= 3 && q < 7)
#pragma unroll
      for (int e = 0; e < 3; e++) sp[(q == 3 ? 9 + e : 12 + 3 * e + q - 4) * nl] = xv[e];
  }
  __syncwarp();
  double X[3];
  {
    double A[9], B[9], C[9], t[9], y[3], v3[3];
    RawA la;
    RawB lb;
    RawC lc;
    Z.load(TR ? 0 : n - 1, la);
    Z.load(TR ? n - 2 : n - 1, lc);
    Z.load(n - 1, lb);
    Z.load_rhs(n - 1, y);
    Z.form(la, t);
#pragma unroll
    for (int e = 0; e < 9; e++) {
      const double w = (M_A >> e & 1) ? t[e] : 0.0;
      if (TR) C[(e % 3) * 3 + e / 3] = w; else A[e] = w;
    }
    Z.form(lc, t);
#pragma unroll
    for (int e = 0; e < 9; e++) {
      const double w = (M_C >> e & 1) ? t[e] : 0.0;
      if (TR) A[(e % 3) * 3 + e / 3] = w; else C[e] = w;
    }
    Z.form(n - 1, lb, t);
#pragma unroll
    for (int e = 0; e < 9; e++) B[TR ? (e % 3) * 3 + e / 3 : e] = (M_B >> e & 1) ? t[e] : 0.0;
#pragma unroll
    for (int e = 0; e < 3; e++) v3[e] = y[e] * S.ih;
#pragma unroll
    for (int w = 0; w < 2; w++) {
      const double* sp = scr + (w ? N - 1 : 0) * W * nl + line;
      double Zc[9], yv[3];
#pragma unroll
      for (int e = 0; e < 9; e++) Zc[e] = sp[(12 + e) * nl];
#pragma unroll
      for (int e = 0; e < 3; e++) yv[e] = sp[(9 + e) * nl];
      sub_mul<0x1ff, 3>(w ? A : C, Zc, B);
      sub_mul<0x1ff, 1>(w ? A : C, yv, v3);
    }
    double Bi[9];
    inverse(B, Bi, bad);
    mv(Bi, v3, X);
  }
  if (valid) {
    for (int m = side * LS + q; m < N; m += 2 * LS) {
      const double* sp = scr + m * W * nl + line;
      double Zc[9], x3[3];
#pragma unroll
      for (int e = 0; e < 9; e++) Zc[e] = sp[(12 + e) * nl];
#pragma unroll
      for (int e = 0; e < 3; e++) x3[e] = sp[(9 + e) * nl];
      sub_mul<0x1ff, 1>(Zc, X, x3);
      emit_cell<D, CYC>(S, a, b, m, x3, ss, bad);
    }
    if (side == 0 && q == 0) emit_cell<D, CYC>(S, a, b, n - 1, X, ss, bad);
  }
}

// Many lines: 32 lines of one kind per block of two warps.  SPLIT (few lines):
// the block lines take 4 (8 on cyclic lines) lanes a side, 8 (4) lines a block.
// Kind 0 (the block lines, the longest) comes first in block order.
template <int D, bool CYC, bool TR, bool SPLIT>
__global__ void __launch_bounds__(64) k_lines(const __grid_constant__ LineArgs S) {
  __shared__ double ex[2 * NEX][32];
  const int kind = blockIdx.y, nl = S.nl[kind], lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int LS = CYC ? 8 : 4, LW = 16 / LS;   // lanes a side, lines a warp (SPLIT)
  const bool split = SPLIT && kind == 0;
  const int per = split ? 2 * LW : 32;
  if ((int)blockIdx.x * per >= nl) return;  // no line of this kind left
  const int side = split ? lane >> 4 : warp;
  const int l0 = blockIdx.x * per + (split ? warp * LW + (lane & 15) / LS : lane);
  const bool valid = l0 < nl;
  const int line = valid ? l0 : nl - 1;
  const int a = line / S.nb[kind] + S.a0[kind], b = line % S.nb[kind] + S.b0[kind];
  SqSum<double> ss;
  int bad = 0;
  if (kind == 0) {
    if constexpr (SPLIT)
      block_line_split<D, CYC, TR>(S, line, valid, a, b, side, lane - lane % LS, lane % LS, ss, &bad);
    else
      block_line<D, CYC, TR>(S, ex, line, valid, a, b, side, ss, &bad);
  } else if (kind == 1) {
    scalar_line<D, 1, CYC, TR>(S, ex, line, valid, a, b, side, ss, &bad);
  } else {
    scalar_line<D, 2, CYC, TR>(S, ex, line, valid, a, b, side, ss, &bad);
  }
  if (bad && valid) atomicOr(S.flag, bad);
  add_norms(S, ss);
}

}  // namespace f64
