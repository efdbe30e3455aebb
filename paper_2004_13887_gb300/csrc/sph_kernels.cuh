// sph_kernels.cuh -- device code of the scheme's stages (Section 2.2, eqs.
// chapter3mainsd, splitting2, spl1-spl3) that every part of the library shares: the
// averaging kernel, the one-thread-per-line block and scalar line solvers, and what
// the other line solvers take from them.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "sph_device.cuh"

namespace sph {}
using namespace sph;

#define FLAG_NONFINITE 1
#define FLAG_SINGULAR 2

// ------------------------------------------------------------------ kernels

// Ubar = (U^n + U^k)/2 for the five fields in one launch (blockIdx.y = field),
// two values per thread per pass (16-byte loads, 8-byte stores in FP32).
// Ubar = (a + b)/2 and D = b - a (a = U^n, b = U^{n+1,k}; D is the -(U^k - U^n)
// part of the right-hand side, so that stage reads neither FP64 state).  In
// FP32 mode both are formed as pairs on the FP32 pipe: o = Ubar rounded, and
// for the velocity components lo[f] (when not null) = the remainder, so that
// div(Ubar) can be formed to ~48 bits; D is rounded once from the exact pair.
// same = 1 (the first iteration of a step, U^k = U^n): b is not read and D is
// not written (the right-hand side does not read it then); Ubar = a is split
// into its pair directly, which gives the same bits as (a + a)/2 in pairs.
template <typename R>
struct AvgArgs { const double* a[5]; const double* b[5]; R* o[5]; R* lo[5]; R* d[5]; long n[5]; int same; };

template <typename R>
__device__ __forceinline__ void avg1(const double x, const double y, R* o, R* lo, R* d, long t) {
  if constexpr (sizeof(R) == sizeof(double)) {
    o[t] = (R)(0.5 * (x + y));
    d[t] = (R)(y - x);
  } else {
    float xh, xl, yh, yl, h, l;
    d2ff(x, xh, xl);
    d2ff(y, yh, yl);
    ff_add(xh, xl, yh, yl, h, l);
    o[t] = 0.5f * h;
    if (lo) lo[t] = 0.5f * l;
    ff_sub(yh, yl, xh, xl, h, l);
    d[t] = h + l;
  }
}

template <typename R>
__device__ __forceinline__ void split1(const double x, R* o, R* lo, long t) {
  if constexpr (sizeof(R) == sizeof(double)) {
    o[t] = (R)x;
  } else {
    float h, l;
    d2ff(x, h, l);
    o[t] = h;
    if (lo) lo[t] = l;
  }
}

template <typename R>
__global__ void k_avg(AvgArgs<R> A) {
  const int f = blockIdx.y;
  const double* __restrict__ a = A.a[f];
  const double* __restrict__ b = A.b[f];
  R* __restrict__ o = A.o[f];
  R* __restrict__ lo = A.lo[f];
  R* __restrict__ d = A.d[f];
  long n = A.n[f], n2 = n >> 1;
  long s = (long)gridDim.x * blockDim.x;
  if (A.same) {
    for (long t = (long)blockIdx.x * blockDim.x + threadIdx.x; t < n2; t += s) {
      double2 x = reinterpret_cast<const double2*>(a)[t];
      split1(x.x, o, lo, 2 * t);
      split1(x.y, o, lo, 2 * t + 1);
    }
    if ((n & 1) && blockIdx.x == 0 && threadIdx.x == 0) split1(a[n - 1], o, lo, n - 1);
    return;
  }
  for (long t = (long)blockIdx.x * blockDim.x + threadIdx.x; t < n2; t += s) {
    double2 x = reinterpret_cast<const double2*>(a)[t], y = reinterpret_cast<const double2*>(b)[t];
    avg1(x.x, y.x, o, lo, d, 2 * t);
    avg1(x.y, y.y, o, lo, d, 2 * t + 1);
  }
  if ((n & 1) && blockIdx.x == 0 && threadIdx.x == 0) avg1(a[n - 1], b[n - 1], o, lo, d, n - 1);
}

template <typename R>
__global__ void k_cvt(long n, const R* __restrict__ a, double* __restrict__ o) {
  long s = (long)gridDim.x * blockDim.x;
  for (long t = (long)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += s) o[t] = (double)a[t];
}

template <typename R>
__global__ void k_cvt_in(long n, const double* __restrict__ a, R* __restrict__ o) {
  long s = (long)gridDim.x * blockDim.x;
  for (long t = (long)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += s) o[t] = (R)a[t];
}

// The stencil kernels run on tiles of TK x TJ x TI points (phi fastest; 128
// threads; the shape is set per context, sph_set_tile).  A block takes the
// fast path when its whole tile has its +-2 neighbourhood in r and theta
// inside the grid (a uniform choice).  The default is one r row of 1, 2 or 4 theta
// rows by the length of a phi row; the ensemble's autotuner picks the shape per grid.
template <typename G>
__device__ __forceinline__ bool tile_inner_at(const G& g, int i0, int j0, int ti, int tj) {
  return inner_ij(g, i0, j0) && inner_ij(g, i0 + ti - 1, j0 + tj - 1);
}
template <typename G>
__device__ __forceinline__ bool tile_inner(const G& g) {
  return tile_inner_at(g, blockIdx.z * blockDim.z, blockIdx.y * blockDim.y, (int)blockDim.z, (int)blockDim.y);
}
// grid of tiles of tj x ti rows of phi points (128 / (tj ti) each) over an
// nk x nj x ni index box
static dim3 tile_grid_of(int tj, int ti, int nk, int nj, int ni) {
  int tk = 128 / (tj * ti);
  return dim3((nk + tk - 1) / tk, (nj + tj - 1) / tj, (ni + ti - 1) / ti);
}
#define tile_grid(nk, nj, ni) tile_grid_of(c->tile_j, c->tile_i, nk, nj, ni)
#define TILE_BLOCK dim3(128 / (c->tile_j * c->tile_i), c->tile_j, c->tile_i)

// ------------------------------------------------------------ line solvers

template <typename R>
__device__ __forceinline__ bool inv3(const R* S, R* I) {
  R c00 = S[4] * S[8] - S[5] * S[7];
  R c01 = S[5] * S[6] - S[3] * S[8];
  R c02 = S[3] * S[7] - S[4] * S[6];
  R det = S[0] * c00 + S[1] * c01 + S[2] * c02;
  if (det == R(0) || !isfinite(det)) return false;
  R id = sdiv(R(1), det);
  I[0] = c00 * id; I[3] = c01 * id; I[6] = c02 * id;
  I[1] = (S[2] * S[7] - S[1] * S[8]) * id;
  I[4] = (S[0] * S[8] - S[2] * S[6]) * id;
  I[7] = (S[1] * S[6] - S[0] * S[7]) * id;
  I[2] = (S[1] * S[5] - S[2] * S[4]) * id;
  I[5] = (S[2] * S[3] - S[0] * S[5]) * id;
  I[8] = (S[0] * S[4] - S[1] * S[3]) * id;
  return true;
}

// position of cell m on the line (a, b) along d
__device__ __forceinline__ void line_pos(int d, int a, int b, int m, int& i, int& j, int& k) {
  if (d == 0) { i = m; j = a; k = b; }
  else if (d == 1) { i = a; j = m; k = b; }
  else { i = a; j = b; k = m; }
}

template <typename G>
__device__ __forceinline__ int face_idx(const G& g, int d, int i, int j, int k) {
  return d == 0 ? IRf(g, i, j, k) : d == 1 ? ITf(g, i, j, k) : IPf(g, i, j, k);
}

// Assemble block m of (I + h D_d) on a line from the loaded centre values (cq)
// and, when the line has face m+1 (m < n-1 or cyclic), the face values fq at
// face coordinates (fi, fj); h = tau/2.
template <typename R>
__device__ __forceinline__ void assemble_pts(const Geo<R>& g, const Par& P, const CPt<R>& cq, const FPt<R>& fq, int d,
                                             int n, int cyc, int m, int i, int j, int fi, int fj, R h, R* A, R* B,
                                             R* C) {
  RowC<R> w;
#pragma unroll
  for (int q = 0; q < 9; q++) { A[q] = R(0); B[q] = R(0); C[q] = R(0); }
  row_cw(g, P, cq, d, 0, i, j, w);
  A[0] = h * w.wp[0]; A[1] = h * w.wT[0]; A[2] = h * (w.a * w.gd[0] + w.wv[0]);
  B[0] = h * w.wp[1]; B[1] = h * w.wT[1]; B[2] = h * (w.a * w.gd[1] + w.wv[1]);
  C[0] = h * w.wp[2]; C[1] = h * w.wT[2];
  row_cw(g, P, cq, d, 1, i, j, w);
  A[4] = h * w.wT[0]; A[5] = h * (w.a * w.gd[0] + w.wv[0]);
  B[4] = h * w.wT[1]; B[5] = h * (w.a * w.gd[1] + w.wv[1]);
  C[4] = h * w.wT[2];
  if (m < n - 1 || cyc) {
    R fp[2], fu[3];
    row_fw(g, P, fq, d, fi, fj, fp, fu);
    A[8] = h * fu[0];
    B[6] = h * fp[0]; B[8] = h * fu[1];
    C[6] = h * fp[1]; C[8] = h * fu[2];
  }
  B[0] += R(1); B[4] += R(1); B[8] += R(1);
  if (!cyc) {
    if (m == 0) {
      B[0] += A[0]; B[1] += A[1]; B[3] += A[3]; B[4] += A[4];
#pragma unroll
      for (int q = 0; q < 9; q++) A[q] = R(0);
    }
    if (m == n - 1) {
      B[0] += C[0]; B[1] += C[1]; B[3] += C[3]; B[4] += C[4];
#pragma unroll
      for (int q = 0; q < 9; q++) C[q] = R(0);
      B[2] = R(0); B[5] = R(0);
      A[8] = R(0); B[6] = R(0); B[7] = R(0); B[8] = R(1);
    }
  }
}

// face m+1 of cell m on a line along d (wrapping to 0 on a cyclic line; the wall
// face n of a walled one)
__device__ __forceinline__ void next_face(int d, int n, int cyc, int m, int i, int j, int k, int& fi, int& fj, int& fk) {
  fi = i; fj = j; fk = k;
  if (d == 0) fi = m + 1; else if (d == 1) fj = m + 1; else fk = (cyc && m + 1 == n) ? 0 : m + 1;
}

// Assemble block m of (I + h D_d) on a line; h = tau/2.
template <typename R>
__device__ void assemble_block(const Geo<R>& g, const Par& P, const Coef<R>& c, const CF<R>& ub, int d, int n, int cyc,
                               int m, int i, int j, int k, R h, R* A, R* B, R* C) {
  CPt<R> cq = load_c(c, d, IC(g, i, j, k));
  FPt<R> fq = {R(1), R(1), R(0)};
  int fi, fj, fk;
  next_face(d, n, cyc, m, i, j, k, fi, fj, fk);
  if (m < n - 1 || cyc) fq = load_f(g, c, ub.f[1 + d], d, fi, fj, fk);
  assemble_pts(g, P, cq, fq, d, n, cyc, m, i, j, fi, fj, h, A, B, C);
}

template <typename R>
struct SweepArgs {
  Geo<R> g; Par P; Coef<R> c; CF<R> ub;
  int d; R h;
  CF<R> rhs;              // right-hand side fields
  MF<R> x;                // output increments (mode 0)
  int update;             // mode 1: uk = base + x (FP64), accumulate norms
  CF<double> base; MF<double> uk;
  R* scr;                 // scratch
  int scr_off[3];         // offsets of the three kinds
  int nl[3];              // lines per kind
  int a0[3], nb[3], b0[3];
  double* acc;            // 5 sums of squares (mode 1, when norms is set)
  int norms;
  int* flag;
  // FP32 lines: the tables of the direction's block and scalar lines
  // (sph_lines2.cuh) and the constants their rows use
  const float *tb, *ts[2];
  float hgm, hgm1, hvp2, hmu2, gm1, iRg;
};

// Per-thread sums of squares of the increments, per field (the iteration
// residual).  FP64 mode: plain FP64 sums.  FP32 mode: each sum is an
// unevaluated pair hi + lo (the square's rounding error by FMA, the addition's
// by two_sum), ~48 bits like an FP64 sum, on the FP32 pipe; the warp's pairs are
// combined the same way and reach the FP64 accumulator as hi + lo.
template <typename R>
struct SqSum {
  R h[5] = {0, 0, 0, 0, 0};
  __device__ __forceinline__ void add(int f, R r) { h[f] += r * r; }
  __device__ __forceinline__ double warp_total(int f) const {
    R v = h[f];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return f2d(v);
  }
};
template <>
struct SqSum<float> {
  float h[5] = {0, 0, 0, 0, 0}, l[5] = {0, 0, 0, 0, 0};
  __device__ __forceinline__ void add(int f, float r) {
    float p = r * r, e = fmaf(r, r, -p), s, t;
    two_sum(h[f], p, s, t);
    h[f] = s;
    l[f] += t + e;
  }
  __device__ __forceinline__ double warp_total(int f) const {
    float hv = h[f], lv = l[f];
    for (int o = 16; o > 0; o >>= 1) {
      float ho = __shfl_down_sync(0xffffffffu, hv, o), lo = __shfl_down_sync(0xffffffffu, lv, o), s, t;
      two_sum(hv, ho, s, t);
      hv = s;
      lv += lo + t;
    }
    return f2d(hv) + f2d(lv);
  }
};
// The same with plain FP32 partial sums per thread (a few squares each: the
// scalar line kernels, whose 48-register budget has no room for the pairs) and
// the pair combination from the warp reduction on.
struct SqSumLite {
  float h[5] = {0, 0, 0, 0, 0};
  __device__ __forceinline__ void add(int f, float r) { h[f] = fmaf(r, r, h[f]); }
  __device__ __forceinline__ double warp_total(int f) const {
    float hv = h[f], lv = 0.f;
    for (int o = 16; o > 0; o >>= 1) {
      float ho = __shfl_down_sync(0xffffffffu, hv, o), lo = __shfl_down_sync(0xffffffffu, lv, o), s, t;
      two_sum(hv, ho, s, t);
      hv = s;
      lv += lo + t;
    }
    return f2d(hv) + f2d(lv);
  }
};

// store a value of field f at flat index idx: x (mode 0) or uk = base + v (mode
// 1, the one FP64 add per value of the mixed path), with the square of v summed
template <typename R, typename V, typename Acc>
__device__ __forceinline__ void put(const SweepArgs<R>& A, int f, int idx, V v, Acc& ss, int* bad) {
  if (!A.update) {
    A.x.f[f][idx] = (R)v;
  } else {
    double nv = A.base.f[f][idx] + f2d(v);
    if (!isfinite(v)) *bad |= FLAG_NONFINITE;  // the state was finite; only a non-finite increment spoils it
    A.uk.f[f][idx] = nv;
    if (A.norms) ss.add(f, (R)v);
  }
}
// the update-mode store with the FP64 state value already loaded
template <typename R, typename V, typename Acc>
__device__ __forceinline__ void put_upd(const SweepArgs<R>& A, int f, int idx, double base, V v, Acc& ss, int* bad) {
  if (!isfinite(v)) *bad |= FLAG_NONFINITE;
  A.uk.f[f][idx] = base + f2d(v);
  if (A.norms) ss.add(f, (R)v);
}
// wall face of field f: x = 0, or uk = base (mode 1)
template <typename R>
__device__ __forceinline__ void put_wall(const SweepArgs<R>& A, int f, int idx) {
  if (!A.update) A.x.f[f][idx] = R(0);
  else A.uk.f[f][idx] = A.base.f[f][idx];
}

// Blocks of row m of the transposed line matrix: (M^T)_{m,m-1} = C_{m-1}^T,
// (M^T)_{m,m} = B_m^T, (M^T)_{m,m+1} = A_{m+1}^T, wrapping on a cyclic line and
// zero past the ends of a walled one (the adjoint's transposed line solves).
template <typename R>
__device__ __forceinline__ void transposed_blocks(const SweepArgs<R>& S, int d, int n, int cyc, int a, int b, int m,
                                                  R* A, R* B, R* C) {
  R X[9], Y[9], Z[9];
  int i, j, k;
  line_pos(d, a, b, m, i, j, k);
  assemble_block(S.g, S.P, S.c, S.ub, d, n, cyc, m, i, j, k, S.h, X, Y, Z);
#pragma unroll
  for (int r = 0; r < 3; r++)
#pragma unroll
    for (int q = 0; q < 3; q++) B[r * 3 + q] = Y[q * 3 + r];
  int mp = m - 1, mn = m + 1;
  if (cyc) { mp = mp < 0 ? n - 1 : mp; mn = mn == n ? 0 : mn; }
#pragma unroll
  for (int q = 0; q < 9; q++) { A[q] = R(0); C[q] = R(0); }
  if (mp >= 0) {
    line_pos(d, a, b, mp, i, j, k);
    assemble_block(S.g, S.P, S.c, S.ub, d, n, cyc, mp, i, j, k, S.h, X, Y, Z);
#pragma unroll
    for (int r = 0; r < 3; r++)
#pragma unroll
      for (int q = 0; q < 3; q++) A[r * 3 + q] = Z[q * 3 + r];
  }
  if (mn < n) {
    line_pos(d, a, b, mn, i, j, k);
    assemble_block(S.g, S.P, S.c, S.ub, d, n, cyc, mn, i, j, k, S.h, X, Y, Z);
#pragma unroll
    for (int r = 0; r < 3; r++)
#pragma unroll
      for (int q = 0; q < 3; q++) C[r * 3 + q] = X[q * 3 + r];
  }
}

// One block line along D: solve (I + h D_D) x = rhs (TR: its transpose) by
// block Thomas, Woodbury-corrected on a cyclic line.
template <typename R, int D, bool TR = false>
__device__ void block_line(const SweepArgs<R>& S, int line, int a, int b, SqSum<R>& ss, int* bad) {
  const Geo<R>& g = S.g;
  constexpr int d = D;
  int n = d == 0 ? g.nr : d == 1 ? g.nt : g.np;
  int cyc = (d == 2 && g.per);
  int nl = S.nl[0];
  R* scr = S.scr + S.scr_off[0];
  const int W = cyc ? 21 : 12;  // C' (9) + d' (3 per right-hand side)
  const int NR = cyc ? 4 : 1;
  R Cp[9], dp[12];
  R GiA[9];                     // cyclic: Gam^{-1} A_0
  // The inputs of cell m + 1 (its centre coefficients, the face values of its
  // row, its right-hand side) are loaded before cell m is eliminated, so that
  // their memory latency overlaps the elimination (the forward pass).
  CPt<R> cqn;
  FPt<R> fqn;
  R r0n = R(0), r4n = R(0), run = R(0);
  auto fetch = [&](int m) {
    int i, j, k, fi, fj, fk;
    line_pos(d, a, b, m, i, j, k);
    const int ic = IC(g, i, j, k);
    cqn = load_c(S.c, d, ic);
    fqn = {R(1), R(1), R(0)};
    run = R(0);
    if (m < n - 1 || cyc) {
      next_face(d, n, cyc, m, i, j, k, fi, fj, fk);
      fqn = load_f(g, S.c, S.ub.f[1 + d], d, fi, fj, fk);
      run = S.rhs.f[1 + d][face_idx(g, d, fi, fj, fk)];
    }
    r0n = S.rhs.f[0][ic];
    r4n = S.rhs.f[4][ic];
  };
  if constexpr (!TR) fetch(0);
  for (int m = 0; m < n; m++) {
    int i, j, k;
    line_pos(d, a, b, m, i, j, k);
    R A[9], B[9], C[9];
    R rr[12];
    if constexpr (TR) {
      transposed_blocks(S, d, n, cyc, a, b, m, A, B, C);
      int ic = IC(g, i, j, k);
      rr[0] = S.rhs.f[0][ic];
      rr[NR] = S.rhs.f[4][ic];
      R ru = R(0);
      if (m < n - 1 || cyc) {
        int fi = i, fj = j, fk = k;
        if (d == 0) fi = m + 1; else if (d == 1) fj = m + 1; else fk = (m + 1 == n) ? 0 : m + 1;
        ru = S.rhs.f[1 + d][face_idx(g, d, fi, fj, fk)];
      }
      rr[2 * NR] = ru;
    } else {
      const CPt<R> cq = cqn;
      const FPt<R> fq = fqn;
      rr[0] = r0n;
      rr[NR] = r4n;
      rr[2 * NR] = run;
      if (m + 1 < n) fetch(m + 1);
      int fi, fj, fk;
      next_face(d, n, cyc, m, i, j, k, fi, fj, fk);
      assemble_pts(g, S.P, cq, fq, d, n, cyc, m, i, j, fi, fj, S.h, A, B, C);
    }
    if (cyc) {
      // right-hand-side columns 1..3 of U = [Gam; 0; ..; C_{n-1}]
      for (int r = 0; r < 3; r++)
        for (int q = 0; q < 3; q++) rr[r * NR + 1 + q] = R(0);
      if (m == 0) {
        R Gam[9], Gi[9];
        for (int q = 0; q < 9; q++) Gam[q] = -B[q];
        if (!inv3(Gam, Gi)) { *bad |= FLAG_SINGULAR; return; }
        for (int r = 0; r < 3; r++)
          for (int q = 0; q < 3; q++) GiA[r * 3 + q] = Gi[r * 3] * A[q] + Gi[r * 3 + 1] * A[3 + q] + Gi[r * 3 + 2] * A[6 + q];
        for (int q = 0; q < 9; q++) B[q] -= Gam[q];
        for (int r = 0; r < 3; r++)
          for (int q = 0; q < 3; q++) rr[r * NR + 1 + q] = Gam[r * 3 + q];
      }
      if (m == n - 1) {
        for (int r = 0; r < 3; r++)
          for (int q = 0; q < 3; q++) {
            B[r * 3 + q] -= C[r * 3] * GiA[q] + C[r * 3 + 1] * GiA[3 + q] + C[r * 3 + 2] * GiA[6 + q];
            rr[r * NR + 1 + q] = C[r * 3 + q];
          }
      }
    }
    // S = B - A C'_{m-1};  y = rr - A d'_{m-1}
    R Sm[9], y[12];
    if (m == 0) {
      for (int q = 0; q < 9; q++) Sm[q] = B[q];
      for (int q = 0; q < 3 * NR; q++) y[q] = rr[q];
    } else {
      for (int r = 0; r < 3; r++) {
        for (int q = 0; q < 3; q++)
          Sm[r * 3 + q] = B[r * 3 + q] - (A[r * 3] * Cp[q] + A[r * 3 + 1] * Cp[3 + q] + A[r * 3 + 2] * Cp[6 + q]);
        for (int q = 0; q < NR; q++)
          y[r * NR + q] = rr[r * NR + q] - (A[r * 3] * dp[q] + A[r * 3 + 1] * dp[NR + q] + A[r * 3 + 2] * dp[2 * NR + q]);
      }
    }
    R Si[9];
    if (!inv3(Sm, Si)) { *bad |= FLAG_SINGULAR; return; }
    for (int r = 0; r < 3; r++) {
      for (int q = 0; q < 3; q++)
        Cp[r * 3 + q] = Si[r * 3] * C[q] + Si[r * 3 + 1] * C[3 + q] + Si[r * 3 + 2] * C[6 + q];
      for (int q = 0; q < NR; q++)
        dp[r * NR + q] = Si[r * 3] * y[q] + Si[r * 3 + 1] * y[NR + q] + Si[r * 3 + 2] * y[2 * NR + q];
    }
    if (m < n - 1) {
      R* s = scr + m * W * nl + line;
      for (int q = 0; q < 9; q++) s[q * nl] = Cp[q];
      for (int q = 0; q < 3 * NR; q++) s[(9 + q) * nl] = dp[q];
    }
  }
  // back substitution, all NR columns; the factors of cell m - 1 are loaded
  // before cell m is substituted
  R xs[12];
  for (int q = 0; q < 3 * NR; q++) xs[q] = dp[q];
  R x0[12];
  R Cn[9], dn[12];
  if (n >= 2) {
    const R* s = scr + (n - 2) * W * nl + line;
    for (int q = 0; q < 9; q++) Cn[q] = s[q * nl];
    for (int q = 0; q < 3 * NR; q++) dn[q] = s[(9 + q) * nl];
  }
  for (int m = n - 1; m >= 0; m--) {
    if (m < n - 1) {
      R C_[9], d_[12];
      for (int q = 0; q < 9; q++) C_[q] = Cn[q];
      for (int q = 0; q < 3 * NR; q++) d_[q] = dn[q];
      if (m >= 1) {
        const R* s = scr + (m - 1) * W * nl + line;
        for (int q = 0; q < 9; q++) Cn[q] = s[q * nl];
        for (int q = 0; q < 3 * NR; q++) dn[q] = s[(9 + q) * nl];
      }
      R xn[12];
      for (int r = 0; r < 3; r++)
        for (int q = 0; q < NR; q++)
          xn[r * NR + q] = d_[r * NR + q] - (C_[r * 3] * xs[q] + C_[r * 3 + 1] * xs[NR + q] + C_[r * 3 + 2] * xs[2 * NR + q]);
      for (int q = 0; q < 3 * NR; q++) xs[q] = xn[q];
    }
    if (!cyc) {
      int i, j, k;
      line_pos(d, a, b, m, i, j, k);
      int ic = IC(g, i, j, k);
      put(S, 0, ic, xs[0], ss, bad);
      put(S, 4, ic, xs[1], ss, bad);
      if (m < n - 1) {
        int fi = i, fj = j, fk = k;
        if (d == 0) fi = m + 1; else if (d == 1) fj = m + 1; else fk = m + 1;
        put(S, 1 + d, face_idx(g, d, fi, fj, fk), xs[2], ss, bad);
      } else {
        int fi = i, fj = j, fk = k;
        if (d == 0) fi = n; else if (d == 1) fj = n; else fk = n;
        put_wall(S, 1 + d, face_idx(g, d, fi, fj, fk));
        int gi = i, gj = j, gk = k;
        if (d == 0) gi = 0; else if (d == 1) gj = 0; else gk = 0;
        put_wall(S, 1 + d, face_idx(g, d, gi, gj, gk));
      }
    } else {
      // keep x (all columns) in the d'-slots for the Woodbury combination
      R* s = scr + m * W * nl + line;
      for (int q = 0; q < 3 * NR; q++) s[(9 + q) * nl] = xs[q];
      if (m == 0) for (int q = 0; q < 12; q++) x0[q] = xs[q];
    }
  }
  if (cyc) {
    // V^T y = y_0 + GiA y_{n-1};  V^T Z = Z_0 + GiA Z_{n-1};  f = (I + V^T Z)^{-1} V^T y  (FP64)
    const R* sl = scr + (n - 1) * W * nl + line;
    double xl[12], vy[3], vz[9], vi[9], fcor[3];
    for (int q = 0; q < 12; q++) xl[q] = (double)sl[(9 + q) * nl];
    for (int r = 0; r < 3; r++) {
      vy[r] = (double)x0[r * 4] + (double)GiA[r * 3] * xl[0] + (double)GiA[r * 3 + 1] * xl[4] + (double)GiA[r * 3 + 2] * xl[8];
      for (int q = 0; q < 3; q++)
        vz[r * 3 + q] = (double)x0[r * 4 + 1 + q] + (double)GiA[r * 3] * xl[1 + q] + (double)GiA[r * 3 + 1] * xl[5 + q]
                      + (double)GiA[r * 3 + 2] * xl[9 + q] + (r == q ? 1.0 : 0.0);
    }
    if (!inv3(vz, vi)) { *bad |= FLAG_SINGULAR; return; }
    for (int r = 0; r < 3; r++) fcor[r] = vi[r * 3] * vy[0] + vi[r * 3 + 1] * vy[1] + vi[r * 3 + 2] * vy[2];
    for (int m = 0; m < n; m++) {
      const R* s = scr + m * W * nl + line;
      double xv[3];
      for (int r = 0; r < 3; r++) {
        xv[r] = (double)s[(9 + r * 4) * nl];
        for (int q = 0; q < 3; q++) xv[r] -= (double)s[(9 + r * 4 + 1 + q) * nl] * fcor[q];
      }
      int i, j, k;
      line_pos(d, a, b, m, i, j, k);
      int ic = IC(g, i, j, k);
      put(S, 0, ic, xv[0], ss, bad);
      put(S, 4, ic, xv[1], ss, bad);
      int fk = (m + 1 == n) ? 0 : m + 1;
      put(S, 3, IPf(g, i, j, fk), xv[2], ss, bad);
    }
  }
}

// transverse component of kind 1/2 along d
__host__ __device__ constexpr int trans_comp(int d, int kind) {
  return d == 0 ? (kind == 1 ? 1 : 2) : d == 1 ? (kind == 1 ? 0 : 2) : (kind == 1 ? 0 : 1);
}

// the wall faces of component cc next to the first / last transverse line
template <typename R>
__device__ __forceinline__ void scalar_walls(const SweepArgs<R>& S, int cc, int i, int j, int k) {
  const Geo<R>& g = S.g;
  int lo = (cc == 0) ? (i == 1) : (cc == 1) ? (j == 1) : (k == 1);
  int hi = (cc == 0) ? (i == g.nr - 1) : (cc == 1) ? (j == g.nt - 1) : (k == g.np - 1);
  if (cc == 2 && g.per) lo = hi = 0;
  if (lo) {
    int wi = i, wj = j, wk = k;
    if (cc == 0) wi = 0; else if (cc == 1) wj = 0; else wk = 0;
    put_wall(S, 1 + cc, face_idx(g, cc, wi, wj, wk));
  }
  if (hi) {
    int wi = i, wj = j, wk = k;
    if (cc == 0) wi = g.nr; else if (cc == 1) wj = g.nt; else wk = g.np;
    put_wall(S, 1 + cc, face_idx(g, cc, wi, wj, wk));
  }
}

// output of a transverse line value at cell m, plus the wall faces of that
// component next to the first / last line
template <typename R, typename V, typename Acc>
__device__ __forceinline__ void scalar_put(const SweepArgs<R>& S, int cc, int i, int j, int k, V v, Acc& ss, int* bad) {
  put(S, 1 + cc, face_idx(S.g, cc, i, j, k), v, ss, bad);
  scalar_walls(S, cc, i, j, k);
}

// coefficients (a_m, b_m, c_m) of row m of a transverse scalar line, the
// no-slip fold at the walls of a walled line included
template <typename R>
__device__ __forceinline__ void scalar_row(const SweepArgs<R>& S, int cc, int d, int n, int cyc, int a, int b, int m,
                                           R& am, R& bm, R& cm) {
  int i, j, k;
  line_pos(d, a, b, m, i, j, k);
  R w[3];
  row_s(S.g, S.P, S.c, S.ub, cc, d, i, j, k, w);
  am = S.h * w[0]; bm = R(1) + S.h * w[1]; cm = S.h * w[2];
  if (!cyc) {
    if (m == 0) { bm -= am; am = R(0); }
    if (m == n - 1) { bm -= cm; cm = R(0); }
  }
}

// One transverse scalar line (component trans_comp(D, KIND)) along D: Thomas,
// Sherman-Morrison-corrected on a cyclic line; TR: the transposed system.
template <typename R, int D, int KIND, bool TR = false>
__device__ void scalar_line(const SweepArgs<R>& S, int line, int a, int b, SqSum<R>& ss, int* bad) {
  const Geo<R>& g = S.g;
  constexpr int d = D, kind = KIND;
  int cc = trans_comp(d, kind);
  int n = d == 0 ? g.nr : d == 1 ? g.nt : g.np;
  int cyc = (d == 2 && g.per);
  int nl = S.nl[kind];
  R* scr = S.scr + S.scr_off[kind];
  const R* rhs = S.rhs.f[1 + cc];
  R cp = R(0), dy = R(0), dz = R(0);
  R a0 = R(0), gam = R(1);
  // the row inputs and right-hand side of cell m + 1, loaded before cell m is
  // eliminated (the forward pass)
  SPt<R> qn;
  R rn = R(0);
  auto fetch = [&](int m) {
    int i, j, k;
    line_pos(d, a, b, m, i, j, k);
    qn = load_s(g, S.c, S.ub, cc, d, i, j, k);
    rn = rhs[face_idx(g, cc, i, j, k)];
  };
  if constexpr (!TR) fetch(0);
  for (int m = 0; m < n; m++) {
    int i, j, k;
    line_pos(d, a, b, m, i, j, k);
    R am, bm, cm, r;
    if constexpr (TR) {
      // row m of the transpose: c_{m-1}, b_m, a_{m+1} (wrapping when cyclic)
      R x0, x1, x2;
      scalar_row(S, cc, d, n, cyc, a, b, m, x0, bm, x2);
      am = cm = R(0);
      int mp = m - 1, mn = m + 1;
      if (cyc) { mp = mp < 0 ? n - 1 : mp; mn = mn == n ? 0 : mn; }
      if (mp >= 0) scalar_row(S, cc, d, n, cyc, a, b, mp, x0, x1, am);
      if (mn < n) scalar_row(S, cc, d, n, cyc, a, b, mn, cm, x1, x2);
      r = rhs[face_idx(g, cc, i, j, k)];
    } else {
      const SPt<R> q = qn;
      r = rn;
      if (m + 1 < n) fetch(m + 1);
      R w[3];
      row_sw(g, S.P, q, cc, d, i, j, w);
      am = S.h * w[0]; bm = R(1) + S.h * w[1]; cm = S.h * w[2];
      if (!cyc) {
        if (m == 0) { bm -= am; am = R(0); }
        if (m == n - 1) { bm -= cm; cm = R(0); }
      }
    }
    R zr = R(0);
    if (cyc) {
      // Sherman-Morrison split: gam = -b_0, u = [gam, 0, .., c_{n-1}], v = [1, 0, .., a_0/gam]
      if (m == 0) { a0 = am; gam = -bm; bm -= gam; zr = gam; am = R(0); }
      if (m == n - 1) { bm -= a0 * cm / gam; zr = cm; cm = R(0); }
    }
    R den = bm - am * cp;
    if (den == R(0) || !isfinite(den)) { *bad |= FLAG_SINGULAR; return; }
    R iden = sdiv(R(1), den);
    cp = cm * iden;
    dy = (r - am * dy) * iden;
    R* s = scr + m * 3 * nl + line;
    s[0] = cp;
    s[nl] = dy;
    if (cyc) { dz = (zr - am * dz) * iden; s[2 * nl] = dz; }
  }
  if (!cyc) {
    R xy = dy;
    // the factors of cell m - 1 are loaded before cell m is substituted
    R cn = R(0), yn = R(0);
    if (n >= 2) { cn = scr[(n - 2) * 3 * nl + line]; yn = scr[(n - 2) * 3 * nl + nl + line]; }
    for (int m = n - 1; m >= 0; m--) {
      if (m < n - 1) {
        const R c_ = cn, y_ = yn;
        if (m >= 1) { cn = scr[(m - 1) * 3 * nl + line]; yn = scr[(m - 1) * 3 * nl + nl + line]; }
        xy = y_ - c_ * xy;
      }
      int i, j, k;
      line_pos(d, a, b, m, i, j, k);
      scalar_put(S, cc, i, j, k, xy, ss, bad);
    }
    return;
  }
  // cyclic: back-substitute both columns, then combine in FP64
  R xy = dy, xz = dz, yl = dy, zl = dz;
  for (int m = n - 2; m >= 0; m--) {
    R* t = scr + m * 3 * nl + line;
    xy = t[nl] - t[0] * xy;
    xz = t[2 * nl] - t[0] * xz;
    t[nl] = xy;
    t[2 * nl] = xz;
  }
  {
    R* t = scr + (n - 1) * 3 * nl + line;
    t[nl] = yl;
    t[2 * nl] = zl;
  }
  double ag = (double)a0 / (double)gam;
  double vy = (double)xy + ag * (double)yl, vz = (double)xz + ag * (double)zl;
  double f = vy / (1.0 + vz);
  for (int m = 0; m < n; m++) {
    const R* t = scr + m * 3 * nl + line;
    int i, j, k;
    line_pos(d, a, b, m, i, j, k);
    scalar_put(S, cc, i, j, k, (double)t[nl] - f * (double)t[2 * nl], ss, bad);
  }
}

template <typename R, int D, bool TR = false>
__global__ void __launch_bounds__(128) k_sweep(SweepArgs<R> S) {
  int kind = blockIdx.y;
  int line = blockIdx.x * blockDim.x + threadIdx.x;
  SqSum<R> ss;
  int bad = 0;
  if (line < S.nl[kind]) {
    int a = (int)(line / S.nb[kind]) + S.a0[kind];
    int b = (int)(line % S.nb[kind]) + S.b0[kind];
    if (kind == 0) block_line<R, D, TR>(S, line, a, b, ss, &bad);
    else if (kind == 1) scalar_line<R, D, 1, TR>(S, line, a, b, ss, &bad);
    else scalar_line<R, D, 2, TR>(S, line, a, b, ss, &bad);
  }
  if (bad) atomicOr(S.flag, bad);
  if (S.update && S.norms) {
    for (int f = 0; f < 5; f++) {
      double v = ss.warp_total(f);
      if ((threadIdx.x & 31) == 0 && v != 0.0) atomicAdd(S.acc + f, v);
    }
  }
}
