// sph_fp64.cu -- launches of the FP64 mode's kernels (sph_fp64.cuh,
// sph_fp64_lines.cuh): the coefficients frozen at Ubar, the right-hand side of
// eq. spl1 with the line rows it stores, and the sweeps of eqs. spl1-spl3
// (Section 2.2) with their transposes.
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include "../../include/sph.h"
#include "sph_kernels.cuh"
#include "sph_host.cuh"
#include "sph_fp64.cuh"
#include "sph_fp64_lines.cuh"
#include "sph_adjoint.cuh"

// what the FP64 mode's coefficient and right-hand-side kernels take
static f64::Args args64(sph_ctx* c, CF<double> ub) {
  f64::Args A;
  memset(&A, 0, sizeof A);
  A.g = c->d64.g;
  A.k = f64::consts_of(c->d64.g, c->P);
  A.T = c->tabs;
  A.c = c->d64.c;
  A.ub = ub;
  A.rows = c->rows;
  return A;
}

// on the context's stream, in order after the uploads of the tables it reads
void f64_tables(sph_ctx* c) {
  const Geo<double>& g = c->d64.g;
  f64::k_tab<<<((g.nr + 1) * (g.nt + 1) + 127) / 128, 128, 0, c->st>>>(g, c->P, c->tabs);
}

void f64_coef(sph_ctx* c, CF<double> ub) {
  const Geo<double>& g = c->d64.g;
  f64::k_coef<<<tile_grid(g.np, g.nt, g.nr), TILE_BLOCK, 0, c->st>>>(args64(c, ub));
}

void f64_rhs(sph_ctx* c, CF<double> ub, CF<double> D, int hasD, double tau, CF<double> src, int has_src, MF<double> R) {
  const Geo<double>& g = c->d64.g;
  f64::Args A = args64(c, ub);
  A.D = D; A.hasD = hasD; A.src = src; A.has_src = has_src; A.tau = tau; A.R = R;
  f64::k_rhs_c<<<tile_grid(g.np, g.nt, g.nr), TILE_BLOCK, 0, c->st>>>(A);
  f64::k_rhs_u<0><<<tile_grid(g.np, g.nt, g.nr + 1), TILE_BLOCK, 0, c->aux[0]>>>(A);
  f64::k_rhs_u<1><<<tile_grid(g.np, g.nt + 1, g.nr), TILE_BLOCK, 0, c->aux[1]>>>(A);
  f64::k_rhs_u<2><<<tile_grid(g.npf, g.nt, g.nr), TILE_BLOCK, 0, c->aux[2]>>>(A);
}

void f64_rows(sph_ctx* c, CF<double> ub, int dir) {
  size_t mx = 0;
  for (int f = 0; f < 5; f++) mx = c->nf[f] > mx ? c->nf[f] : mx;
  const dim3 grid((unsigned)((mx + 127) / 128), 4);   // centres, then the faces of each kind
  const f64::Args A = args64(c, ub);
  if (dir == 0) f64::k_rows<0><<<grid, 128, 0, c->st>>>(A);
  else if (dir == 1) f64::k_rows<1><<<grid, 128, 0, c->st>>>(A);
  else f64::k_rows<2><<<grid, 128, 0, c->st>>>(A);
}

// Block lines below which the FP64 sweeps split a line's 3x3 arithmetic over
// lanes: a warp then holds 4 lines (2 cyclic ones) instead of 16, and its
// serial chain is about 0.4 times as long, at 1.6 times the FP64 instructions in
// all.  The split pays while the unsplit launch, nl / 16 warps on 4 nsm SM quarters,
// leaves half of them idle: 32 lines an SM.  (4096 lines of 128 cells along theta,
// 8192 along r of 32 cells, unsplit: 413 and 262 us; 4096 cyclic ones split 1102.)
static int lines64_split(const sph_ctx* c, int nl) { return nl <= 32 * c->nsm; }

template <int D, bool CYC, bool TR>
static void launch_lines64(sph_ctx* c, const f64::LineArgs& S) {
  const int mx = S.nl[1] > S.nl[2] ? S.nl[1] : S.nl[2];
  if (lines64_split(c, S.nl[0])) {
    const int per = CYC ? 4 : 8, nb = (S.nl[0] + per - 1) / per, ns = (mx + 31) / 32;
    f64::k_lines<D, CYC, TR, true><<<dim3(nb > ns ? nb : ns, 3), 64, 0, c->st>>>(S);
  } else {
    const int m = mx > S.nl[0] ? mx : S.nl[0];
    f64::k_lines<D, CYC, TR, false><<<dim3((m + 31) / 32, 3), 64, 0, c->st>>>(S);
  }
}

void f64_lines(sph_ctx* c, int d, double tau, CF<double> rhs, MF<double> x, int update, CF<double> base, MF<double> uk,
               bool transposed, bool norms) {
  SweepArgs<double> L;
  memset(&L, 0, sizeof L);
  line_layout(c->d64.g, d, L);
  f64::LineArgs S;
  memset(&S, 0, sizeof S);
  S.g = c->d64.g; S.rows = c->rows; S.beta = c->d64.c.beta; S.tab = c->tabs.s[d]; S.ih = 2.0 / tau;
  S.rhs = rhs; S.x = x; S.update = update; S.norms = norms; S.base = base; S.uk = uk;
  S.scr = c->d64.scr; S.acc = c->acc; S.flag = c->flag;
  for (int q = 0; q < 3; q++) {
    S.scr_off[q] = L.scr_off[q]; S.nl[q] = L.nl[q]; S.a0[q] = L.a0[q]; S.nb[q] = L.nb[q]; S.b0[q] = L.b0[q];
  }
#define SPH_LINES64(D, C) (transposed ? launch_lines64<D, C, true>(c, S) : launch_lines64<D, C, false>(c, S))
  if (d == 0) SPH_LINES64(0, false);
  else if (d == 1) SPH_LINES64(1, false);
  else if (c->d64.g.per) SPH_LINES64(2, true);
  else SPH_LINES64(2, false);
#undef SPH_LINES64
}

void f64_adjoint(sph_ctx* c, double tau, CF<double> ub, const CF<double>* mu, const CF<double>* x, double* const* lam) {
  static_assert(f64::NL == f64::ADJ_PLANES, "the accumulators of k_adj_u");
  const Geo<double>& g = c->d64.g;
  f64::AdjArgs A;
  memset(&A, 0, sizeof A);
  A.g = g; A.k = f64::consts_of(g, c->P); A.T = c->tabs; A.c = c->d64.c; A.ub = ub; A.tau = tau;
  for (int d = 0; d < 3; d++) { A.mu[d] = mu[d]; A.x[d] = x[d]; }
  for (int f = 0; f < 5; f++) A.lam[f] = lam[f];
  for (int q = 0; q < f64::NL; q++) A.pl[q] = c->adjC + (size_t)q * c->N;
  f64::k_adj_u<0><<<tile_grid(g.np, g.nt, g.nr + 1), TILE_BLOCK, 0, c->st>>>(A);
  f64::k_adj_u<1><<<tile_grid(g.np, g.nt + 1, g.nr), TILE_BLOCK, 0, c->st>>>(A);
  f64::k_adj_u<2><<<tile_grid(g.npf, g.nt, g.nr), TILE_BLOCK, 0, c->st>>>(A);
  f64::k_adj_c<<<tile_grid(g.np, g.nt, g.nr), TILE_BLOCK, 0, c->st>>>(A);
}

void f64_axpy(sph_ctx* c, long n, double s, const double* x, double* y) {
  const long b = (n + 255) / 256;
  f64::k_axpy<<<(unsigned)(b < 16L * c->nsm ? b : 16L * c->nsm), 256, 0, c->st>>>(n, s, x, y);
}

#ifdef SPH_CHECKED
int bounds_take_f64(int* h) {
  int z[5] = {0, 0, 0, 0, 0};
  if (cudaMemcpyFromSymbol(h, g_bounds, 5 * sizeof(int)) != cudaSuccess ||
      cudaMemcpyToSymbol(g_bounds, z, sizeof z) != cudaSuccess)
    return SPH_ERR_CUDA;
  return SPH_OK;
}
#endif
