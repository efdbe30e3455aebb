// sph_lines2.cu -- launches of the sweeps of the mixed mode over many lines
// (sph_lines2.cuh; Section 2.2, eqs. spl1-spl3).
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include "../../include/sph.h"
#include "sph_kernels.cuh"
#include "sph_host.cuh"
#include "sph_lines2.cuh"
#include "sph_lines2_kernels.cuh"

static lines2::Tabs tabs(const sph_ctx* c) { return lines2::tabs_of(c->tab32, c->d64.g.nr, c->d64.g.nt); }

size_t lines2_tab_floats(int nr, int nt) { return lines2::tabs_floats(nr, nt); }

void lines2_tables(sph_ctx* c) {
  const Geo<double>& g = c->d64.g;
  lines2::k_tab<<<((g.nr + 1) * (g.nt + 1) + 127) / 128, 128, 0, c->st>>>(g, c->P, tabs(c));
}

// blocks of 32 lines: block lines, first and second transverse kind
static void blocks_of(const Geo<double>& g, int d, int nb[3]) {
  if (d == 2) {
    nb[0] = (g.nr * g.nt + 31) / 32;
    nb[1] = ((g.nr - 1) * g.nt + 31) / 32;
    nb[2] = (g.nr * (g.nt - 1) + 31) / 32;
    return;
  }
  const int na = d == 0 ? g.nt : g.nr, inner = g.np - (g.per ? 0 : 1);   // u_phi: interior faces
  nb[0] = (na * g.np + 31) / 32;
  nb[1] = ((na - 1) * g.np + 31) / 32;
  nb[2] = (na * inner + 31) / 32;
}

size_t lines2_scratch(const Geo<double>& g, int d) {
  int nb[3];
  blocks_of(g, d, nb);
  const bool cyc = d == 2 && g.per;
  return (size_t)(d == 0 ? g.nr : d == 1 ? g.nt : g.np) * 32 *
         ((cyc ? 21 : 12) * (size_t)nb[0] + (cyc ? 3 : 2) * (size_t)(nb[1] + nb[2]));
}

void lines2_rows(const sph_ctx* c, int d, double tau, SweepArgs<float>* S) {
  const lines2::Tabs T = tabs(c);
  const double h = 0.5 * tau, gm = c->P.gamma, mu = c->P.mu;
  S->tb = T.b[d];
  S->ts[0] = T.s[d][0]; S->ts[1] = T.s[d][1];
  S->hgm = (float)(h * gm); S->hgm1 = (float)(h * (gm - 1.0)); S->hvp2 = (float)(h * 2.0 * mu * (gm - 1.0));
  S->hmu2 = (float)(h * 2.0 * mu); S->gm1 = (float)(gm - 1.0); S->iRg = c->P.iRg_f;
}

void lines2_fill(const sph_ctx* c, int d, double tau, CF<float> ub, CF<float> rhs, MF<float> x, lines2::Args* A, int* nblk,
                 int* nsca) {
  int nb[3];
  blocks_of(c->d64.g, d, nb);
  memset(A, 0, sizeof *A);
  A->g = c->d32.g; A->c = c->d32.c; A->ub = ub; A->rhs = rhs; A->x = x; A->T = tabs(c);
  const double h = 0.5 * tau, gm = c->P.gamma, mu = c->P.mu;
  A->h = (float)h; A->hgm = (float)(h * gm); A->hgm1 = (float)(h * (gm - 1.0));
  A->hvp2 = (float)(h * 2.0 * mu * (gm - 1.0)); A->hmu2 = (float)(h * 2.0 * mu);
  A->gm1 = (float)(gm - 1.0); A->iRg = c->P.iRg_f;
  A->scr = c->d32.scr; A->nb0 = nb[0]; A->nb1 = nb[1]; A->flag = c->flag;
  *nblk = nb[0];
  *nsca = nb[1] + nb[2];
}

void lines2_run(sph_ctx* c, int d, double tau, CF<float> ub, CF<float> rhs, MF<float> x, int update, int norms,
                CF<double> base, MF<double> uk, cudaStream_t st_sca) {
  const Geo<double>& g = c->d64.g;
  lines2::Args A;
  int nb, ns;
  lines2_fill(c, d, tau, ub, rhs, x, &A, &nb, &ns);
  A.update = update; A.norms = update && norms; A.base = base; A.uk = uk; A.acc = c->acc;
#define SPH_LINES2(KB, KS) do { KB<<<nb, 64, 0, c->st>>>(A); if (ns > 0) KS<<<ns, 64, 0, st_sca>>>(A); } while (0)
  if (d == 0) SPH_LINES2((lines2::k_blk<0>), (lines2::k_sca<0>));
  else if (d == 1) SPH_LINES2((lines2::k_blk<1>), (lines2::k_sca<1>));
  else {
    // every float row starts on a 16-byte boundary when np is a multiple of 4
    // (the fields' and planes' own bases are allocations' starts or multiples of
    // the cell count), the FP64 state's rows too
    const bool vec = g.np % 4 == 0;
    if (g.per && vec) SPH_LINES2((lines2::k_blk_phi<true, true>), (lines2::k_sca_phi<true, true>));
    else if (g.per) SPH_LINES2((lines2::k_blk_phi<true, false>), (lines2::k_sca_phi<true, false>));
    else if (vec) SPH_LINES2((lines2::k_blk_phi<false, true>), (lines2::k_sca_phi<false, true>));
    else SPH_LINES2((lines2::k_blk_phi<false, false>), (lines2::k_sca_phi<false, false>));
  }
#undef SPH_LINES2
}

#ifdef SPH_CHECKED
int bounds_take_lines2(int* h) {
  int z[5] = {0, 0, 0, 0, 0};
  if (cudaMemcpyFromSymbol(h, g_bounds, 5 * sizeof(int)) != cudaSuccess ||
      cudaMemcpyToSymbol(g_bounds, z, sizeof z) != cudaSuccess)
    return SPH_ERR_CUDA;
  return SPH_OK;
}
#endif
