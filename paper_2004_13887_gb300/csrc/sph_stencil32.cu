// sph_stencil32.cu -- launches of the mixed mode's stencil stages
// (sph_stencil32.cuh): the coefficients frozen at Ubar and the right-hand side of
// eq. spl1 (Section 2.2), and their tables.
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include "../../include/sph.h"
#include "sph_kernels.cuh"
#include "sph_host.cuh"
#include "sph_stencil32.cuh"

namespace s32 {

// the FP32 tables from the FP64 ones (sph_fp64.cuh's k_tab) and the background
__global__ void k_pack(Geo<double> g, f64::Tabs S, Tabs T) {
  using namespace f64;
  const int e = blockIdx.x * blockDim.x + threadIdx.x, i = e / (g.nt + 1), j = e % (g.nt + 1);
  if (i > g.nr) return;
  if (i < g.nr && j < g.nt) {
    const double* c = S.c + (size_t)(i * g.nt + j) * f64::NC;
    float* q = T.q + (size_t)(i * g.nt + j) * NQ;
    const int from[9] = {C_IR, C_MT, C_MP, C_COTIR, C_E00, C_E01, C_E10, C_E11, C_IT};
    for (int z = 0; z < NQ; z++) q[z] = z < 9 ? (float)c[from[z]] : 0.f;
    float* k = T.k + (size_t)(i * g.nt + j) * NK;
    const int kf[8] = {C_IR, C_COT, C_HMT, C_HMP, C_L00, C_L01, C_L10, C_L11};
    for (int z = 0; z < NK; z++) k[z] = z < 8 ? (float)c[kf[z]] : 0.f;
    k[K_LAPT] = (float)g.lapT[i];
    float* u = T.u[2] + (size_t)(i * g.nt + j) * NU;
    const int uf[11] = {C_HMP, P_F, P_R0, P_R1, P_T0, P_T1, C_QMT, C_HIR, C_HCOTIR, P_OC, P_OS};
    for (int z = 0; z < NU; z++) u[z] = z < 11 ? (float)c[uf[z]] : 0.f;
  }
  if (i >= 1 && i < g.nr && j < g.nt) {
    const double* r = S.r + (size_t)(i * g.nt + j) * f64::NR;
    float* u = T.u[0] + (size_t)(i * g.nt + j) * NU;
    const int f[NU] = {R_F0, R_F1, R_F2, R_T0, R_T1, R_P, R_QT, R_QP, R_QIR, R_E, R_GE, R_OM};
    for (int z = 0; z < NU; z++) u[z] = (float)r[f[z]];
  }
  if (i < g.nr && j >= 1 && j < g.nt) {
    const double* t = S.t + (size_t)(i * (g.nt + 1) + j) * f64::NT;
    float* u = T.u[1] + (size_t)(i * (g.nt + 1) + j) * NU;
    const int f[NU] = {T_HADV, T_F0, T_F1, T_F2, T_R0, T_R1, T_P, T_QP, T_HIR, T_C, T_D0, T_D1};
    for (int z = 0; z < NU; z++) u[z] = (float)t[f[z]];
  }
}

template <bool W>
__global__ void __launch_bounds__(128, 12) k_coef(const __grid_constant__ Args A) {
  const Geo<float>& g = A.g;
  const int k = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y,
            i = blockIdx.z * blockDim.z + threadIdx.z;
  const bool inner = !W && tile_inner(g);   // with wall data every tile takes the checked path
  if (k >= g.np || j >= g.nt || i >= g.nr) return;
  const Loc L = loc_of(g, i, j, k);
  if (inner) coef<0>(A, L);
  else coef<W ? 2 : 1>(A, L);
}

template <bool W>
__global__ void __launch_bounds__(128, 9) k_rhs(const __grid_constant__ Args A) {
  __shared__ float own[NO][128];
  const int i0 = blockIdx.z * blockDim.z, j0 = blockIdx.y * blockDim.y;
  float* sh = &own[0][(threadIdx.z * blockDim.y + threadIdx.y) * blockDim.x + threadIdx.x];
  rhs_cell<W>(A, i0 + threadIdx.z, j0 + threadIdx.y, blockIdx.x * blockDim.x + threadIdx.x,
              !W && tile_inner_at(A.g, i0, j0, (int)blockDim.z, (int)blockDim.y), sh);
}

}  // namespace s32

size_t s32_tab_floats(int nr, int nt) { return s32::tabs_floats(nr, nt); }

// after f64_tables on the same stream
void s32_tables(sph_ctx* c) {
  const Geo<double>& g = c->d64.g;
  s32::k_pack<<<((g.nr + 1) * (g.nt + 1) + 127) / 128, 128, 0, c->st>>>(g, c->tabs, s32::tabs_of(c->tab32s, g.nr, g.nt));
}

void s32_fill(const sph_ctx* c, CF<float> ub, double tau, s32::Args* A) {
  const Geo<double>& g = c->d64.g;
  memset(A, 0, sizeof *A);
  A->g = c->d32.g; A->c = c->d32.c; A->ub = ub;
  for (int f = 0; f < 5; f++) { A->ul.f[f] = c->d32.UbLo[f]; A->D.f[f] = c->d32.Db[f]; A->R.f[f] = c->d32.Rb[f]; }
  A->T = s32::tabs_of(c->tab32s, g.nr, g.nt);
  s32::fill_consts(*A, c->P, g, tau);
}

void s32_coef(sph_ctx* c, CF<float> ub, int thermo) {
  const Geo<double>& g = c->d64.g;
  s32::Args A;
  s32_fill(c, ub, 0.0, &A);
  A.thermo = thermo;
  if (c->d32.g.hasw) s32::k_coef<true><<<tile_grid(g.np, g.nt, g.nr), TILE_BLOCK, 0, c->st>>>(A);
  else s32::k_coef<false><<<tile_grid(g.np, g.nt, g.nr), TILE_BLOCK, 0, c->st>>>(A);
}

void s32_rhs(sph_ctx* c, CF<float> ub, int hasD, double tau, CF<double> src, int has_src, MF<float> R) {
  s32::Args A;
  s32_fill(c, ub, tau, &A);
  A.hasD = hasD; A.src = src; A.has_src = has_src; A.R = R;
  const Geo<double>& g = c->d64.g;
  if (c->d32.g.hasw) s32::k_rhs<true><<<tile_grid(g.np, g.nt, g.nr), TILE_BLOCK, 0, c->st>>>(A);
  else s32::k_rhs<false><<<tile_grid(g.np, g.nt, g.nr), TILE_BLOCK, 0, c->st>>>(A);
}

#ifdef SPH_CHECKED
int bounds_take_s32(int* h) {
  int z[5] = {0, 0, 0, 0, 0};
  if (cudaMemcpyFromSymbol(h, g_bounds, 5 * sizeof(int)) != cudaSuccess ||
      cudaMemcpyToSymbol(g_bounds, z, sizeof z) != cudaSuccess)
    return SPH_ERR_CUDA;
  return SPH_OK;
}
#endif
