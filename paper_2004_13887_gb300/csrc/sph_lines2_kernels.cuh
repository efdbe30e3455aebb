// sph_lines2_kernels.cuh -- the single-problem launches of sph_lines2.cuh and the
// kernel that makes their tables.
#pragma once

namespace lines2 {

// one thread per (i, j), i <= nr, j <= nt (FP64 arithmetic, rounded at the end)
__global__ void k_tab(Geo<double> g, Par P, Tabs T) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x, i = e / (g.nt + 1), j = e % (g.nt + 1);
  if (i > g.nr) return;
  const double mu = P.mu, kap = P.kappa;
  if (i < g.nr) {   // u_theta on the theta-face j, along phi (the pole faces are no unknowns)
    const double mpf = g.irc[i] * g.isf[j] * g.idph;
    float* s = T.s[2][1] + (size_t)NS * (i * (g.nt + 1) + j);
    s[S_W0] = s[S_W2] = (float)(-2.0 * mu * mpf * mpf);
    s[S_W1] = (float)(4.0 * mu * mpf * mpf);
    s[S_Q] = (float)(0.25 * mpf);
  }
  if (j == g.nt) return;
  {                 // u_r on the r-face i, along phi
    const double mpf = g.irf[i] * g.isc[j] * g.idph;
    float* s = T.s[2][0] + (size_t)NS * (i * g.nt + j);
    s[S_W0] = s[S_W2] = (float)(-2.0 * mu * mpf * mpf);
    s[S_W1] = (float)(4.0 * mu * mpf * mpf);
    s[S_Q] = (float)(0.25 * mpf);
  }
  if (i < g.nr) {
    const double ir = g.irc[i], is = g.isc[j], mt = ir * g.idth;
    const double f0 = g.rf[i] * g.rf[i], f1 = g.rf[i + 1] * g.rf[i + 1];
    const double g00 = f0 * ir * ir * g.idr, g01 = f1 * ir * ir * g.idr, l00 = g00 * g.idr, l01 = g01 * g.idr;
    if (j == 0) {
      float* b = T.b[0] + (size_t)NB * i;
      b[B_G0] = (float)g00; b[B_G1] = (float)g01;
      b[B_K0] = (float)(-kap * l00); b[B_K1] = (float)(-kap * l01);
      b[B_LIN] = (float)(-0.5 * ir); b[B_COT2] = 0.f;
      b[B_M] = (float)g.idr; b[B_HM] = (float)(0.5 * g.idr);
      double w[4] = {0.0, 0.0, 0.0, 0.0};
      if (i + 1 < g.nr) {   // the r-face i + 1
        const double q = g.irf[i + 1] * g.irf[i + 1], m2 = g.idr * g.idr;
        const double c0 = g.rc[i] * g.rc[i], c1 = g.rc[i + 1] * g.rc[i + 1];
        const double ic0 = g.irc[i] * g.irc[i], ic1 = g.irc[i + 1] * g.irc[i + 1];
        const double fp = g.rf[i + 2] * g.rf[i + 2];
        w[0] = 2.0 * g.idr;
        w[1] = -2.0 * mu * m2 * (q * c0 + f0 * ic0 / 3.0);
        w[2] = 2.0 * mu * m2 * (q * (c0 + c1) + f1 * (ic1 + ic0) / 3.0);
        w[3] = -2.0 * mu * m2 * (q * c1 + fp * ic1 / 3.0);
      }
      b[B_WP] = (float)w[0]; b[B_F0] = (float)w[1]; b[B_FS] = (float)(w[1] + w[2] + w[3]); b[B_F2] = (float)w[3];
      float* s = T.s[0][0] + (size_t)NS * i;
      s[S_W0] = (float)(-2.0 * mu * l00); s[S_W1] = (float)(2.0 * mu * (l00 + l01)); s[S_W2] = (float)(-2.0 * mu * l01);
      s[S_Q] = (float)(0.25 * g.idr);
    }
    const double g10 = g.sf[j] * is * mt, g11 = g.sf[j + 1] * is * mt, l10 = g10 * mt, l11 = g11 * mt;
    float* b = T.b[1] + (size_t)NB * (i * g.nt + j);
    b[B_G0] = (float)g10; b[B_G1] = (float)g11;
    b[B_K0] = (float)(-kap * l10); b[B_K1] = (float)(-kap * l11);
    b[B_LIN] = (float)(-0.25 * ir); b[B_COT2] = (float)(2.0 * g.cotc[j]);
    b[B_M] = (float)mt; b[B_HM] = (float)(0.5 * mt);
    double w[4] = {0.0, 0.0, 0.0, 0.0};
    if (j + 1 < g.nt) {   // the theta-face j + 1
      const double isf = g.isf[j + 1], c0 = g.sc[j], c1 = g.sc[j + 1], ic0 = g.isc[j], ic1 = g.isc[j + 1], m2 = mt * mt;
      w[0] = 2.0 * mt;
      w[1] = -2.0 * mu * m2 * (isf * c0 + g.sf[j] * ic0 / 3.0);
      w[2] = 2.0 * mu * m2 * (isf * (c0 + c1) + g.sf[j + 1] * (ic1 + ic0) / 3.0);
      w[3] = -2.0 * mu * m2 * (isf * c1 + g.sf[j + 2] * ic1 / 3.0);
    }
    b[B_WP] = (float)w[0]; b[B_F0] = (float)w[1]; b[B_FS] = (float)(w[1] + w[2] + w[3]); b[B_F2] = (float)w[3];
    const double mp = ir * is * g.idph;
    float* f = T.b[2] + (size_t)NB * (i * g.nt + j);
    f[B_G0] = f[B_G1] = (float)mp;
    f[B_K0] = f[B_K1] = (float)(-kap * mp * mp);
    f[B_LIN] = (float)(0.25 * ir); f[B_COT2] = (float)g.cotc[j];
    f[B_M] = (float)mp; f[B_HM] = (float)(0.5 * mp);
    f[B_WP] = (float)(2.0 * mp);
    f[B_F0] = f[B_F2] = (float)(-8.0 / 3.0 * mu * mp * mp); f[B_FS] = 0.f;
    float* s = T.s[1][1] + (size_t)NS * (i * g.nt + j);
    s[S_W0] = (float)(-2.0 * mu * l10); s[S_W1] = (float)(2.0 * mu * (l10 + l11)); s[S_W2] = (float)(-2.0 * mu * l11);
    s[S_Q] = (float)(0.25 * mt);
  }
  // u_r on the r-face i, along theta
  const double irf = g.irf[i], at = irf * irf * g.idth * g.idth * g.isc[j];
  float* s = T.s[1][0] + (size_t)NS * (i * g.nt + j);
  s[S_W0] = (float)(-2.0 * mu * at * g.sf[j]); s[S_W1] = (float)(2.0 * mu * at * (g.sf[j] + g.sf[j + 1]));
  s[S_W2] = (float)(-2.0 * mu * at * g.sf[j + 1]);
  s[S_Q] = (float)(0.25 * irf * g.idth);
}

template <int D>
__global__ void __launch_bounds__(64, LINES2_MINB) k_blk(const __grid_constant__ Args A) {
  __shared__ float ex[NEX][32];
  __shared__ float rings[2 * RING][32];
  int bad = 0;
  block_lines<D>(A, ex, rings, blockIdx.x, &bad);
  if (bad) atomicOr(A.flag, bad);
}
// both transverse kinds: blocks [0, nb1) take kind 1
template <int D>
__global__ void __launch_bounds__(64) k_sca(const __grid_constant__ Args A) {
  __shared__ float ex[4][32];
  __shared__ float rings[2 * SRING][32];
  int bad = 0;
  if ((int)blockIdx.x < A.nb1) scalar_lines<D, 1>(A, ex, rings, blockIdx.x, blockIdx.x, &bad);
  else scalar_lines<D, 2>(A, ex, rings, blockIdx.x - A.nb1, blockIdx.x, &bad);
  if (bad) atomicOr(A.flag, bad);
}

__device__ __forceinline__ void finish(const Args& A, const SqSum<float>& ss, int bad) {
  if (bad) atomicOr(A.flag, bad);
  if (A.norms) {
    for (int f = 0; f < 5; f++) {
      const double v = ss.warp_total(f);
      if ((threadIdx.x & 31) == 0 && v != 0.0) atomicAdd(A.acc + f, v);
    }
  }
}
// (6 blocks an SM, 168 registers: at 175, 5 blocks, the scalar lines no longer fit beside
// them and the step of 100 x 200 x 200 takes 4.98 ms instead of 4.47)
template <bool CYC, bool VEC>
__global__ void __launch_bounds__(64, 6) k_blk_phi(const __grid_constant__ Args A) {
  __shared__ float ex[CYC ? 42 : NEX][32];
  int bad = 0;
  SqSum<float> ss;
  block_lines_phi<CYC, VEC>(A, ex, blockIdx.x, ss, &bad);
  finish(A, ss, bad);
}
template <bool CYC, bool VEC>
__global__ void __launch_bounds__(64) k_sca_phi(const __grid_constant__ Args A) {
  __shared__ float ex[6][32];
  int bad = 0;
  SqSum<float> ss;
  if ((int)blockIdx.x < A.nb1) scalar_lines_phi<1, CYC, VEC>(A, ex, blockIdx.x, blockIdx.x, ss, &bad);
  else scalar_lines_phi<2, CYC, VEC>(A, ex, blockIdx.x - A.nb1, blockIdx.x, ss, &bad);
  finish(A, ss, bad);
}

}  // namespace lines2
