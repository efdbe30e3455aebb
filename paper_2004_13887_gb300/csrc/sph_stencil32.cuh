// sph_stencil32.cuh -- the stencil stages of the mixed mode in FP32: coefficients
// frozen at Ubar and the right-hand side (Section 2.2, eqs. chapter3mainsd, spl1;
// operators of Appendix B), shared by the single-problem launches and the batched
// ones.
//
// What bounds them: the latency of loads that miss L1 (28 to 37 % hit; DRAM at 40 %
// and issue at 43 to 62 % of their rates), so instructions and loads a cell first.
// As in the FP64 mode (sph_fp64.cuh) what depends on (i, j) alone comes from one
// table entry per row (12 values), the p- and T-rows share their arithmetic, Pb,
// Tb, beta and the centre velocities are formed from values a row reads anyway, and
// the planes Pb, Tb, beta are written only for the line solver that reads them.
// One thread takes a cell's centre and its three lower faces in the right-hand
// side, so that a value two of them use is loaded once, and its own 27 values come
// by asynchronous copies into shared memory, all in flight at once without
// registers; neighbours are found by steps (Loc) instead of checked indices.
// Instructions a cell: coefficients 473 -> 369, right-hand side 1266 (four launches
// side by side) -> 877.
// 128 x 256 x 256 cells, two steps (four of each stage): 8240 us with a launch per
// kind of row, 8101 one thread a cell, 7902 with steps, 7803 with the coefficients
// at 40 registers (12 blocks of 128 an SM; 16 blocks 7922, 9 7865, 6 7940), 7747
// with the copies to shared memory.  Blocks an SM of the right-hand side: 9 (56
// registers) 7747; 12 7830, 10 7846, 8 7776, 7 7820, 5 7970.
#pragma once

#include "sph_fp64_tab.cuh"

namespace s32 {

enum { Q_IR, Q_MT, Q_MP, Q_COTIR, Q_E00, Q_E01, Q_E10, Q_E11, Q_IT, NQ = 12 };
enum { K_IR, K_COT, K_HMT, K_HMP, K_L00, K_L01, K_L10, K_L11, K_LAPT, NK = 12 };
enum { U0_F0, U0_F1, U0_F2, U0_T0, U0_T1, U0_P, U0_QT, U0_QP, U0_QIR, U0_E, U0_GE, U0_OM };
enum { U1_HADV, U1_F0, U1_F1, U1_F2, U1_R0, U1_R1, U1_P, U1_QP, U1_HIR, U1_C, U1_D0, U1_D1 };
enum { U2_HMP, U2_F, U2_R0, U2_R1, U2_T0, U2_T1, U2_QMT, U2_HIR, U2_HCOTIR, U2_OC, U2_OS };
constexpr int NU = 12;

struct Tabs { float *q, *k, *u[3]; };
inline size_t tabs_floats(int nr, int nt) {
  return (size_t)nr * nt * (NQ + NK + NU) + (size_t)NU * ((size_t)(nr + 1) * nt + (size_t)nr * (nt + 1));
}
inline Tabs tabs_of(float* p, int nr, int nt) {
  Tabs T;
  T.q = p; p += (size_t)nr * nt * NQ;
  T.k = p; p += (size_t)nr * nt * NK;
  T.u[0] = p; p += (size_t)(nr + 1) * nt * NU;
  T.u[1] = p; p += (size_t)nr * (nt + 1) * NU;
  T.u[2] = p;
  return T;
}

struct Args {
  Geo<float> g;
  Coef<float> c;
  CF<float> ub, ul, D;     // Ubar, its velocities' remainders, U^k - U^n (hasD)
  CF<double> src;          // S (has_src)
  MF<float> R;
  Tabs T;
  float tau, gm, gm1, iRg, vp2, mu2, kap, difp, idr, hidr, qidr;
  // 2/dr; 64 mu, 8 mu and 2 mu/(3 dr) (viscous factors of the r-faces from 1/(4r));
  // -1/dphi^2; -4 mu/3 (from half metric factors); -16 mu; -3/(4 dphi^2)
  float om, wpr, v64, v8, v3r, vt, vd, v16, vf;
  int hasD, has_src, rot;
  int thermo;              // write the planes Pb, Tb, beta (read by the one-thread-per-line solver only)
};
inline void fill_consts(Args& A, const Par& P, const Geo<double>& g, double tau) {
  A.tau = (float)tau;
  A.gm = P.gamma_f; A.gm1 = (float)(P.gamma - 1.0); A.iRg = P.iRg_f;
  A.vp2 = (float)(2.0 * P.mu * (P.gamma - 1.0)); A.mu2 = (float)(2.0 * P.mu);
  A.kap = P.kappa_f; A.difp = (float)((P.gamma - 1.0) * P.kappa);
  A.idr = (float)g.idr; A.hidr = (float)(0.5 * g.idr); A.qidr = (float)(0.25 * g.idr);
  A.rot = P.omega != 0.0;
  A.om = P.omega_f;
  A.wpr = (float)(2.0 * g.idr); A.v64 = (float)(64.0 * P.mu); A.v8 = (float)(8.0 * P.mu);
  A.v3r = (float)(2.0 / 3.0 * P.mu * g.idr); A.vt = (float)(-1.0 / (g.idph * g.idph)); A.vd = (float)(-4.0 / 3.0 * P.mu);
  A.v16 = (float)(-16.0 * P.mu); A.vf = (float)(-0.75 / (g.idph * g.idph));
}

// N entries of a table row (16-byte aligned, N a multiple of 4) into registers
template <int N>
__device__ __forceinline__ void entries(const float* p, float* m) {
#pragma unroll
  for (int q = 0; q < N / 4; q++) {
    const float4 v = reinterpret_cast<const float4*>(p)[q];
    m[4 * q] = v.x; m[4 * q + 1] = v.y; m[4 * q + 2] = v.z; m[4 * q + 3] = v.w;
  }
}

// Where a cell's own values lie (centre, lower faces) and the steps to its
// neighbours.  Beyond a phi wall the step is 0: the value is the cell's own, with
// the sign s for a velocity along the wall (walls at rest).
struct Loc {
  int i, j, k;
  int t[4];        // flat index in the centre fields, u_r, u_theta, u_phi
  int sj[4], si[4];
  int dm, dp, ep;  // phi: down, up, up in u_phi
  float sm, sp;
};
__device__ __forceinline__ Loc loc_of(const Geo<float>& g, int i, int j, int k) {
  Loc L;
  L.i = i; L.j = j; L.k = k;
  L.sj[0] = L.sj[1] = L.sj[2] = g.np; L.sj[3] = g.npf;
  L.si[0] = L.si[1] = g.nt * g.np; L.si[2] = (g.nt + 1) * g.np; L.si[3] = g.nt * g.npf;
  L.t[0] = L.t[1] = IC(g, i, j, k); L.t[2] = ITf(g, i, j, k); L.t[3] = IPf(g, i, j, k);
  const bool lo = k == 0, hi = k == g.np - 1;
  L.dm = lo ? (g.per ? g.np - 1 : 0) : -1;
  L.dp = hi ? (g.per ? 1 - g.np : 0) : 1;
  L.ep = g.per ? L.dp : 1;
  L.sm = lo && !g.per ? -1.f : 1.f;
  L.sp = hi && !g.per ? -1.f : 1.f;
  return L;
}
// flat index of the neighbour (DI, DJ, DK) in field F (0 centres, 1 u_r, 2 u_theta, 3 u_phi)
template <int F, int DI, int DJ, int DK>
__device__ __forceinline__ int nb_index(const Geo<float>& g, const Loc& L) {
  const int e = L.t[F] + DI * L.si[F] + DJ * L.sj[F] + (DK == 0 ? 0 : DK < 0 ? L.dm : F == 3 ? L.ep : L.dp);
#ifdef SPH_CHECKED
  // the same index from checked coordinates (a mismatch counts as a violation)
  const int k = L.k + DK, i = L.i + DI, j = L.j + DJ;
  const int kk = g.per ? wrapk(g, k) : F == 3 ? (k < 0 ? 0 : k) : clampi(k, 0, g.np - 1);
  const int w = F == 0 ? IC(g, i, j, kk) : F == 1 ? IRf(g, i, j, kk) : F == 2 ? ITf(g, i, j, kk) : IPf(g, i, j, kk);
  if (w != e) return IC(g, -1, j, kk);
#endif
  return e;
}
// The neighbour's value.  Inner tiles (CIJ = 0) take it from the steps: with the
// checked accessors every access along phi costs its own branches and index.
template <int CIJ, int F, int DI, int DJ, int DK>
__device__ __forceinline__ float nb(const Geo<float>& g, const float* f, const Loc& L) {
  if constexpr (CIJ == 0) {
    const float v = f[nb_index<F, DI, DJ, DK>(g, L)];
    return DK == 0 || F == 0 || F == 3 ? v : (DK < 0 ? L.sm : L.sp) * v;
  } else {
    const int i = L.i + DI, j = L.j + DJ, k = L.k + DK;
    return F == 0 ? cpert<CIJ>(g, f, i, j, k) : F == 1 ? vr<CIJ>(g, f, i, j, k) : F == 2 ? vt<CIJ>(g, f, i, j, k)
                                                                                    : vp<CIJ>(g, f, i, j, k);
  }
}

// The coefficients of a centre.
template <int CIJ>
__device__ __forceinline__ void coef(const Args& A, const Loc& L) {
  const Geo<float>& g = A.g;
  const Coef<float>& c = A.c;
  const int i = L.i, j = L.j, t = L.t[0];
  float m[NQ];
  entries<NQ>(A.T.q + (size_t)(i * g.nt + j) * NQ, m);
  const float *UR = A.ub.f[1], *UT = A.ub.f[2], *UP = A.ub.f[3];
  const float pp = A.ub.f[0][t], Tp = A.ub.f[4][t], pref = g.pcen[i], Tref = g.Tcen[i];
  const float Pb = pref + pp, Tb = Tref + Tp, iT = __fdividef(1.f, Tb);
  c.rho[t] = Pb * iT * A.iRg;
  // rho - rho_ref has no cancellation between large terms in this form
  c.drho[t] = (pp * Tref - pref * Tp) * iT * m[Q_IT];
  if (A.thermo) {
    c.Pb[t] = Pb;
    c.Tb[t] = Tb;
    c.beta[t] = __fdividef(A.gm1 * Tb, Pb);
  }
  const float r0 = nb<CIJ, 1, 0, 0, 0>(g, UR, L), r1 = nb<CIJ, 1, 1, 0, 0>(g, UR, L);
  const float t0 = nb<CIJ, 2, 0, 0, 0>(g, UT, L), t1 = nb<CIJ, 2, 0, 1, 0>(g, UT, L);
  const float p0 = nb<CIJ, 3, 0, 0, 0>(g, UP, L), p1 = nb<CIJ, 3, 0, 0, 1>(g, UP, L);
  const float ur = 0.5f * (r0 + r1), ut = 0.5f * (t0 + t1), up = 0.5f * (p0 + p1);
  c.uc0[t] = ur; c.uc1[t] = ut; c.uc2[t] = up;
  const float x = ur * m[Q_IR], dr_ = (r1 - r0) * A.idr, dt_ = (t1 - t0) * m[Q_MT], dvp = (p1 - p0) * m[Q_MP];
  c.grr[t] = dr_;
  c.gtt[t] = dt_ + x;
  c.gpp[t] = fmaf(ut, m[Q_COTIR], dvp + x);
  // centred derivatives of centre-averaged velocities: sums of the four faces
  const float qmt = 0.25f * m[Q_MT], qmp = 0.25f * m[Q_MP];
  const float drt = (nb<CIJ, 2, 1, 0, 0>(g, UT, L) + nb<CIJ, 2, 1, 1, 0>(g, UT, L)) -
                    (nb<CIJ, 2, -1, 0, 0>(g, UT, L) + nb<CIJ, 2, -1, 1, 0>(g, UT, L));
  const float dtr = (nb<CIJ, 1, 0, 1, 0>(g, UR, L) + nb<CIJ, 1, 1, 1, 0>(g, UR, L)) -
                    (nb<CIJ, 1, 0, -1, 0>(g, UR, L) + nb<CIJ, 1, 1, -1, 0>(g, UR, L));
  c.srt[t] = fmaf(-ut, m[Q_IR], fmaf(dtr, qmt, drt * A.qidr));
  const float drp = (nb<CIJ, 3, 1, 0, 0>(g, UP, L) + nb<CIJ, 3, 1, 0, 1>(g, UP, L)) -
                    (nb<CIJ, 3, -1, 0, 0>(g, UP, L) + nb<CIJ, 3, -1, 0, 1>(g, UP, L));
  const float dpr = (nb<CIJ, 1, 0, 0, 1>(g, UR, L) + nb<CIJ, 1, 1, 0, 1>(g, UR, L)) -
                    (nb<CIJ, 1, 0, 0, -1>(g, UR, L) + nb<CIJ, 1, 1, 0, -1>(g, UR, L));
  c.srp[t] = fmaf(-up, m[Q_IR], fmaf(dpr, qmp, drp * A.qidr));
  const float dtp = (nb<CIJ, 3, 0, 1, 0>(g, UP, L) + nb<CIJ, 3, 0, 1, 1>(g, UP, L)) -
                    (nb<CIJ, 3, 0, -1, 0>(g, UP, L) + nb<CIJ, 3, 0, -1, 1>(g, UP, L));
  const float dpt = (nb<CIJ, 2, 0, 0, 1>(g, UT, L) + nb<CIJ, 2, 0, 1, 1>(g, UT, L)) -
                    (nb<CIJ, 2, 0, 0, -1>(g, UT, L) + nb<CIJ, 2, 0, 1, -1>(g, UT, L));
  c.stp[t] = fmaf(-up, m[Q_COTIR], fmaf(dpt, qmp, dtp * qmt));
  // the plain difference, rounded relative to itself, plus the small rest
  c.dvr[t] = fmaf(m[Q_E01], r1, fmaf(-m[Q_E00], r0, dr_));
  c.dvt[t] = fmaf(m[Q_E11], t1, fmaf(-m[Q_E10], t0, dt_));
  c.dvp[t] = dvp;
}

// A cell's own values for the right-hand side, in shared memory: slot q of a
// thread at sh[q * 128].
enum { O_P, O_UR, O_UT, O_UP, O_T, O_GRR, O_GTT, O_GPP, O_SRT, O_SRP, O_STP, O_RHO, O_DRHO, O_U0, O_U1, O_U2, O_DVR, O_DVT,
       O_DVP, O_LR, O_LT, O_LP, O_D, NO = O_D + 5 };
__device__ __forceinline__ void cpa(float* dst, const float* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void own_load(const Args& A, const Loc& L, float* sh) {
  const Coef<float>& c = A.c;
  const int t = L.t[0];
  cpa(sh + O_P * 128, A.ub.f[0] + t); cpa(sh + O_T * 128, A.ub.f[4] + t);
  cpa(sh + O_UR * 128, A.ub.f[1] + L.t[1]); cpa(sh + O_UT * 128, A.ub.f[2] + L.t[2]); cpa(sh + O_UP * 128, A.ub.f[3] + L.t[3]);
  cpa(sh + O_GRR * 128, c.grr + t); cpa(sh + O_GTT * 128, c.gtt + t); cpa(sh + O_GPP * 128, c.gpp + t);
  cpa(sh + O_SRT * 128, c.srt + t); cpa(sh + O_SRP * 128, c.srp + t); cpa(sh + O_STP * 128, c.stp + t);
  cpa(sh + O_LR * 128, A.ul.f[1] + L.t[1]); cpa(sh + O_LT * 128, A.ul.f[2] + L.t[2]); cpa(sh + O_LP * 128, A.ul.f[3] + L.t[3]);
  cpa(sh + O_RHO * 128, c.rho + t); cpa(sh + O_DRHO * 128, c.drho + t);
  cpa(sh + O_U0 * 128, c.uc0 + t); cpa(sh + O_U1 * 128, c.uc1 + t); cpa(sh + O_U2 * 128, c.uc2 + t);
  cpa(sh + O_DVR * 128, c.dvr + t); cpa(sh + O_DVT * 128, c.dvt + t); cpa(sh + O_DVP * 128, c.dvp + t);
  if (A.hasD) {
    cpa(sh + O_D * 128, A.D.f[0] + t); cpa(sh + (O_D + 4) * 128, A.D.f[4] + t);
#pragma unroll
    for (int q = 1; q < 4; q++) cpa(sh + (O_D + q) * 128, A.D.f[q] + L.t[q]);
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// div(Ubar) at centre (i,j,k) from the pair (hi = Ubar, lo) of the velocity
// components: each face flux and each difference is carried as a pair, so the
// cancellation of nearly equal fluxes (and of the three directions against each
// other) at low Mach number costs no accuracy.  r, t, p: the hi values on the
// cell's faces.
__device__ __forceinline__ float div_pair(const Args& A, const Loc& L, const float* sh, const float* r, const float* t, const float* p,
                                          float mt, float mp) {
  const Geo<float>& g = A.g;
  const int i = L.i, j = L.j;
  const float *lr = A.ul.f[1], *lt = A.ul.f[2], *lp = A.ul.f[3];
  const float ir = g.irc[i], is = g.isc[j];
  float h0, l0, h1, l1, dh, dl, th, tl, zh, zl;
  ff_mul(g.rf2h[i + 1], g.rf2l[i + 1], r[1], lr[nb_index<1, 1, 0, 0>(g, L)], h1, l1);
  ff_mul(g.rf2h[i], g.rf2l[i], r[0], sh[O_LR * 128], h0, l0);
  ff_sub(h1, l1, h0, l0, dh, dl);
  ff_mul(dh, dl, ir * ir * A.idr, 0.f, zh, zl);
  ff_mul(g.sfh[j + 1], g.sfl[j + 1], t[1], lt[nb_index<2, 0, 1, 0>(g, L)], h1, l1);
  ff_mul(g.sfh[j], g.sfl[j], t[0], sh[O_LT * 128], h0, l0);
  ff_sub(h1, l1, h0, l0, dh, dl);
  ff_mul(dh, dl, is * mt, 0.f, th, tl);
  ff_add(zh, zl, th, tl, zh, zl);
  ff_sub(p[1], lp[nb_index<3, 0, 0, 1>(g, L)], p[0], sh[O_LP * 128], dh, dl);
  ff_mul(dh, dl, mp, 0.f, th, tl);
  ff_add(zh, zl, th, tl, zh, zl);
  return zh + zl;
}

// one direction of the p- and T-rows: advection into accp, accT, the geometric
// Laplacian of T into lap, the viscous u_d terms (over twice the factor) into vis
template <int CIJ, int D>
__device__ __forceinline__ void cen_dir(const Args& A, const Loc& L, float T0, float adv, float l0, float l1, float lin,
                                        float m0, const float* u, float& accp, float& accT, float& lap, float& vis) {
  const Geo<float>& g = A.g;
  constexpr int di = D == 0, dj = D == 1, dk = D == 2;
  const float *Pp = A.ub.f[0], *TT = A.ub.f[4];
  float dp = nb<CIJ, 0, di, dj, dk>(g, Pp, L) - nb<CIJ, 0, -di, -dj, -dk>(g, Pp, L);
  const float Tm = nb<CIJ, 0, -di, -dj, -dk>(g, TT, L), Tn = nb<CIJ, 0, di, dj, dk>(g, TT, L);
  float dT = Tn - Tm;
  lap = fmaf(l1, Tn - T0, fmaf(l0, Tm - T0, lap));
  if (D == 0) { dp += g.dbgp[L.i]; dT += g.dbgT[L.i]; }
  accp = fmaf(adv, dp, accp);
  accT = fmaf(adv, dT, accT);
  vis = fmaf(lin, u[0] + u[1], fmaf(m0, u[0] - u[1], vis));
}

// R = -(U^k - U^n) - tau (N(Ubar) + G - S) for the p- and T-rows of a centre.
template <int CIJ>
__device__ __forceinline__ float2 rhs_c(const Args& A, const Loc& L, const float* sh) {
  const Geo<float>& g = A.g;
  const int i = L.i, j = L.j, t = L.t[0];
  const float* m = A.T.k + (size_t)(i * g.nt + j) * NK;
  const float *UR = A.ub.f[1], *UT = A.ub.f[2], *UP = A.ub.f[3];
  const float r[2] = {sh[O_UR * 128], nb<CIJ, 1, 1, 0, 0>(g, UR, L)},
              th[2] = {sh[O_UT * 128], nb<CIJ, 2, 0, 1, 0>(g, UT, L)},
              ph[2] = {sh[O_UP * 128], nb<CIJ, 3, 0, 0, 1>(g, UP, L)};
  const float T0 = sh[O_T * 128], Pb = g.pcen[i] + sh[O_P * 128], Tb = g.Tcen[i] + T0;
  const float be = __fdividef(A.gm1 * Tb, Pb);
  const float grr = sh[O_GRR * 128], gtt = sh[O_GTT * 128], gpp = sh[O_GPP * 128], srt = sh[O_SRT * 128],
              srp = sh[O_SRP * 128], stp = sh[O_STP * 128];
  const float t3 = (grr + gtt + gpp) * (1.f / 3.f), vT2 = A.mu2 * be;
  const float ap = fmaf(A.vp2, t3, A.gm * Pb), aT = fmaf(vT2, t3, A.gm1 * Tb);
  const float ur = 0.5f * (r[0] + r[1]), ut = 0.5f * (th[0] + th[1]), up = 0.5f * (ph[0] + ph[1]);
  float accp = 0.f, accT = 0.f, lap = m[K_LAPT], vis = 0.f;
  const float ir = m[K_IR], cot = m[K_COT], hmt = m[K_HMT], hmp = m[K_HMP], qir = 0.25f * ir, mp2 = 4.f * hmp * hmp;
  cen_dir<CIJ, 0>(A, L, T0, ur * A.hidr, m[K_L00], m[K_L01], -2.f * qir * (gtt + gpp), grr * A.idr, r, accp, accT, lap, vis);
  cen_dir<CIJ, 1>(A, L, T0, ut * hmt, m[K_L10], m[K_L11], -qir * fmaf(2.f * cot, gpp, -srt), 2.f * hmt * gtt, th, accp,
                  accT, lap, vis);
  cen_dir<CIJ, 2>(A, L, T0, up * hmp, mp2, mp2, qir * fmaf(stp, cot, srp), 2.f * hmp * gpp, ph, accp, accT, lap, vis);
  const float div = div_pair(A, L, sh, r, th, ph, 2.f * hmt, 2.f * hmp);
  // cross terms of the viscous dissipation: the centred derivative sums are the
  // S planes plus their metric terms
  const float xrt = fmaf(ut, ir, srt), xrp = fmaf(up, ir, srp), xtp = fmaf(up, cot * ir, stp);
  vis = fmaf(-0.5f, fmaf(stp, xtp, fmaf(srp, xrp, srt * xrt)), vis);
  float Np = fmaf(ap, div, fmaf(A.vp2, vis, fmaf(-A.difp, lap, accp)));
  float NT = fmaf(aT, div, fmaf(vT2, vis, fmaf(-A.kap * be, lap, accT)));
  if (A.has_src) { Np -= d2f(A.src.f[0][t]); NT -= d2f(A.src.f[4][t]); }
  const float d0 = A.hasD ? sh[O_D * 128] : 0.f, d4 = A.hasD ? sh[(O_D + 4) * 128] : 0.f;
  return make_float2(fmaf(-A.tau, Np, -d0), fmaf(-A.tau, NT, -d4));
}

// the row along a transverse direction D applied to component C's field: w0, w1
// multiply the differences towards the two neighbours over rho_0 + rho_1 (its
// viscous weights sum to zero), adv the centred difference
template <int CIJ, int C, int D>
__device__ __forceinline__ void trans(const Args& A, const float* U, float u, const Loc& L, float adv, float w0, float w1,
                                      float& acc, float& vis) {
  constexpr int di = D == 0, dj = D == 1, dk = D == 2;
  const float lo = nb<CIJ, 1 + C, -di, -dj, -dk>(A.g, U, L), hi = nb<CIJ, 1 + C, di, dj, dk>(A.g, U, L);
  acc = fmaf(adv, hi - lo, acc);
  vis = fmaf(w0, lo - u, fmaf(w1, hi - u, vis));
}
// the row along its own direction: w0, w1, w2 over rho_0 + rho_1
template <int CIJ, int C>
__device__ __forceinline__ void normal(const Args& A, const float* U, float u, const Loc& L, float adv, float w0, float w1,
                                       float w2, float& acc, float& vis) {
  constexpr int di = C == 0, dj = C == 1, dk = C == 2;
  const float lo = nb<CIJ, 1 + C, -di, -dj, -dk>(A.g, U, L), hi = nb<CIJ, 1 + C, di, dj, dk>(A.g, U, L);
  acc = fmaf(adv, hi - lo, acc);
  vis = fmaf(w0, lo, fmaf(w1, u, fmaf(w2, hi, vis)));
}

// R for the momentum row of component C on an unknown face.
template <int CIJ, int C>
__device__ __forceinline__ float rhs_u(const Args& A, const Loc& L, const float* sh) {
  const Geo<float>& g = A.g;
  const int i = L.i, j = L.j, t = L.t[1 + C];
  const Coef<float>& c = A.c;
  const float* m = A.T.u[C] + (size_t)(C == 1 ? i * (g.nt + 1) + j : i * g.nt + j) * NU;
  const int c0 = nb_index<0, -(C == 0), -(C == 1), -(C == 2)>(g, L);
  const float iv = __fdividef(1.f, c.rho[c0] + sh[O_RHO * 128]);
  const float* U = A.ub.f[1 + C];
  const float* Pp = A.ub.f[0];
  const float u = sh[(O_UR + C) * 128];
  const float* ua = C == 0 ? c.uc1 : c.uc0;
  const float* ub = C == 2 ? c.uc1 : c.uc2;
  const float a0 = ua[c0], a1 = sh[(C == 0 ? O_U1 : O_U0) * 128], b0 = ub[c0], b1 = sh[(C == 2 ? O_U1 : O_U2) * 128], s1 = a0 + a1, s2 = b0 + b1;
  float acc = 0.f, vis;   // vis: what 1/(rho_0 + rho_1) multiplies
  const float dp = sh[O_P * 128] - Pp[c0];
  if (C == 0) {
    const float qir = m[U0_QIR], qv = A.v8 * qir;
    vis = fmaf(A.wpr, dp, fmaf(u * qir, A.v64 * qir,
               fmaf(sh[O_DVT * 128] + sh[O_DVP * 128], qv - A.v3r, (c.dvt[c0] + c.dvp[c0]) * (qv + A.v3r))));
    normal<CIJ, 0>(A, U, u, L, u * A.hidr, m[U0_F0], m[U0_F1], m[U0_F2], acc, vis);
    trans<CIJ, 0, 1>(A, U, u, L, s1 * m[U0_QT], m[U0_T0], m[U0_T1], acc, vis);
    trans<CIJ, 0, 2>(A, U, u, L, s2 * m[U0_QP], m[U0_P], m[U0_P], acc, vis);
    // hydrostatic part: (1/rho_f) d p_ref/dr + g = (1 - b) e + g b, b = 1 - rho_ref,f / rho_f
    acc += fmaf((c.drho[c0] + sh[O_DRHO * 128]) * iv, m[U0_GE], m[U0_E]);
    acc = fmaf(fmaf(s1, s1, s2 * s2), -qir, acc);
    if (A.rot) acc = fmaf(-m[U0_OM], s2, acc);
  } else if (C == 1) {
    const float hm = m[U1_HADV], hir = m[U1_HIR];
    vis = fmaf(4.f * hm, dp, fmaf(u * m[U1_P], A.vt, (sh[O_DVR * 128] - c.dvr[c0]) * (A.vd * hm)));
    vis = fmaf(c.dvp[c0], m[U1_D0], fmaf(sh[O_DVP * 128], m[U1_D1], vis));
    vis = fmaf(a1 - a0, A.v16 * hir * hm, vis);
    normal<CIJ, 1>(A, U, u, L, u * hm, m[U1_F0], m[U1_F1], m[U1_F2], acc, vis);
    trans<CIJ, 1, 0>(A, U, u, L, s1 * A.qidr, m[U1_R0], m[U1_R1], acc, vis);
    trans<CIJ, 1, 2>(A, U, u, L, s2 * m[U1_QP], m[U1_P], m[U1_P], acc, vis);
    acc = fmaf(u * s1, hir, acc);
    acc = fmaf(s2 * s2, -m[U1_C], acc);
    if (A.rot) acc = fmaf(-A.om * g.cf[j], s2, acc);
  } else {
    const float hm = m[U2_HMP], hir = m[U2_HIR], hcot = m[U2_HCOTIR], f = m[U2_F];
    vis = fmaf(4.f * hm, dp, fmaf(u * f, A.vf, ((sh[O_DVR * 128] - c.dvr[c0]) + (sh[O_DVT * 128] - c.dvt[c0])) * (A.vd * hm)));
    vis = fmaf(fmaf(a1 - a0, hir, (b1 - b0) * hcot), A.v16 * hm, vis);
    normal<CIJ, 2>(A, U, u, L, u * hm, f, -2.f * f, f, acc, vis);
    trans<CIJ, 2, 0>(A, U, u, L, s1 * A.qidr, m[U2_R0], m[U2_R1], acc, vis);
    trans<CIJ, 2, 1>(A, U, u, L, s2 * m[U2_QMT], m[U2_T0], m[U2_T1], acc, vis);
    acc = fmaf(u, fmaf(s2, hcot, s1 * hir), acc);
    if (A.rot) acc = fmaf(m[U2_OC], s2, fmaf(m[U2_OS], s1, acc));
  }
  acc = fmaf(iv, vis, acc);
  if (A.has_src) acc -= d2f(A.src.f[1 + C][t]);
  const float d = A.hasD ? sh[(O_D + 1 + C) * 128] : 0.f;
  return fmaf(-A.tau, acc, -d);
}

// the right-hand side of a cell: its centre and its lower faces, zero on wall
// faces; the last cell of a row also zeroes the wall face beyond it
template <int CIJ>
__device__ __forceinline__ void rhs_cell_at(const Args& A, int i, int j, int k, float* sh) {
  const Geo<float>& g = A.g;
  const Loc L = loc_of(g, i, j, k);
  own_load(A, L, sh);
  const float2 pT = rhs_c<CIJ>(A, L, sh);
  const float ur = CIJ && i == 0 ? 0.f : rhs_u<CIJ, 0>(A, L, sh);
  const float ut = CIJ && j == 0 ? 0.f : rhs_u<CIJ, 1>(A, L, sh);
  const float up = !g.per && k == 0 ? 0.f : rhs_u<CIJ, 2>(A, L, sh);
  A.R.f[0][L.t[0]] = pT.x;
  A.R.f[4][L.t[0]] = pT.y;
  A.R.f[1][L.t[1]] = ur;
  A.R.f[2][L.t[2]] = ut;
  A.R.f[3][L.t[3]] = up;
  if (CIJ && i == g.nr - 1) A.R.f[1][IRf(g, g.nr, j, k)] = 0.f;
  if (CIJ && j == g.nt - 1) A.R.f[2][ITf(g, i, g.nt, k)] = 0.f;
  if (!g.per && k == g.np - 1) A.R.f[3][IPf(g, i, j, g.np)] = 0.f;
}
template <bool W>
__device__ __forceinline__ void rhs_cell(const Args& A, int i, int j, int k, bool inner, float* sh) {
  const Geo<float>& g = A.g;
  if (k >= g.np || j >= g.nt || i >= g.nr) return;
  if (inner) rhs_cell_at<0>(A, i, j, k, sh);
  else rhs_cell_at<W ? 2 : 1>(A, i, j, k, sh);
}

}  // namespace s32
