// sph_stencil32.cuh -- the stencil stages of the mixed mode in FP32: coefficients
// frozen at Ubar and the right-hand side (Section 2.2, eqs. chapter3mainsd, spl1;
// operators of Appendix B), shared by the single-problem launches and the batched
// ones.
//
// What bounds them: load latency and the L1's load path (one 128-byte wavefront a
// cycle and SM, a warp's scalar load of one table value costing as much as 32
// field values), then instruction issue; not DRAM.  The kernels they replace
// issued about 830 instructions a centre and 480 a face on two thirds of the
// cycles, at 30-38 % of the DRAM rate.  So, as in the FP64 mode (sph_fp64.cuh):
// what depends on (i, j) alone comes from one table entry per row (12 values;
// what follows from them by a multiplication is not stored), the p- and T-rows
// share their arithmetic, Pb, Tb, beta and the centre velocities are formed from
// values a row reads anyway, and the planes Pb, Tb, beta are written only for the
// line solver that reads them.
// 128 x 256 x 256 cells, us per launch: coefficients 194 -> 175, right-hand side
// (four launches side by side) 707 -> 452.  All at 32 registers (16 blocks of 128
// an SM) in spite of some spills: 40 registers 205 and 473, 48 in the centre rows
// 487; the four kinds in one launch 504; table values loaded ahead into registers
// 477 (but 175 against 183 for the coefficients, which do so).  The tile shape
// makes no difference (128 x 1 x 1 to 32 x 1 x 4 within 1 %).
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

// The coefficients of centre (i, j, k) (flat index t).
template <int CIJ>
__device__ __forceinline__ void coef(const Args& A, int i, int j, int k, int t) {
  const Geo<float>& g = A.g;
  const Coef<float>& c = A.c;
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
  const float r0 = UR[IRf(g, i, j, k)], r1 = UR[IRf(g, i + 1, j, k)];
  const float t0 = UT[ITf(g, i, j, k)], t1 = UT[ITf(g, i, j + 1, k)];
  const float p0 = vp<CIJ>(g, UP, i, j, k), p1 = vp<CIJ>(g, UP, i, j, k + 1);
  const float ur = 0.5f * (r0 + r1), ut = 0.5f * (t0 + t1), up = 0.5f * (p0 + p1);
  c.uc0[t] = ur; c.uc1[t] = ut; c.uc2[t] = up;
  const float x = ur * m[Q_IR], dr_ = (r1 - r0) * A.idr, dt_ = (t1 - t0) * m[Q_MT], dvp = (p1 - p0) * m[Q_MP];
  c.grr[t] = dr_;
  c.gtt[t] = dt_ + x;
  c.gpp[t] = fmaf(ut, m[Q_COTIR], dvp + x);
  // centred derivatives of centre-averaged velocities: sums of the four faces
  const float qmt = 0.25f * m[Q_MT], qmp = 0.25f * m[Q_MP];
  const float drt = (vt<CIJ>(g, UT, i + 1, j, k) + vt<CIJ>(g, UT, i + 1, j + 1, k)) -
                    (vt<CIJ>(g, UT, i - 1, j, k) + vt<CIJ>(g, UT, i - 1, j + 1, k));
  const float dtr = (vr<CIJ>(g, UR, i, j + 1, k) + vr<CIJ>(g, UR, i + 1, j + 1, k)) -
                    (vr<CIJ>(g, UR, i, j - 1, k) + vr<CIJ>(g, UR, i + 1, j - 1, k));
  c.srt[t] = fmaf(-ut, m[Q_IR], fmaf(dtr, qmt, drt * A.qidr));
  const float drp = (vp<CIJ>(g, UP, i + 1, j, k) + vp<CIJ>(g, UP, i + 1, j, k + 1)) -
                    (vp<CIJ>(g, UP, i - 1, j, k) + vp<CIJ>(g, UP, i - 1, j, k + 1));
  const float dpr = (vr<CIJ>(g, UR, i, j, k + 1) + vr<CIJ>(g, UR, i + 1, j, k + 1)) -
                    (vr<CIJ>(g, UR, i, j, k - 1) + vr<CIJ>(g, UR, i + 1, j, k - 1));
  c.srp[t] = fmaf(-up, m[Q_IR], fmaf(dpr, qmp, drp * A.qidr));
  const float dtp = (vp<CIJ>(g, UP, i, j + 1, k) + vp<CIJ>(g, UP, i, j + 1, k + 1)) -
                    (vp<CIJ>(g, UP, i, j - 1, k) + vp<CIJ>(g, UP, i, j - 1, k + 1));
  const float dpt = (vt<CIJ>(g, UT, i, j, k + 1) + vt<CIJ>(g, UT, i, j + 1, k + 1)) -
                    (vt<CIJ>(g, UT, i, j, k - 1) + vt<CIJ>(g, UT, i, j + 1, k - 1));
  c.stp[t] = fmaf(-up, m[Q_COTIR], fmaf(dpt, qmp, dtp * qmt));
  // the plain difference, rounded relative to itself, plus the small rest
  c.dvr[t] = fmaf(m[Q_E01], r1, fmaf(-m[Q_E00], r0, dr_));
  c.dvt[t] = fmaf(m[Q_E11], t1, fmaf(-m[Q_E10], t0, dt_));
  c.dvp[t] = dvp;
}

// div(Ubar) at centre (i,j,k) from the pair (hi = Ubar, lo) of the velocity
// components: each face flux and each difference is carried as a pair, so the
// cancellation of nearly equal fluxes (and of the three directions against each
// other) at low Mach number costs no accuracy.  r, t, p: the hi values on the
// cell's faces.
__device__ __forceinline__ float div_pair(const Args& A, int i, int j, int k, const float* r, const float* t, const float* p,
                                          float mt, float mp) {
  const Geo<float>& g = A.g;
  const int kp = g.per ? wrapk(g, k + 1) : k + 1;
  const float *lr = A.ul.f[1], *lt = A.ul.f[2], *lp = A.ul.f[3];
  const float ir = g.irc[i], is = g.isc[j];
  float h0, l0, h1, l1, dh, dl, th, tl, sh, sl;
  ff_mul(g.rf2h[i + 1], g.rf2l[i + 1], r[1], lr[IRf(g, i + 1, j, k)], h1, l1);
  ff_mul(g.rf2h[i], g.rf2l[i], r[0], lr[IRf(g, i, j, k)], h0, l0);
  ff_sub(h1, l1, h0, l0, dh, dl);
  ff_mul(dh, dl, ir * ir * A.idr, 0.f, sh, sl);
  ff_mul(g.sfh[j + 1], g.sfl[j + 1], t[1], lt[ITf(g, i, j + 1, k)], h1, l1);
  ff_mul(g.sfh[j], g.sfl[j], t[0], lt[ITf(g, i, j, k)], h0, l0);
  ff_sub(h1, l1, h0, l0, dh, dl);
  ff_mul(dh, dl, is * mt, 0.f, th, tl);
  ff_add(sh, sl, th, tl, sh, sl);
  ff_sub(p[1], lp[IPf(g, i, j, kp)], p[0], lp[IPf(g, i, j, k)], dh, dl);
  ff_mul(dh, dl, mp, 0.f, th, tl);
  ff_add(sh, sl, th, tl, sh, sl);
  return sh + sl;
}

// one direction of the p- and T-rows: advection into accp, accT, the geometric
// Laplacian of T into lap, the viscous u_d terms (over twice the factor) into vis
template <int CIJ, int D>
__device__ __forceinline__ void cen_dir(const Args& A, int i, int j, int k, float T0, float adv, float l0, float l1, float lin,
                                        float m0, const float* u, float& accp, float& accT, float& lap, float& vis) {
  const Geo<float>& g = A.g;
  constexpr int di = D == 0, dj = D == 1, dk = D == 2;
  const float *Pp = A.ub.f[0], *TT = A.ub.f[4];
  float dp = cpert<CIJ>(g, Pp, i + di, j + dj, k + dk) - cpert<CIJ>(g, Pp, i - di, j - dj, k - dk);
  const float Tm = cpert<CIJ>(g, TT, i - di, j - dj, k - dk), Tn = cpert<CIJ>(g, TT, i + di, j + dj, k + dk);
  float dT = Tn - Tm;
  lap = fmaf(l1, Tn - T0, fmaf(l0, Tm - T0, lap));
  if (D == 0) { dp += g.dbgp[i]; dT += g.dbgT[i]; }
  accp = fmaf(adv, dp, accp);
  accT = fmaf(adv, dT, accT);
  vis = fmaf(lin, u[0] + u[1], fmaf(m0, u[0] - u[1], vis));
}

// R = -(U^k - U^n) - tau (N(Ubar) + G - S) for the p- and T-rows of a centre.
template <int CIJ>
__device__ __forceinline__ void rhs_c(const Args& A, int i, int j, int k, int t) {
  const Geo<float>& g = A.g;
  const Coef<float>& c = A.c;
  const float* m = A.T.k + (size_t)(i * g.nt + j) * NK;
  const float *UR = A.ub.f[1], *UT = A.ub.f[2], *UP = A.ub.f[3];
  const float r[2] = {UR[IRf(g, i, j, k)], UR[IRf(g, i + 1, j, k)]}, th[2] = {UT[ITf(g, i, j, k)], UT[ITf(g, i, j + 1, k)]},
              ph[2] = {vp<CIJ>(g, UP, i, j, k), vp<CIJ>(g, UP, i, j, k + 1)};
  const float T0 = A.ub.f[4][t], Pb = g.pcen[i] + A.ub.f[0][t], Tb = g.Tcen[i] + T0;
  const float be = __fdividef(A.gm1 * Tb, Pb);
  const float grr = c.grr[t], gtt = c.gtt[t], gpp = c.gpp[t], srt = c.srt[t], srp = c.srp[t], stp = c.stp[t];
  const float t3 = (grr + gtt + gpp) * (1.f / 3.f), vT2 = A.mu2 * be;
  const float ap = fmaf(A.vp2, t3, A.gm * Pb), aT = fmaf(vT2, t3, A.gm1 * Tb);
  const float ur = 0.5f * (r[0] + r[1]), ut = 0.5f * (th[0] + th[1]), up = 0.5f * (ph[0] + ph[1]);
  float accp = 0.f, accT = 0.f, lap = m[K_LAPT], vis = 0.f;
  const float ir = m[K_IR], cot = m[K_COT], hmt = m[K_HMT], hmp = m[K_HMP], qir = 0.25f * ir, mp2 = 4.f * hmp * hmp;
  cen_dir<CIJ, 0>(A, i, j, k, T0, ur * A.hidr, m[K_L00], m[K_L01], -2.f * qir * (gtt + gpp), grr * A.idr, r, accp, accT, lap, vis);
  cen_dir<CIJ, 1>(A, i, j, k, T0, ut * hmt, m[K_L10], m[K_L11], -qir * fmaf(2.f * cot, gpp, -srt), 2.f * hmt * gtt, th, accp,
                  accT, lap, vis);
  cen_dir<CIJ, 2>(A, i, j, k, T0, up * hmp, mp2, mp2, qir * fmaf(stp, cot, srp), 2.f * hmp * gpp, ph, accp, accT, lap, vis);
  const float div = div_pair(A, i, j, k, r, th, ph, 2.f * hmt, 2.f * hmp);
  // cross terms of the viscous dissipation: the centred derivative sums are the
  // S planes plus their metric terms
  const float xrt = fmaf(ut, ir, srt), xrp = fmaf(up, ir, srp), xtp = fmaf(up, cot * ir, stp);
  vis = fmaf(-0.5f, fmaf(stp, xtp, fmaf(srp, xrp, srt * xrt)), vis);
  float Np = fmaf(ap, div, fmaf(A.vp2, vis, fmaf(-A.difp, lap, accp)));
  float NT = fmaf(aT, div, fmaf(vT2, vis, fmaf(-A.kap * be, lap, accT)));
  if (A.has_src) { Np -= d2f(A.src.f[0][t]); NT -= d2f(A.src.f[4][t]); }
  const float d0 = A.hasD ? A.D.f[0][t] : 0.f, d4 = A.hasD ? A.D.f[4][t] : 0.f;
  A.R.f[0][t] = fmaf(-A.tau, Np, -d0);
  A.R.f[4][t] = fmaf(-A.tau, NT, -d4);
}

// velocity component C beside its face, with the ghosts of the walls
template <int CIJ, int C>
__device__ __forceinline__ float vel(const Geo<float>& g, const float* u, int i, int j, int k) {
  return C == 0 ? vr<CIJ>(g, u, i, j, k) : C == 1 ? vt<CIJ>(g, u, i, j, k) : vp<CIJ>(g, u, i, j, k);
}
// the row along a transverse direction D applied to component C's field: w0, w1
// multiply the differences towards the two neighbours over rho_0 + rho_1 (its
// viscous weights sum to zero), adv the centred difference
template <int CIJ, int C, int D>
__device__ __forceinline__ void trans(const Args& A, const float* U, float u, int i, int j, int k, float adv, float w0, float w1,
                                      float& acc, float& vis) {
  constexpr int di = D == 0, dj = D == 1, dk = D == 2;
  const float lo = vel<CIJ, C>(A.g, U, i - di, j - dj, k - dk), hi = vel<CIJ, C>(A.g, U, i + di, j + dj, k + dk);
  acc = fmaf(adv, hi - lo, acc);
  vis = fmaf(w0, lo - u, fmaf(w1, hi - u, vis));
}
// the row along its own direction: w0, w1, w2 over rho_0 + rho_1
template <int CIJ, int C>
__device__ __forceinline__ void normal(const Args& A, const float* U, float u, int i, int j, int k, float adv, float w0, float w1,
                                       float w2, float& acc, float& vis) {
  constexpr int di = C == 0, dj = C == 1, dk = C == 2;
  const float lo = vel<CIJ, C>(A.g, U, i - di, j - dj, k - dk), hi = vel<CIJ, C>(A.g, U, i + di, j + dj, k + dk);
  acc = fmaf(adv, hi - lo, acc);
  vis = fmaf(w0, lo, fmaf(w1, u, fmaf(w2, hi, vis)));
}

// R for the momentum row of component C on an unknown face.
template <int CIJ, int C>
__device__ __forceinline__ void rhs_u(const Args& A, int i, int j, int k, int t) {
  const Geo<float>& g = A.g;
  const Coef<float>& c = A.c;
  const float* m = A.T.u[C] + (size_t)(C == 1 ? i * (g.nt + 1) + j : i * g.nt + j) * NU;
  const int c1 = IC(g, i, j, k);
  const int c0 = C == 0 ? IC(g, i - 1, j, k) : C == 1 ? IC(g, i, j - 1, k) : IC(g, i, j, g.per ? wrapk(g, k - 1) : k - 1);
  const float iv = __fdividef(1.f, c.rho[c0] + c.rho[c1]);
  const float* U = A.ub.f[1 + C];
  const float* Pp = A.ub.f[0];
  const float u = U[t];
  const float* ua = C == 0 ? c.uc1 : c.uc0;
  const float* ub = C == 2 ? c.uc1 : c.uc2;
  const float a0 = ua[c0], a1 = ua[c1], b0 = ub[c0], b1 = ub[c1], s1 = a0 + a1, s2 = b0 + b1;
  float acc = 0.f, vis;   // vis: what 1/(rho_0 + rho_1) multiplies
  const float dp = Pp[c1] - Pp[c0];
  if (C == 0) {
    const float qir = m[U0_QIR], qv = A.v8 * qir;
    vis = fmaf(A.wpr, dp, fmaf(u * qir, A.v64 * qir,
               fmaf(c.dvt[c1] + c.dvp[c1], qv - A.v3r, (c.dvt[c0] + c.dvp[c0]) * (qv + A.v3r))));
    normal<CIJ, 0>(A, U, u, i, j, k, u * A.hidr, m[U0_F0], m[U0_F1], m[U0_F2], acc, vis);
    trans<CIJ, 0, 1>(A, U, u, i, j, k, s1 * m[U0_QT], m[U0_T0], m[U0_T1], acc, vis);
    trans<CIJ, 0, 2>(A, U, u, i, j, k, s2 * m[U0_QP], m[U0_P], m[U0_P], acc, vis);
    // hydrostatic part: (1/rho_f) d p_ref/dr + g = (1 - b) e + g b, b = 1 - rho_ref,f / rho_f
    acc += fmaf((c.drho[c0] + c.drho[c1]) * iv, m[U0_GE], m[U0_E]);
    acc = fmaf(fmaf(s1, s1, s2 * s2), -qir, acc);
    if (A.rot) acc = fmaf(-m[U0_OM], s2, acc);
  } else if (C == 1) {
    const float hm = m[U1_HADV], hir = m[U1_HIR];
    vis = fmaf(4.f * hm, dp, fmaf(u * m[U1_P], A.vt, (c.dvr[c1] - c.dvr[c0]) * (A.vd * hm)));
    vis = fmaf(c.dvp[c0], m[U1_D0], fmaf(c.dvp[c1], m[U1_D1], vis));
    vis = fmaf(a1 - a0, A.v16 * hir * hm, vis);
    normal<CIJ, 1>(A, U, u, i, j, k, u * hm, m[U1_F0], m[U1_F1], m[U1_F2], acc, vis);
    trans<CIJ, 1, 0>(A, U, u, i, j, k, s1 * A.qidr, m[U1_R0], m[U1_R1], acc, vis);
    trans<CIJ, 1, 2>(A, U, u, i, j, k, s2 * m[U1_QP], m[U1_P], m[U1_P], acc, vis);
    acc = fmaf(u * s1, hir, acc);
    acc = fmaf(s2 * s2, -m[U1_C], acc);
    if (A.rot) acc = fmaf(-A.om * g.cf[j], s2, acc);
  } else {
    const float hm = m[U2_HMP], hir = m[U2_HIR], hcot = m[U2_HCOTIR], f = m[U2_F];
    vis = fmaf(4.f * hm, dp, fmaf(u * f, A.vf, ((c.dvr[c1] - c.dvr[c0]) + (c.dvt[c1] - c.dvt[c0])) * (A.vd * hm)));
    vis = fmaf(fmaf(a1 - a0, hir, (b1 - b0) * hcot), A.v16 * hm, vis);
    normal<CIJ, 2>(A, U, u, i, j, k, u * hm, f, -2.f * f, f, acc, vis);
    trans<CIJ, 2, 0>(A, U, u, i, j, k, s1 * A.qidr, m[U2_R0], m[U2_R1], acc, vis);
    trans<CIJ, 2, 1>(A, U, u, i, j, k, s2 * m[U2_QMT], m[U2_T0], m[U2_T1], acc, vis);
    acc = fmaf(u, fmaf(s2, hcot, s1 * hir), acc);
    if (A.rot) acc = fmaf(m[U2_OC], s2, fmaf(m[U2_OS], s1, acc));
  }
  acc = fmaf(iv, vis, acc);
  if (A.has_src) acc -= d2f(A.src.f[1 + C][t]);
  const float d = A.hasD ? A.D.f[1 + C][t] : 0.f;
  A.R.f[1 + C][t] = fmaf(-A.tau, acc, -d);
}

// the right-hand side of one point of kind 0 (centres) or 1 + C (faces of component
// C) in a tile whose first point is (i0, j0): zero on wall faces
template <bool W>
__device__ __forceinline__ void rhs_point(const Args& A, int kind, int i, int j, int k, bool inner) {
  const Geo<float>& g = A.g;
  if (kind == 0) {
    if (k >= g.np || j >= g.nt || i >= g.nr) return;
    const int t = IC(g, i, j, k);
    if (inner) rhs_c<0>(A, i, j, k, t);
    else rhs_c<W ? 2 : 1>(A, i, j, k, t);
  } else if (kind == 1) {
    if (k >= g.np || j >= g.nt || i > g.nr) return;
    const int t = IRf(g, i, j, k);
    if (i == 0 || i == g.nr) A.R.f[1][t] = 0.f;
    else if (inner) rhs_u<0, 0>(A, i, j, k, t);
    else rhs_u<W ? 2 : 1, 0>(A, i, j, k, t);
  } else if (kind == 2) {
    if (k >= g.np || j > g.nt || i >= g.nr) return;
    const int t = ITf(g, i, j, k);
    if (j == 0 || j == g.nt) A.R.f[2][t] = 0.f;
    else if (inner) rhs_u<0, 1>(A, i, j, k, t);
    else rhs_u<W ? 2 : 1, 1>(A, i, j, k, t);
  } else {
    if (k >= g.npf || j >= g.nt || i >= g.nr) return;
    const int t = IPf(g, i, j, k);
    if (!g.per && (k == 0 || k == g.np)) A.R.f[3][t] = 0.f;
    else if (inner) rhs_u<0, 2>(A, i, j, k, t);
    else rhs_u<W ? 2 : 1, 2>(A, i, j, k, t);
  }
}

}  // namespace s32
