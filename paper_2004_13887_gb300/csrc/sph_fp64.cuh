// sph_fp64.cuh -- the stages of the FP64 mode: coefficients, right-hand side and
// line solves of one Picard iteration (Section 2.2, eqs. chapter3mainsd,
// splitting2, spl1-spl3; operators of Appendix B).
//
// What bounds them: GB300 issues one FP64 instruction of a warp every 64 cycles
// per SM quarter, whatever it is (add, multiply, fused multiply-add), however
// many lanes are active and whether or not it depends on the one before
// (measured: 64.4 cycles independent, 65.4 dependent; 1 to 32 active lanes the
// same).  An FP64 stage costs its count of FP64 instructions; loads, integer
// work and FP32 are nearly free beside them.  So everything that depends only
// on the position (i, j) -- metric products, viscous weights, powers of two --
// is read from tables made once per context (k_tab), the p- and T-rows share
// their arithmetic, a row value is formed once and stored for the line solves
// (Rows), and the 3x3 block products skip the blocks' structural zeros (a
// compiler may not: 0 * x is not 0 for every x).
//
// Measured on 128 x 256 x 256 cells, us per launch, with every product formed
// where it is used -> now: coefficients 1850 -> 1092; right-hand side, centres
// 4592 -> 1453, faces of each component 2270-2410 -> 704-734; sweeps r, theta,
// phi 2841, 3086, 4199 -> 2018, 2064, 2224; the step of two iterations 47.3 ->
// 22.6 ms.  The error against the same scheme in independent FP64 arithmetic is
// that of the former kernels (p 1.8e-16, T 1.8e-16, u 5.4e-16 relative; 2.0,
// 2.2, 4.6e-16 before).
#pragma once

#include "sph_fp64_tab.cuh"

namespace f64 {

// constants of a context in the form the kernels use them
struct K64 {
  double idr, hidr, qidr;     // 1/dr, half, quarter
  double gm, gm1, iRg;        // gamma, gamma - 1, 1/Rg
  double vp2;                 // 2 mu (gamma - 1): twice the p-row's viscous factor
  double mu2;                 // 2 mu (times beta: the T-row's)
  double kap, difp;           // kappa, (gamma - 1) kappa
  int rot;                    // omega != 0
};
inline K64 consts_of(const Geo<double>& g, const Par& P) {
  K64 k;
  k.idr = g.idr; k.hidr = 0.5 * g.idr; k.qidr = 0.25 * g.idr;
  k.gm = P.gamma; k.gm1 = P.gamma - 1.0; k.iRg = 1.0 / P.Rg;
  k.vp2 = 2.0 * P.mu * (P.gamma - 1.0); k.mu2 = 2.0 * P.mu;
  k.kap = P.kappa; k.difp = (P.gamma - 1.0) * P.kappa;
  k.rot = P.omega != 0.0;
  return k;
}

// unevaluated sums of two doubles (~106 bits), so that each table entry is
// rounded once: the weights of a cell's two faces nearly cancel
struct dd { double h, l; };
__device__ __forceinline__ dd prod(double a, double b) { const double p = a * b; return {p, fma(a, b, -p)}; }
__device__ __forceinline__ dd prod(dd a, dd b) {
  const dd p = prod(a.h, b.h);
  const double l = p.l + fma(a.h, b.l, a.l * b.h), h = p.h + l;
  return {h, l - (h - p.h)};
}
__device__ __forceinline__ dd prod(dd a, double b) { return prod(a, dd{b, 0.0}); }
__device__ __forceinline__ dd quot(dd a, dd b) {
  const double q = a.h / b.h;
  const dd p = prod(b, q);
  return {q, ((a.h - p.h) + (a.l - p.l)) / b.h};
}
__device__ __forceinline__ double val(dd a) { return a.h + a.l; }

// one thread per (i, j), i <= nr, j <= nt
__global__ void k_tab(Geo<double> g, Par P, Tabs T) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = e / (g.nt + 1), j = e % (g.nt + 1);
  if (i > g.nr) return;
  const double mu = P.mu, om = P.omega, kap = P.kappa;
  const bool ci = i < g.nr, cj = j < g.nt;
  const double ir = ci ? g.irc[i] : 0.0, is = cj ? g.isc[j] : 0.0;
  const dd one = {1.0, 0.0}, rr = {ci ? g.rc[i] : 1.0, 0.0}, ss = {cj ? g.sc[j] : 1.0, 0.0}, r2 = prod(rr, rr);
  const dd mt2 = quot(prod(one, g.idth), rr), mp2 = quot(prod(one, g.idph), prod(rr, ss));
  const double mt = val(mt2), mp = val(mp2);
  const dd q0 = quot(ci ? prod(g.rf[i], g.rf[i]) : one, r2), q1 = quot(ci ? prod(g.rf[i + 1], g.rf[i + 1]) : one, r2);
  const double g00 = val(prod(q0, g.idr)), g01 = val(prod(q1, g.idr));
  const double l00 = val(prod(q0, prod(g.idr, g.idr))), l01 = val(prod(q1, prod(g.idr, g.idr)));
  if (ci && cj) {
    const dd s0 = prod(quot(dd{g.sf[j], 0.0}, ss), mt2), s1 = prod(quot(dd{g.sf[j + 1], 0.0}, ss), mt2);
    const double g10 = val(s0), g11 = val(s1), l10 = val(prod(s0, mt2)), l11 = val(prod(s1, mt2));
    const double cot = g.cotc[j];
    double* c = T.c + (size_t)(i * g.nt + j) * NC;
    c[C_IR] = ir; c[C_HIR] = 0.5 * ir; c[C_QIR] = 0.25 * ir;
    c[C_MT] = mt; c[C_HMT] = 0.5 * mt; c[C_QMT] = 0.25 * mt;
    c[C_MP] = mp; c[C_HMP] = 0.5 * mp; c[C_QMP] = 0.25 * mp; c[C_MP2] = val(prod(mp2, mp2));
    c[C_G00] = g00; c[C_G01] = g01; c[C_G10] = g10; c[C_G11] = g11;
    const dd h0 = quot(dd{g.sf[j], 0.0}, ss), h1 = quot(dd{g.sf[j + 1], 0.0}, ss);
    c[C_E00] = val(prod(dd{q0.h - 1.0, q0.l}, g.idr)); c[C_E01] = val(prod(dd{q1.h - 1.0, q1.l}, g.idr));
    c[C_E10] = val(prod(dd{h0.h - 1.0, h0.l}, mt2)); c[C_E11] = val(prod(dd{h1.h - 1.0, h1.l}, mt2));
    c[C_L00] = l00; c[C_L01] = l01; c[C_L10] = l10; c[C_L11] = l11;
    c[C_IT] = 1.0 / (P.Rg * g.Tcen[i]);
    c[C_COT] = cot; c[C_COT2] = 2.0 * cot; c[C_COTIR] = cot * ir; c[C_HCOTIR] = 0.5 * cot * ir;
    c[P_WP] = 2.0 * mp; c[P_F] = -8.0 / 3.0 * mu * mp * mp; c[P_F2] = 16.0 / 3.0 * mu * mp * mp;
    c[P_R0] = -2.0 * mu * l00; c[P_R1] = -2.0 * mu * l01; c[P_RS] = 2.0 * mu * (l00 + l01);
    c[P_T0] = -2.0 * mu * l10; c[P_T1] = -2.0 * mu * l11; c[P_TS] = 2.0 * mu * (l10 + l11);
    c[P_V] = 2.0 * mu * ir * ir * is * is; c[P_D] = -2.0 / 3.0 * mu * mp;
    c[P_UR] = -4.0 * mu * ir * mp; c[P_UT] = -4.0 * mu * g.cc[j] * ir * is * mp;
    c[P_OC] = om * g.cc[j]; c[P_OS] = om * g.sc[j];
    const double a0[3] = {l00, l10, mp * mp}, a1[3] = {l01, l11, mp * mp};
    for (int d = 0; d < 3; d++) {
      double* s = T.s[d] + (size_t)(i * g.nt + j) * NS;
      s[S_K0] = -kap * a0[d]; s[S_K1] = -kap * a1[d]; s[S_KS] = kap * (a0[d] + a1[d]);
      const double dp = (P.gamma - 1.0) * kap;
      s[S_D0] = -dp * a0[d]; s[S_D1] = -dp * a1[d]; s[S_DS] = dp * (a0[d] + a1[d]);
    }
  }
  if (cj && i >= 1 && i < g.nr) {
    const double irf = g.irf[i], m2 = g.idr * g.idr, q = irf * irf;
    const double c0 = g.rc[i - 1] * g.rc[i - 1], c1 = g.rc[i] * g.rc[i];
    const double ic0 = g.irc[i - 1] * g.irc[i - 1], ic1 = g.irc[i] * g.irc[i];
    const double fm = g.rf[i - 1] * g.rf[i - 1], fc = g.rf[i] * g.rf[i], fp = g.rf[i + 1] * g.rf[i + 1];
    const double at = q * g.idth * g.idth * is, mpf = irf * is * g.idph;
    double* r = T.r + (size_t)(i * g.nt + j) * NR;
    r[R_WP] = 2.0 * g.idr;
    r[R_F0] = -2.0 * mu * m2 * (q * c0 + fm * ic0 / 3.0);
    r[R_F1] = 2.0 * mu * m2 * (q * (c0 + c1) + fc * (ic1 + ic0) / 3.0);
    r[R_F2] = -2.0 * mu * m2 * (q * c1 + fp * ic1 / 3.0);
    r[R_T0] = -2.0 * mu * at * g.sf[j]; r[R_T1] = -2.0 * mu * at * g.sf[j + 1];
    r[R_TS] = 2.0 * mu * at * (g.sf[j] + g.sf[j + 1]);
    r[R_QT] = 0.25 * irf * g.idth;
    r[R_P] = -2.0 * mu * mpf * mpf; r[R_P2] = 4.0 * mu * mpf * mpf; r[R_QP] = 0.25 * mpf;
    r[R_QIR] = 0.25 * irf; r[R_V] = 4.0 * mu * q;
    r[R_Q0] = 2.0 * mu * (irf + g.idr / 3.0); r[R_Q1] = 2.0 * mu * (irf - g.idr / 3.0);
    r[R_OM] = om * g.sc[j];
    r[R_E] = g.ehyd[i]; r[R_GE] = P.g - g.ehyd[i];
  }
  if (ci && j >= 1 && j < g.nt) {
    const double isf = g.isf[j], cf = g.cf[j], c0 = g.sc[j - 1], c1 = g.sc[j], ic0 = g.isc[j - 1], ic1 = g.isc[j];
    const double m2 = mt * mt, mpf = ir * isf * g.idph, d = -2.0 / 3.0 * mu * mt, e = 2.0 * mu * cf * ir * isf * isf;
    double* t = T.t + (size_t)(i * (g.nt + 1) + j) * NT;
    t[T_WP] = 2.0 * mt; t[T_HADV] = 0.5 * mt;
    t[T_F0] = -2.0 * mu * m2 * (isf * c0 + g.sf[j - 1] * ic0 / 3.0);
    t[T_F1] = 2.0 * mu * m2 * (isf * (c0 + c1) + g.sf[j] * (ic1 + ic0) / 3.0);
    t[T_F2] = -2.0 * mu * m2 * (isf * c1 + g.sf[j + 1] * ic1 / 3.0);
    t[T_R0] = -2.0 * mu * l00; t[T_R1] = -2.0 * mu * l01; t[T_RS] = 2.0 * mu * (l00 + l01);
    t[T_P] = -2.0 * mu * mpf * mpf; t[T_P2] = 4.0 * mu * mpf * mpf; t[T_QP] = 0.25 * mpf;
    t[T_HIR] = 0.5 * ir; t[T_C] = 0.25 * g.cotf[j] * ir; t[T_V] = 2.0 * mu * ir * ir * isf * isf;
    t[T_D] = d; t[T_D0] = -d + e * c0; t[T_D1] = d + e * c1;
    t[T_UR] = -4.0 * mu * ir * mt; t[T_OM] = om * cf;
  }
}

// ------------------------------------------------------------- coefficients

// What a coefficient or right-hand-side kernel reads and writes.
struct Args {
  Geo<double> g;
  K64 k;
  Tabs T;
  Coef<double> c;
  CF<double> ub;     // Ubar
  CF<double> D;      // U^k - U^n (hasD)
  CF<double> src;    // S (has_src)
  int hasD, has_src;
  double tau;
  MF<double> R;
  Rows rows;
};

// The 17 coefficients of a centre (67 FP64 instructions, from 116).
__global__ void __launch_bounds__(128) k_coef(const __grid_constant__ Args A) {
  const Geo<double>& g = A.g;
  const int k = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y,
            i = blockIdx.z * blockDim.z + threadIdx.z;
  if (k >= g.np || j >= g.nt || i >= g.nr) return;
  const int t = IC(g, i, j, k);
  const double* m = A.T.c + (size_t)(i * g.nt + j) * NC;
  const double *UR = A.ub.f[1], *UT = A.ub.f[2], *UP = A.ub.f[3];
  const Coef<double>& c = A.c;
  const double pp = A.ub.f[0][t], Tp = A.ub.f[4][t], pref = g.pcen[i], Tref = g.Tcen[i];
  const double Pb = pref + pp, Tb = Tref + Tp;
  const double iT = 1.0 / Tb;
  c.Pb[t] = Pb;
  c.Tb[t] = Tb;
  c.rho[t] = Pb * iT * A.k.iRg;
  // rho - rho_ref, without cancellation between large terms
  c.drho[t] = (pp * Tref - pref * Tp) * iT * m[C_IT];
  c.beta[t] = (1.0 / Pb) * (A.k.gm1 * Tb);
  const double r0 = UR[IRf(g, i, j, k)], r1 = UR[IRf(g, i + 1, j, k)];
  const double t0 = UT[ITf(g, i, j, k)], t1 = UT[ITf(g, i, j + 1, k)];
  const double p0 = vp<2>(g, UP, i, j, k), p1 = vp<2>(g, UP, i, j, k + 1);
  const double ur = 0.5 * (r0 + r1), ut = 0.5 * (t0 + t1), up = 0.5 * (p0 + p1);
  c.uc0[t] = ur; c.uc1[t] = ut; c.uc2[t] = up;
  const double x = ur * m[C_IR], dr_ = (r1 - r0) * A.k.idr, dt_ = (t1 - t0) * m[C_MT], dvp = (p1 - p0) * m[C_MP],
               cotir = m[C_COTIR];
  c.grr[t] = dr_;
  c.gtt[t] = dt_ + x;
  c.gpp[t] = fma(ut, cotir, dvp + x);
  // centred derivatives of centre-averaged velocities: sums of the four faces
  const double qt = m[C_QMT], qp = m[C_QMP], qr = A.k.qidr;
  const double drt = (vt<2>(g, UT, i + 1, j, k) + vt<2>(g, UT, i + 1, j + 1, k)) -
                     (vt<2>(g, UT, i - 1, j, k) + vt<2>(g, UT, i - 1, j + 1, k));
  const double dtr = (vr<2>(g, UR, i, j + 1, k) + vr<2>(g, UR, i + 1, j + 1, k)) -
                     (vr<2>(g, UR, i, j - 1, k) + vr<2>(g, UR, i + 1, j - 1, k));
  c.srt[t] = fma(-ut, m[C_IR], fma(dtr, qt, drt * qr));
  const double drp = (vp<2>(g, UP, i + 1, j, k) + vp<2>(g, UP, i + 1, j, k + 1)) -
                     (vp<2>(g, UP, i - 1, j, k) + vp<2>(g, UP, i - 1, j, k + 1));
  const double dpr = (vr<2>(g, UR, i, j, k + 1) + vr<2>(g, UR, i + 1, j, k + 1)) -
                     (vr<2>(g, UR, i, j, k - 1) + vr<2>(g, UR, i + 1, j, k - 1));
  c.srp[t] = fma(-up, m[C_IR], fma(dpr, qp, drp * qr));
  const double dtp = (vp<2>(g, UP, i, j + 1, k) + vp<2>(g, UP, i, j + 1, k + 1)) -
                     (vp<2>(g, UP, i, j - 1, k) + vp<2>(g, UP, i, j - 1, k + 1));
  const double dpt = (vt<2>(g, UT, i, j, k + 1) + vt<2>(g, UT, i, j + 1, k + 1)) -
                     (vt<2>(g, UT, i, j, k - 1) + vt<2>(g, UT, i, j + 1, k - 1));
  c.stp[t] = fma(-up, cotir, fma(dpt, qp, dtp * qt));
  // the plain difference, rounded relative to itself, plus the small rest
  c.dvr[t] = fma(m[C_E01], r1, fma(-m[C_E00], r0, dr_));
  c.dvt[t] = fma(m[C_E11], t1, fma(-m[C_E10], t0, dt_));
  c.dvp[t] = dvp;
}

// ------------------------------------------------------- rows at the centres

// What the p- and T-rows of every direction at a centre share.
struct CenC {
  double ap, aT, vT2, be;     // divergence coefficients, twice the T-row's viscous factor, beta
  double grr, gtt, gpp, srt, srp, stp;
};
__device__ __forceinline__ CenC cen_load(const K64& k, const Coef<double>& c, int t) {
  CenC q;
  q.grr = c.grr[t]; q.gtt = c.gtt[t]; q.gpp = c.gpp[t];
  q.srt = c.srt[t]; q.srp = c.srp[t]; q.stp = c.stp[t];
  q.be = c.beta[t];
  const double t3 = (q.grr + q.gtt + q.gpp) * (1.0 / 3.0);
  q.vT2 = k.mu2 * q.be;
  q.ap = fma(k.vp2, t3, k.gm * c.Pb[t]);
  q.aT = fma(q.vT2, t3, k.gm1 * c.Tb[t]);
  return q;
}
// The part of the u_d couplings that is not the divergence's: twice the viscous
// factor times (s, u) on the cell's two faces, s = lin + m0, u = lin - m0.
template <int D>
__device__ __forceinline__ void cen_visc(const K64& k, const CenC& q, const double* m, double& s, double& u) {
  double lin, m0;
  if (D == 0) { lin = (q.gtt + q.gpp) * -m[C_HIR]; m0 = q.grr * k.idr; }
  else if (D == 1) { lin = fma(q.gpp, m[C_COT2], -q.srt) * -m[C_QIR]; m0 = q.gtt * m[C_MT]; }
  else { lin = fma(q.stp, m[C_COT], q.srp) * m[C_QIR]; m0 = q.gpp * m[C_MP]; }
  s = lin + m0;
  u = lin - m0;
}
template <int D>
__device__ __forceinline__ double cen_adv(const K64& k, const Coef<double>& c, const double* m, int t) {
  return D == 0 ? c.uc0[t] * k.hidr : D == 1 ? c.uc1[t] * m[C_HMT] : c.uc2[t] * m[C_HMP];
}
template <int D>
__device__ __forceinline__ void cen_store(const K64& k, const Rows& o, const CenC& q, const double* m, double adv,
                                          double s, double u, int t) {
  double* p = o.c[D] + t;
  const long n = o.nc;
  p[0] = adv;
  if (D == 2) {
    const double x = q.ap * m[C_MP], y = q.aT * m[C_MP];
    p[n] = fma(k.vp2, s, -x); p[2 * n] = fma(k.vp2, u, x);
    p[3 * n] = fma(q.vT2, s, -y); p[4 * n] = fma(q.vT2, u, y);
  } else {
    const double g0 = m[D == 0 ? C_G00 : C_G10], g1 = m[D == 0 ? C_G01 : C_G11];
    p[n] = fma(-q.ap, g0, k.vp2 * s); p[2 * n] = fma(q.ap, g1, k.vp2 * u);
    p[3 * n] = fma(-q.aT, g0, q.vT2 * s); p[4 * n] = fma(q.aT, g1, q.vT2 * u);
  }
}

// one direction of the p- and T-rows applied to Ubar: sums of the advection of
// p and T, the geometric Laplacian of T and the viscous u_d terms
template <int D>
__device__ __forceinline__ void cen_apply(const Args& A, const CenC& q, const double* m, int i, int j, int k, int t,
                                          double& accp, double& accT, double& lap, double& vis) {
  const Geo<double>& g = A.g;
  constexpr int di = D == 0, dj = D == 1, dk = D == 2;
  const double adv = cen_adv<D>(A.k, A.c, m, t);
  double s, u;
  cen_visc<D>(A.k, q, m, s, u);
  cen_store<D>(A.k, A.rows, q, m, adv, s, u, t);
  const double *Pp = A.ub.f[0], *TT = A.ub.f[4], *U = A.ub.f[1 + D];
  double dp = cpert<2>(g, Pp, i + di, j + dj, k + dk) - cpert<2>(g, Pp, i - di, j - dj, k - dk);
  const double Tm = cpert<2>(g, TT, i - di, j - dj, k - dk), T0 = TT[t], Tn = cpert<2>(g, TT, i + di, j + dj, k + dk);
  double dT = Tn - Tm;
  if (D == 2) lap = fma(m[C_MP2], fma(-2.0, T0, Tm + Tn), lap);
  else lap = fma(m[D == 0 ? C_L01 : C_L11], Tn - T0, fma(m[D == 0 ? C_L00 : C_L10], Tm - T0, lap));
  if (D == 0) { dp += g.dbgp[i]; dT += g.dbgT[i]; }
  accp = fma(adv, dp, accp);
  accT = fma(adv, dT, accT);
  const double u0 = D == 2 ? vp<2>(g, U, i, j, k) : U[t + (D == 1 ? i * g.np : 0)];
  const double u1 = D == 0 ? U[IRf(g, i + 1, j, k)] : D == 1 ? U[ITf(g, i, j + 1, k)] : vp<2>(g, U, i, j, k + 1);
  vis = fma(s, u0, fma(u, u1, vis));
}

// R = -(U^k - U^n) - tau (N(Ubar) + G - S) for the p- and T-rows, storing the
// rows of the three directions: one thread per centre (99 FP64 instructions,
// from 293).
__global__ void __launch_bounds__(128) k_rhs_c(const __grid_constant__ Args A) {
  const Geo<double>& g = A.g;
  const int k = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y,
            i = blockIdx.z * blockDim.z + threadIdx.z;
  if (k >= g.np || j >= g.nt || i >= g.nr) return;
  const int t = IC(g, i, j, k);
  const double* m = A.T.c + (size_t)(i * g.nt + j) * NC;
  const Coef<double>& c = A.c;
  const CenC q = cen_load(A.k, c, t);
  double accp = 0.0, accT = 0.0, lap = g.lapT[i], vis = 0.0;
  cen_apply<0>(A, q, m, i, j, k, t, accp, accT, lap, vis);
  cen_apply<1>(A, q, m, i, j, k, t, accp, accT, lap, vis);
  cen_apply<2>(A, q, m, i, j, k, t, accp, accT, lap, vis);
  // cross terms of the viscous dissipation: the centred derivative sums are the
  // S planes plus their metric terms
  const double ut = c.uc1[t], up = c.uc2[t], ir = m[C_IR];
  const double xrt = fma(ut, ir, q.srt), xrp = fma(up, ir, q.srp), xtp = fma(up, m[C_COTIR], q.stp);
  const double cross = fma(q.stp, xtp, fma(q.srp, xrp, q.srt * xrt));
  vis = fma(-0.5, cross, vis);
  const double div = c.dvr[t] + c.dvt[t] + c.dvp[t];
  double Np = fma(q.ap, div, fma(A.k.vp2, vis, fma(-A.k.difp, lap, accp)));
  double NT_ = fma(q.aT, div, fma(q.vT2, vis, fma(-(A.k.kap * q.be), lap, accT)));
  if (A.has_src) { Np -= A.src.f[0][t]; NT_ -= A.src.f[4][t]; }
  const double d0 = A.hasD ? A.D.f[0][t] : 0.0, d4 = A.hasD ? A.D.f[4][t] : 0.0;
  A.R.f[0][t] = fma(-A.tau, Np, -d0);
  A.R.f[4][t] = fma(-A.tau, NT_, -d4);
}

// ---------------------------------------------------------- rows at the faces

// Values of the two centres beside a face (c0 below, c1 above) that its rows use.
struct FaceC { double iv; int c0, c1; };
template <int C>
__device__ __forceinline__ FaceC face_load(const Geo<double>& g, const Coef<double>& c, int i, int j, int k) {
  FaceC q;
  q.c0 = C == 0 ? IC(g, i - 1, j, k) : C == 1 ? IC(g, i, j - 1, k) : IC(g, i, j, g.per ? wrapk(g, k - 1) : k - 1);
  q.c1 = IC(g, i, j, k);
  q.iv = 1.0 / (c.rho[q.c0] + c.rho[q.c1]);
  return q;
}
// the table row of a face of component C
template <int C>
__device__ __forceinline__ const double* face_tab(const Geo<double>& g, const Tabs& T, int i, int j) {
  return C == 0 ? T.r + (size_t)(i * g.nt + j) * NR : C == 1 ? T.t + (size_t)(i * (g.nt + 1) + j) * NT
                                                             : T.c + (size_t)(i * g.nt + j) * NC;
}
// the normal row: p weight wp (the one below is -wp), u weights w
template <int C>
__device__ __forceinline__ void face_normal(const K64& k, const double* m, double iv, double u, double& wp, double* w) {
  if (C == 0) {
    const double adv = u * k.hidr;
    wp = iv * m[R_WP];
    w[0] = fma(iv, m[R_F0], -adv); w[1] = iv * m[R_F1]; w[2] = fma(iv, m[R_F2], adv);
  } else if (C == 1) {
    const double adv = u * m[T_HADV];
    wp = iv * m[T_WP];
    w[0] = fma(iv, m[T_F0], -adv); w[1] = iv * m[T_F1]; w[2] = fma(iv, m[T_F2], adv);
  } else {
    const double adv = u * m[C_HMP];
    wp = iv * m[P_WP];
    w[0] = fma(iv, m[P_F], -adv); w[1] = iv * m[P_F2]; w[2] = fma(iv, m[P_F], adv);
  }
}
// the row along the transverse direction D; ua2 = the sum of the advecting
// velocity's two centre values
template <int C, int D>
__device__ __forceinline__ void face_trans(const K64& k, const double* m, double iv, double ua2, double* w) {
  double a, w0, w1, w2;
  if (C == 0 && D == 1) { a = m[R_QT]; w0 = m[R_T0]; w1 = m[R_TS]; w2 = m[R_T1]; }
  else if (C == 0) { a = m[R_QP]; w0 = w2 = m[R_P]; w1 = m[R_P2]; }
  else if (C == 1 && D == 0) { a = k.qidr; w0 = m[T_R0]; w1 = m[T_RS]; w2 = m[T_R1]; }
  else if (C == 1) { a = m[T_QP]; w0 = w2 = m[T_P]; w1 = m[T_P2]; }
  else if (D == 0) { a = k.qidr; w0 = m[P_R0]; w1 = m[P_RS]; w2 = m[P_R1]; }
  else { a = m[C_QMT]; w0 = m[P_T0]; w1 = m[P_TS]; w2 = m[P_T1]; }
  const double adv = ua2 * a;
  w[0] = fma(iv, w0, -adv); w[1] = iv * w1; w[2] = fma(iv, w2, adv);
}
template <int D>
__device__ __forceinline__ const double* ucen(const Coef<double>& c) { return D == 0 ? c.uc0 : D == 1 ? c.uc1 : c.uc2; }

__device__ __forceinline__ void store_normal(const Rows& o, int d, int t, double wp, const double* w) {
  double* p = o.f[d] + t;
  const long n = o.nf[d];
  p[0] = wp; p[n] = w[0]; p[2 * n] = w[1]; p[3 * n] = w[2];
}
__device__ __forceinline__ void store_trans(const Rows& o, int cc, int d, int t, const double* w) {
  const long n = o.nf[cc];
  double* p = o.s[cc] + 3 * trans_slot(cc, d) * n + t;
  p[0] = w[0]; p[n] = w[1]; p[2 * n] = w[2];
}

// velocity component C at an index beside its own face along direction D, with
// the ghosts of the walls
template <int C>
__device__ __forceinline__ double vel(const Geo<double>& g, const double* u, int i, int j, int k) {
  return C == 0 ? vr<2>(g, u, i, j, k) : C == 1 ? vt<2>(g, u, i, j, k) : vp<2>(g, u, i, j, k);
}

// R for the momentum row of component C on its faces, storing its three line
// rows: one thread per face, zero on wall faces (which are not unknowns).  48
// FP64 instructions, from about 150.
template <int C>
__global__ void __launch_bounds__(128) k_rhs_u(const __grid_constant__ Args A) {
  const Geo<double>& g = A.g;
  const int nj = g.nt + (C == 1), nk = C == 2 ? g.npf : g.np;
  const int k = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y,
            i = blockIdx.z * blockDim.z + threadIdx.z;
  if (k >= nk || j >= nj || i >= g.nr + (C == 0)) return;
  const int t = (i * nj + j) * nk + k;
  const bool wall = C == 0 ? (i == 0 || i == g.nr) : C == 1 ? (j == 0 || j == g.nt) : (!g.per && (k == 0 || k == g.np));
  if (wall) { A.R.f[1 + C][t] = 0.0; return; }
  const Coef<double>& c = A.c;
  const FaceC q = face_load<C>(g, c, i, j, k);
  const double* m = face_tab<C>(g, A.T, i, j);
  const double iv = q.iv;
  const double* U = A.ub.f[1 + C];
  const double u = U[t];
  constexpr int D1 = C == 0 ? 1 : 0, D2 = C == 2 ? 1 : 2;   // the transverse directions
  double wp, w[3];
  face_normal<C>(A.k, m, iv, u, wp, w);
  store_normal(A.rows, C, t, wp, w);
  const double* Pp = A.ub.f[0];
  double acc = wp * (Pp[q.c1] - Pp[q.c0]);
  acc = fma(w[0], vel<C>(g, U, i - (C == 0), j - (C == 1), k - (C == 2)),
            fma(w[1], u, fma(w[2], vel<C>(g, U, i + (C == 0), j + (C == 1), k + (C == 2)), acc)));
  const double s1 = ucen<D1>(c)[q.c0] + ucen<D1>(c)[q.c1], s2 = ucen<D2>(c)[q.c0] + ucen<D2>(c)[q.c1];
  face_trans<C, D1>(A.k, m, iv, s1, w);
  store_trans(A.rows, C, D1, t, w);
  acc = fma(w[0], vel<C>(g, U, i - (D1 == 0), j - (D1 == 1), k), fma(w[1], u, fma(w[2], vel<C>(g, U, i + (D1 == 0), j + (D1 == 1), k), acc)));
  face_trans<C, D2>(A.k, m, iv, s2, w);
  store_trans(A.rows, C, D2, t, w);
  acc = fma(w[0], vel<C>(g, U, i, j - (D2 == 1), k - (D2 == 2)),
            fma(w[1], u, fma(w[2], vel<C>(g, U, i, j + (D2 == 1), k + (D2 == 2)), acc)));
  double vis;   // the viscous terms of D_M over 1/(rho_0 + rho_1)
  if (C == 0) {
    // hydrostatic part: (1/rho_f) d p_ref/dr + g = (1 - b) e + g b, b = 1 - rho_ref,f / rho_f
    acc += fma((c.drho[q.c0] + c.drho[q.c1]) * iv, m[R_GE], m[R_E]);
    acc = fma(fma(s1, s1, s2 * s2), -m[R_QIR], acc);
    if (A.k.rot) acc = fma(-m[R_OM], s2, acc);
    vis = fma(u, m[R_V], fma(c.dvt[q.c1] + c.dvp[q.c1], m[R_Q1], (c.dvt[q.c0] + c.dvp[q.c0]) * m[R_Q0]));
  } else if (C == 1) {
    acc = fma(u * s1, m[T_HIR], acc);
    acc = fma(s2 * s2, -m[T_C], acc);
    if (A.k.rot) acc = fma(-m[T_OM], s2, acc);
    vis = fma(u, m[T_V], (c.dvr[q.c1] - c.dvr[q.c0]) * m[T_D]);
    vis = fma(c.dvp[q.c0], m[T_D0], fma(c.dvp[q.c1], m[T_D1], vis));
    vis = fma(c.uc0[q.c1] - c.uc0[q.c0], m[T_UR], vis);
  } else {
    acc = fma(u, fma(s2, m[C_HCOTIR], s1 * m[C_HIR]), acc);
    if (A.k.rot) acc = fma(m[P_OC], s2, fma(m[P_OS], s1, acc));
    vis = fma(u, m[P_V], ((c.dvr[q.c1] - c.dvr[q.c0]) + (c.dvt[q.c1] - c.dvt[q.c0])) * m[P_D]);
    vis = fma(c.uc0[q.c1] - c.uc0[q.c0], m[P_UR], fma(c.uc1[q.c1] - c.uc1[q.c0], m[P_UT], vis));
  }
  acc = fma(iv, vis, acc);
  if (A.has_src) acc -= A.src.f[1 + C][t];
  const double d = A.hasD ? A.D.f[1 + C][t] : 0.0;
  A.R.f[1 + C][t] = fma(-A.tau, acc, -d);
}

// Only the rows along direction D (a sweep called on its own): blockIdx.z walks
// the four kinds of points (centres, faces of u_r, u_theta, u_phi) in turn.
template <int D, int C>
__device__ __forceinline__ void face_rows(const Args& A, int i, int j, int k, int t) {
  const FaceC q = face_load<C>(A.g, A.c, i, j, k);
  const double* m = face_tab<C>(A.g, A.T, i, j);
  double wp, w[3];
  if (C == D) {
    face_normal<C>(A.k, m, q.iv, A.ub.f[1 + C][t], wp, w);
    store_normal(A.rows, C, t, wp, w);
  } else {
    face_trans<C, D>(A.k, m, q.iv, ucen<D>(A.c)[q.c0] + ucen<D>(A.c)[q.c1], w);
    store_trans(A.rows, C, D, t, w);
  }
}
template <int D>
__global__ void __launch_bounds__(128) k_rows(const __grid_constant__ Args A) {
  const Geo<double>& g = A.g;
  const int kind = blockIdx.y;
  const int ni = g.nr + (kind == 1), nj = g.nt + (kind == 2), nk = kind == 3 ? g.npf : g.np;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= ni * nj * nk) return;
  const int k = t % nk, j = (t / nk) % nj, i = t / (nk * nj);
  if (kind == 0) {
    const double* m = A.T.c + (size_t)(i * g.nt + j) * NC;
    const CenC q = cen_load(A.k, A.c, t);
    double s, u;
    cen_visc<D>(A.k, q, m, s, u);
    cen_store<D>(A.k, A.rows, q, m, cen_adv<D>(A.k, A.c, m, t), s, u, t);
    return;
  }
  if (kind == 1 && i > 0 && i < g.nr) face_rows<D, 0>(A, i, j, k, t);
  if (kind == 2 && j > 0 && j < g.nt) face_rows<D, 1>(A, i, j, k, t);
  if (kind == 3 && (g.per || (k > 0 && k < g.np))) face_rows<D, 2>(A, i, j, k, t);
}

}  // namespace f64
