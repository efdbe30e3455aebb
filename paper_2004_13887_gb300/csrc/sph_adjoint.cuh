// sph_adjoint.cuh -- reverse mode of one Picard iteration of the scheme of
// Section 2.2 (eqs. chapter3mainsd, splitting2, spl1-spl3), FP64.
//
// One iteration maps (a, b) = (U^n, U^{n+1,k}) to
//   out = b + x_phi,  x_phi = A_phi^{-1} x_theta,  x_theta = A_theta^{-1} x_r,
//   x_r = A_r^{-1} R,  R = -(b - a) - tau [N(Ubar) + G - S],  Ubar = (a + b)/2,
// with A_d = I + tau/2 D_d(Ubar) and every coefficient frozen at Ubar.  Given
// lambda = dJ/d out, the adjoint is
//   mu_phi = A_phi^{-T} lambda, mu_theta = A_theta^{-T} mu_phi, mu_r = A_r^{-T} mu_theta
//   dJ/db = lambda - mu_r + g/2,  dJ/da = mu_r + g/2,
//   g = grad over Ubar of  <mu_r, R(Ubar)> - sum_d <mu_d, A_d(Ubar) x_d>
// (the x_d and mu_d held fixed).  The transposed solves are the line solvers of
// sph_fp64_lines.cuh with TR = true.
//
// g is taken by hand-derived adjoints of the rows in sph_fp64.cuh.  A row of
// D_d enters both the right-hand side (applied to Ubar, weight -tau mu_r) and the
// line operator (applied to x_d, weight -tau/2 mu_d), with the same weights, so
// their cotangents add before the one pass back through the weights.  Two
// kernels per iteration, bound like the forward ones by their FP64
// instructions (sph_fp64.cuh): k_adj_u at the faces of each component (the
// momentum rows; what they give to the coefficient planes and to Ubar is added
// with FP64 atomics, which the L2 performs), then k_adj_c at the centres (the p-
// and T-rows, and everything back through the coefficients to Ubar).
// Measured on 96 x 192 x 192 cells, ms per iteration: 4.3 (k_adj_c 2.0, k_adj_u
// 0.71-0.80 a component) where recording the rows on a tape per thread and
// sweeping it back (370 nodes a row set in global memory) took 193; the adjoint
// of a step of two iterations 441 -> 29.9 ms.
#pragma once

namespace f64 {

// coefficient planes the momentum rows read: the accumulators of their cotangents
enum { L_RHO, L_DRHO, L_UC0, L_UC1, L_UC2, L_DVR, L_DVT, L_DVP, NL };

struct AdjArgs {
  Geo<double> g;
  K64 k;
  Tabs T;
  Coef<double> c;       // coefficient planes at Ubar
  CF<double> ub;        // Ubar
  double tau;
  CF<double> mu[3];     // mu_r (the right-hand side's weight too), mu_theta, mu_phi
  CF<double> x[3];      // the forward sweeps' solutions x_r, x_theta, x_phi
  double* lam[5];       // gradient over Ubar (added to)
  double* pl[NL];       // cotangents of the planes (zero before k_adj_u)
};

// add v to the cotangent of the value that an accessor with ghosts reads at
// (i, j, k): p and T (zero gradient at the walls), or velocity component C
// (ghost = 2 wall - interior; the wall value is a constant)
__device__ __forceinline__ void scat_c(const Geo<double>& g, double* lam, int i, int j, int k, double v) {
  const int kk = g.per ? wrapk(g, k) : clampi(k, 0, g.np - 1);
  atomicAdd(lam + IC(g, clampi(i, 0, g.nr - 1), clampi(j, 0, g.nt - 1), kk), v);
}
template <int C>
__device__ __forceinline__ void scat_v(const Geo<double>& g, double* lam, int i, int j, int k, double v) {
  if (C != 0 && (i < 0 || i >= g.nr)) { i = i < 0 ? 0 : g.nr - 1; v = -v; }
  if (C != 1 && (j < 0 || j >= g.nt)) { j = j < 0 ? 0 : g.nt - 1; v = -v; }
  if (g.per) k = wrapk(g, k);
  else if (C != 2 && (k < 0 || k >= g.np)) { k = k < 0 ? 0 : g.np - 1; v = -v; }
  atomicAdd(lam + face_idx(g, C, i, j, k), v);
}
// an increment's velocity component beside its face: homogeneous ghosts
template <int C>
__device__ __forceinline__ double vel0(const Geo<double>& g, const double* u, int i, int j, int k) {
  return C == 0 ? vr<1>(g, u, i, j, k) : C == 1 ? vt<1>(g, u, i, j, k) : vp<1>(g, u, i, j, k);
}

// the transverse row of component C along D: cotangents of 1/(rho_0 + rho_1) and
// of the advecting velocity's sum; Ubar's share is scattered
template <int C, int D>
__device__ __forceinline__ void adj_trans(const AdjArgs& A, const double* m, int i, int j, int k, int t, double iv,
                                          double ua2, double a, double u, double& civ, double& cua, double& cu) {
  const Geo<double>& g = A.g;
  constexpr int di = D == 0, dj = D == 1, dk = D == 2;
  double q, f0, f1, f2;
  if (C == 0 && D == 1) { q = m[R_QT]; f0 = m[R_T0]; f1 = m[R_TS]; f2 = m[R_T1]; }
  else if (C == 0) { q = m[R_QP]; f0 = f2 = m[R_P]; f1 = m[R_P2]; }
  else if (C == 1 && D == 0) { q = A.k.qidr; f0 = m[T_R0]; f1 = m[T_RS]; f2 = m[T_R1]; }
  else if (C == 1) { q = m[T_QP]; f0 = f2 = m[T_P]; f1 = m[T_P2]; }
  else if (D == 0) { q = A.k.qidr; f0 = m[P_R0]; f1 = m[P_RS]; f2 = m[P_R1]; }
  else { q = m[C_QMT]; f0 = m[P_T0]; f1 = m[P_TS]; f2 = m[P_T1]; }
  const double* U = A.ub.f[1 + C];
  const double* X = A.x[D].f[1 + C];
  const double cd = -0.5 * A.tau * A.mu[D].f[1 + C][t];
  const double zl = fma(a, vel<C>(g, U, i - di, j - dj, k - dk), cd * vel0<C>(g, X, i - di, j - dj, k - dk));
  const double zh = fma(a, vel<C>(g, U, i + di, j + dj, k + dk), cd * vel0<C>(g, X, i + di, j + dj, k + dk));
  const double z0 = fma(a, u, cd * X[t]);
  civ = fma(f0, zl, fma(f1, z0, fma(f2, zh, civ)));
  cua = fma(q, zh - zl, cua);
  const double adv = ua2 * q;
  scat_v<C>(g, A.lam[1 + C], i - di, j - dj, k - dk, a * fma(iv, f0, -adv));
  scat_v<C>(g, A.lam[1 + C], i + di, j + dj, k + dk, a * fma(iv, f2, adv));
  cu = fma(a, iv * f1, cu);
}

// the momentum rows of component C: one thread per face
template <int C>
__global__ void __launch_bounds__(128) k_adj_u(const __grid_constant__ AdjArgs A) {
  const Geo<double>& g = A.g;
  const int nj = g.nt + (C == 1), nk = C == 2 ? g.npf : g.np;
  const int k = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y,
            i = blockIdx.z * blockDim.z + threadIdx.z;
  if (k >= nk || j >= nj || i >= g.nr + (C == 0)) return;
  if (C == 0 ? (i == 0 || i == g.nr) : C == 1 ? (j == 0 || j == g.nt) : (!g.per && (k == 0 || k == g.np))) return;
  const int t = (i * nj + j) * nk + k;
  constexpr int D1 = C == 0 ? 1 : 0, D2 = C == 2 ? 1 : 2;   // the transverse directions
  const Coef<double>& c = A.c;
  const FaceC q = face_load<C>(g, c, i, j, k);
  const double* m = face_tab<C>(g, A.T, i, j);
  const double iv = q.iv;
  const double* U = A.ub.f[1 + C];
  const double* Pp = A.ub.f[0];
  const double u = U[t];
  const double a = -A.tau * A.mu[0].f[1 + C][t], cn = -0.5 * A.tau * A.mu[C].f[1 + C][t];
  double civ, cu, cs1 = 0.0, cs2 = 0.0;
  {
    // the normal row
    const double* X = A.x[C].f[1 + C];
    const double* Xp = A.x[C].f[0];
    double wp, w[3];
    face_normal<C>(A.k, m, iv, u, wp, w);
    constexpr int di = C == 0, dj = C == 1, dk = C == 2;
    const double zp = fma(a, Pp[q.c1] - Pp[q.c0], cn * (Xp[q.c1] - Xp[q.c0]));
    const double zm = fma(a, vel<C>(g, U, i - di, j - dj, k - dk), cn * vel0<C>(g, X, i - di, j - dj, k - dk));
    const double zn = fma(a, vel<C>(g, U, i + di, j + dj, k + dk), cn * vel0<C>(g, X, i + di, j + dj, k + dk));
    const double z0 = fma(a, u, cn * X[t]);
    const double fw = m[C == 0 ? R_WP : C == 1 ? T_WP : P_WP], f0 = m[C == 0 ? R_F0 : C == 1 ? T_F0 : P_F],
                 f1 = m[C == 0 ? R_F1 : C == 1 ? T_F1 : P_F2], f2 = m[C == 0 ? R_F2 : C == 1 ? T_F2 : P_F];
    civ = fma(fw, zp, fma(f0, zm, fma(f1, z0, f2 * zn)));
    cu = fma(a, w[1], (zn - zm) * (C == 0 ? A.k.hidr : C == 1 ? m[T_HADV] : m[C_HMP]));
    atomicAdd(A.lam[0] + q.c1, a * wp);
    atomicAdd(A.lam[0] + q.c0, -a * wp);
    scat_v<C>(g, A.lam[1 + C], i - di, j - dj, k - dk, a * w[0]);
    scat_v<C>(g, A.lam[1 + C], i + di, j + dj, k + dk, a * w[2]);
  }
  const double s1 = ucen<D1>(c)[q.c0] + ucen<D1>(c)[q.c1], s2 = ucen<D2>(c)[q.c0] + ucen<D2>(c)[q.c1];
  adj_trans<C, D1>(A, m, i, j, k, t, iv, s1, a, u, civ, cs1, cu);
  adj_trans<C, D2>(A, m, i, j, k, t, iv, s2, a, u, civ, cs2, cu);
  const double ai = a * iv;
  double vis;
  if (C == 0) {
    vis = fma(u, m[R_V], fma(c.dvt[q.c1] + c.dvp[q.c1], m[R_Q1], (c.dvt[q.c0] + c.dvp[q.c0]) * m[R_Q0]));
    vis = fma(c.drho[q.c0] + c.drho[q.c1], m[R_GE], vis);
    const double cd = ai * m[R_GE], v1 = ai * m[R_Q1], v0 = ai * m[R_Q0], a2 = -2.0 * a * m[R_QIR];
    atomicAdd(A.pl[L_DRHO] + q.c0, cd);
    atomicAdd(A.pl[L_DRHO] + q.c1, cd);
    atomicAdd(A.pl[L_DVT] + q.c0, v0);
    atomicAdd(A.pl[L_DVP] + q.c0, v0);
    atomicAdd(A.pl[L_DVT] + q.c1, v1);
    atomicAdd(A.pl[L_DVP] + q.c1, v1);
    cs1 = fma(a2, s1, cs1);
    cs2 = fma(a2, s2, fma(-a, m[R_OM], cs2));
    cu = fma(ai, m[R_V], cu);
    atomicAdd(A.pl[L_UC1] + q.c0, cs1);
    atomicAdd(A.pl[L_UC1] + q.c1, cs1);
    atomicAdd(A.pl[L_UC2] + q.c0, cs2);
    atomicAdd(A.pl[L_UC2] + q.c1, cs2);
  } else if (C == 1) {
    vis = fma(u, m[T_V], (c.dvr[q.c1] - c.dvr[q.c0]) * m[T_D]);
    vis = fma(c.dvp[q.c0], m[T_D0], fma(c.dvp[q.c1], m[T_D1], vis));
    vis = fma(c.uc0[q.c1] - c.uc0[q.c0], m[T_UR], vis);
    const double d = ai * m[T_D], r = ai * m[T_UR];
    atomicAdd(A.pl[L_DVR] + q.c0, -d);
    atomicAdd(A.pl[L_DVR] + q.c1, d);
    atomicAdd(A.pl[L_DVP] + q.c0, ai * m[T_D0]);
    atomicAdd(A.pl[L_DVP] + q.c1, ai * m[T_D1]);
    cs1 = fma(a * u, m[T_HIR], cs1);
    cs2 = fma(-2.0 * a * m[T_C], s2, fma(-a, m[T_OM], cs2));
    cu = fma(a * s1, m[T_HIR], fma(ai, m[T_V], cu));
    atomicAdd(A.pl[L_UC0] + q.c0, cs1 - r);
    atomicAdd(A.pl[L_UC0] + q.c1, cs1 + r);
    atomicAdd(A.pl[L_UC2] + q.c0, cs2);
    atomicAdd(A.pl[L_UC2] + q.c1, cs2);
  } else {
    vis = fma(u, m[P_V], ((c.dvr[q.c1] - c.dvr[q.c0]) + (c.dvt[q.c1] - c.dvt[q.c0])) * m[P_D]);
    vis = fma(c.uc0[q.c1] - c.uc0[q.c0], m[P_UR], fma(c.uc1[q.c1] - c.uc1[q.c0], m[P_UT], vis));
    const double d = ai * m[P_D], r = ai * m[P_UR], p = ai * m[P_UT], au = a * u;
    atomicAdd(A.pl[L_DVR] + q.c0, -d);
    atomicAdd(A.pl[L_DVR] + q.c1, d);
    atomicAdd(A.pl[L_DVT] + q.c0, -d);
    atomicAdd(A.pl[L_DVT] + q.c1, d);
    cs1 = fma(au, m[C_HIR], fma(a, m[P_OS], cs1));
    cs2 = fma(au, m[C_HCOTIR], fma(a, m[P_OC], cs2));
    cu = fma(a, fma(s2, m[C_HCOTIR], s1 * m[C_HIR]), fma(ai, m[P_V], cu));
    atomicAdd(A.pl[L_UC0] + q.c0, cs1 - r);
    atomicAdd(A.pl[L_UC0] + q.c1, cs1 + r);
    atomicAdd(A.pl[L_UC1] + q.c0, cs2 - p);
    atomicAdd(A.pl[L_UC1] + q.c1, cs2 + p);
  }
  atomicAdd(A.lam[1 + C] + t, cu);
  const double cr = -iv * iv * fma(a, vis, civ);
  atomicAdd(A.pl[L_RHO] + q.c0, cr);
  atomicAdd(A.pl[L_RHO] + q.c1, cr);
}

// the cotangents of a centre's coefficients
struct CenCot {
  double Pb, Tb, be, grr, gtt, gpp, srt, srp, stp, uc[3];
  double ap, aT, vT2;
};

// one direction of the p- and T-rows: a, b weight the right-hand side's rows
template <int D>
__device__ __forceinline__ void adj_cen(const AdjArgs& A, const CenC& q, const double* m, int i, int j, int k, int t,
                                        double a, double b, double e, double& vis, double& lap, CenCot& o) {
  const Geo<double>& g = A.g;
  constexpr int di = D == 0, dj = D == 1, dk = D == 2;
  const double cp = -0.5 * A.tau * A.mu[D].f[0][t], cT = -0.5 * A.tau * A.mu[D].f[4][t];
  const double hm = D == 0 ? A.k.hidr : m[D == 1 ? C_HMT : C_HMP];
  const double adv = cen_adv<D>(A.k, A.c, m, t);
  double s, u;
  cen_visc<D>(A.k, q, m, s, u);
  const double l0 = m[D == 0 ? C_L00 : D == 1 ? C_L10 : C_MP2], l1 = m[D == 0 ? C_L01 : D == 1 ? C_L11 : C_MP2];
  const double g0 = m[D == 0 ? C_G00 : D == 1 ? C_G10 : C_MP], g1 = m[D == 0 ? C_G01 : D == 1 ? C_G11 : C_MP];
  const double *Pp = A.ub.f[0], *TT = A.ub.f[4], *U = A.ub.f[1 + D];
  const double *Xp = A.x[D].f[0], *XT = A.x[D].f[4], *XU = A.x[D].f[1 + D];
  // the rows' operands: Ubar's (with the background) and the sweep solution's
  double dp = cpert<2>(g, Pp, i + di, j + dj, k + dk) - cpert<2>(g, Pp, i - di, j - dj, k - dk);
  const double Tm = cpert<2>(g, TT, i - di, j - dj, k - dk), T0 = TT[t], Tn = cpert<2>(g, TT, i + di, j + dj, k + dk);
  double dT = Tn - Tm;
  lap = fma(l1, Tn - T0, fma(l0, Tm - T0, lap));
  if (D == 0) { dp += g.dbgp[i]; dT += g.dbgT[i]; }
  const double xp = cpert<2>(g, Xp, i + di, j + dj, k + dk) - cpert<2>(g, Xp, i - di, j - dj, k - dk);
  const double Xm = cpert<2>(g, XT, i - di, j - dj, k - dk), X0 = XT[t], Xn = cpert<2>(g, XT, i + di, j + dj, k + dk);
  const double xl = fma(l1, Xn - X0, l0 * (Xm - X0));
  const int f0 = face_idx(g, D, i, j, k);
  const int f1 = face_idx(g, D, i + di, j + dj, D == 2 && g.per ? wrapk(g, k + 1) : k + dk);
  const double u0 = U[f0], u1 = U[f1], x0 = XU[f0], x1 = XU[f1];
  const double dx = fma(g1, x1, -(g0 * x0)), vx = fma(s, x0, u * x1);
  vis = fma(s, u0, fma(u, u1, vis));
  // cotangents of the row weights
  const double ce = fma(cp, A.k.vp2, cT * q.vT2);
  const double cs = fma(e, u0, ce * x0), cu = fma(e, u1, ce * x1);
  o.ap = fma(cp, dx, o.ap);
  o.aT = fma(cT, dx, o.aT);
  o.vT2 = fma(cT, vx, o.vT2);
  o.be = fma(-A.k.kap * cT, xl, o.be);
  o.uc[D] = fma(hm, fma(a, dp, fma(b, dT, fma(cp, xp, cT * (Xn - Xm)))), o.uc[D]);
  const double cl = cs + cu, cm = cs - cu;
  if (D == 0) {
    const double z = -m[C_HIR] * cl;
    o.gtt += z;
    o.gpp += z;
    o.grr = fma(A.k.idr, cm, o.grr);
  } else if (D == 1) {
    const double z = m[C_QIR] * cl;
    o.gpp = fma(-z, m[C_COT2], o.gpp);
    o.srt += z;
    o.gtt = fma(m[C_MT], cm, o.gtt);
  } else {
    const double z = m[C_QIR] * cl;
    o.stp = fma(z, m[C_COT], o.stp);
    o.srp += z;
    o.gpp = fma(m[C_MP], cm, o.gpp);
  }
  // Ubar as the right-hand side's operand
  const double aa = a * adv, bb = b * adv, ct = -fma(A.k.difp, a, A.k.kap * q.be * b);
  scat_c(g, A.lam[0], i + di, j + dj, k + dk, aa);
  scat_c(g, A.lam[0], i - di, j - dj, k - dk, -aa);
  scat_c(g, A.lam[4], i + di, j + dj, k + dk, fma(ct, l1, bb));
  scat_c(g, A.lam[4], i - di, j - dj, k - dk, fma(ct, l0, -bb));
  atomicAdd(A.lam[4] + t, -ct * (l0 + l1));
  atomicAdd(A.lam[1 + D] + f0, e * s);
  atomicAdd(A.lam[1 + D] + f1, e * u);
}

// The p- and T-rows at the centres and the coefficients' adjoint: one thread
// per centre, after k_adj_u has added the planes' cotangents.
__global__ void __launch_bounds__(128) k_adj_c(const __grid_constant__ AdjArgs A) {
  const Geo<double>& g = A.g;
  const int k = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y,
            i = blockIdx.z * blockDim.z + threadIdx.z;
  if (k >= g.np || j >= g.nt || i >= g.nr) return;
  const int t = IC(g, i, j, k);
  const double* m = A.T.c + (size_t)(i * g.nt + j) * NC;
  const Coef<double>& c = A.c;
  const K64& K = A.k;
  const CenC q = cen_load(K, c, t);
  const double a = -A.tau * A.mu[0].f[0][t], b = -A.tau * A.mu[0].f[4][t];
  const double e = fma(a, K.vp2, b * q.vT2);        // cotangent of the viscous sum
  const double div = c.dvr[t] + c.dvt[t] + c.dvp[t];
  CenCot o;
  o.Pb = o.Tb = o.be = o.grr = o.gtt = o.gpp = o.srt = o.srp = o.stp = 0.0;
  o.uc[0] = A.pl[L_UC0][t]; o.uc[1] = A.pl[L_UC1][t]; o.uc[2] = A.pl[L_UC2][t];
  o.ap = a * div;
  o.aT = b * div;
  o.vT2 = 0.0;
  double vis = 0.0, lap = g.lapT[i];
  adj_cen<0>(A, q, m, i, j, k, t, a, b, e, vis, lap, o);
  adj_cen<1>(A, q, m, i, j, k, t, a, b, e, vis, lap, o);
  adj_cen<2>(A, q, m, i, j, k, t, a, b, e, vis, lap, o);
  const double ir = m[C_IR], cotir = m[C_COTIR];
  {
    // -1/2 cross of the viscous sum
    const double ut = c.uc1[t], up = c.uc2[t], he = -0.5 * e;
    const double xrt = fma(ut, ir, q.srt), xrp = fma(up, ir, q.srp), xtp = fma(up, cotir, q.stp);
    vis = fma(-0.5, fma(q.stp, xtp, fma(q.srp, xrp, q.srt * xrt)), vis);
    o.srt = fma(he, q.srt + xrt, o.srt);
    o.srp = fma(he, q.srp + xrp, o.srp);
    o.stp = fma(he, q.stp + xtp, o.stp);
    o.uc[1] = fma(he * q.srt, ir, o.uc[1]);
    o.uc[2] = fma(he, fma(q.srp, ir, q.stp * cotir), o.uc[2]);
  }
  // a_p = gamma Pb + vp2 t3, a_T = (gamma-1) Tb + vT2 t3, vT2 = 2 mu beta, t3 = tr G / 3
  const double t3 = (q.grr + q.gtt + q.gpp) * (1.0 / 3.0);
  o.vT2 = fma(b, vis, fma(t3, o.aT, o.vT2));
  o.be = fma(K.mu2, o.vT2, fma(-K.kap * b, lap, o.be));
  o.Pb = K.gm * o.ap;
  o.Tb = K.gm1 * o.aT;
  const double ct = fma(K.vp2, o.ap, q.vT2 * o.aT) * (1.0 / 3.0);
  o.grr += ct;
  o.gtt += ct;
  o.gpp += ct;
  // the coefficients of the centre back to Ubar
  const double cdiv = fma(a, q.ap, b * q.aT);
  const double cdr = A.pl[L_DVR][t] + cdiv, cdt = A.pl[L_DVT][t] + cdiv, cdp = A.pl[L_DVP][t] + cdiv;
  {
    const double iT = 1.0 / c.Tb[t], iP = 1.0 / c.Pb[t], cr = A.pl[L_RHO][t], cd = A.pl[L_DRHO][t];
    const double w = iT * m[C_IT];
    const double lp = fma(cd, g.Tcen[i] * w, fma(cr, iT * K.iRg, fma(-o.be * q.be, iP, o.Pb)));
    const double lT = fma(o.be, iP * K.gm1, fma(-cd, fma(g.pcen[i], w, c.drho[t] * iT), fma(-cr, c.rho[t] * iT, o.Tb)));
    atomicAdd(A.lam[0] + t, lp);
    atomicAdd(A.lam[4] + t, lT);
  }
  const double cur = 0.5 * fma(ir, o.gtt + o.gpp, o.uc[0]);
  const double cut = 0.5 * fma(cotir, o.gpp, fma(-ir, o.srt, o.uc[1]));
  const double cup = 0.5 * fma(-ir, o.srp, fma(-cotir, o.stp, o.uc[2]));
  const double zr = K.idr * (o.grr + cdr), zt = m[C_MT] * (o.gtt + cdt), zp = m[C_MP] * (o.gpp + cdp);
  const int kp = g.per ? wrapk(g, k + 1) : k + 1;
  atomicAdd(A.lam[1] + IRf(g, i, j, k), fma(-m[C_E00], cdr, cur - zr));
  atomicAdd(A.lam[1] + IRf(g, i + 1, j, k), fma(m[C_E01], cdr, cur + zr));
  atomicAdd(A.lam[2] + ITf(g, i, j, k), fma(-m[C_E10], cdt, cut - zt));
  atomicAdd(A.lam[2] + ITf(g, i, j + 1, k), fma(m[C_E11], cdt, cut + zt));
  atomicAdd(A.lam[3] + IPf(g, i, j, k), cup - zp);
  atomicAdd(A.lam[3] + IPf(g, i, j, kp), cup + zp);
  const double qt = m[C_QMT], qp = m[C_QMP], qr = K.qidr;
  const double rt = qr * o.srt, tr = qt * o.srt, rp = qr * o.srp, pr = qp * o.srp, tp = qt * o.stp, pt = qp * o.stp;
#pragma unroll
  for (int s = 0; s < 2; s++) {
    scat_v<1>(g, A.lam[2], i + 1, j + s, k, rt);
    scat_v<1>(g, A.lam[2], i - 1, j + s, k, -rt);
    scat_v<0>(g, A.lam[1], i + s, j + 1, k, tr);
    scat_v<0>(g, A.lam[1], i + s, j - 1, k, -tr);
    scat_v<2>(g, A.lam[3], i + 1, j, k + s, rp);
    scat_v<2>(g, A.lam[3], i - 1, j, k + s, -rp);
    scat_v<0>(g, A.lam[1], i + s, j, k + 1, pr);
    scat_v<0>(g, A.lam[1], i + s, j, k - 1, -pr);
    scat_v<2>(g, A.lam[3], i, j + 1, k + s, tp);
    scat_v<2>(g, A.lam[3], i, j - 1, k + s, -tp);
    scat_v<1>(g, A.lam[2], i, j + s, k + 1, pt);
    scat_v<1>(g, A.lam[2], i, j + s, k - 1, -pt);
  }
}

// y += s * x over n elements
__global__ void k_axpy(long n, double s, const double* __restrict__ x, double* __restrict__ y) {
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < n; e += (long)gridDim.x * blockDim.x) y[e] += s * x[e];
}

}  // namespace f64
