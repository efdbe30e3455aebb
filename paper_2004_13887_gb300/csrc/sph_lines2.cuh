// sph_lines2.cuh -- the sweeps of the mixed mode over many lines: one lane per line
// and side, block Thomas from both ends in FP32 (eqs. spl1-spl3: (I + h D_d) x = r, h =
// tau/2, with the rows assembled from Ubar's planes).
//
// Along r and theta the lanes of a warp hold 32 lines adjacent in phi (the last of a
// phi row and the first of the next side by side), so every load and store of the
// chain is coalesced as it stands: no lane exchanges and no reduction across lanes --
// 340 instructions a cell along r against 850 in the partitioned solver's phi lines
// (sph_lines.cuh), which is the better one only where there are too few lines to
// fill the SMs (it has 4 to 128 lanes a line).  Two warps of a block take the two
// sides of the same lines; q = n/2 is the middle cell of a walled line:
//   top, cells 0 .. q-1, unknowns (p, T) of a cell and u on its upper face m + 1:
//     S_m = B_m - A_m E_{m-1}, E_m = S_m^{-1} C_m, g_m = S_m^{-1} (r_m - A_m g_{m-1}),
//     x_m = g_m - E_m x_{m+1};
//   bottom, cells n-1 .. q+1, unknowns (p, T) of a cell and u on its lower face m: the
//     same elimination of the line turned round (L, B, U of form_down);
//   the middle cell's p- and T-rows and the u-rows the sides left close the line
//     (meet), then each side substitutes outwards.
// (Both sides with u on the upper face, meeting in a 3x3 system, had up to 4.7 times
// the one-sided solver's error in u on long stiff lines: from below, a cell's
// pressure is then eliminated before the face that its flux leaves by.  Against FP64,
// lines of 512 and 200 stiff cells along r, smooth right-hand side: 1.7e-3 and 1.6e-4
// then, 2.9e-4 and 6.3e-5 now, 3.9e-4 and 7.8e-5 one-sided.)  Any length n >= 4.  (E, g)
// of a side's cells go to a scratch region of the block (12 floats a cell,
// lane-interleaved: 128-byte rows), read back in reverse and then discarded from L2.
#pragma once

#include "sph_blk3.cuh"

// Lines from which these kernels are the faster ones along r and theta, where the
// partitioned solver takes the length (lines of 192 cells: from more), and lines and
// cells from which they are where it does not (the measurements: lines2_use).
#define LINES2_MIN 10240
#define LINES2_MIN_192 12288
#define LINES2_MIN_OTHER 1024
#define LINES2_MIN_CELLS 4
#ifndef LINES2_MINB
#define LINES2_MINB 8
#endif

namespace lines2 {

using namespace blk3;

// FP32 tables, rounded once from FP64.  Per cell of a block line (along r: per i;
// along theta: per (i, j)); face entries are those of face m + 1, B_FS the sum of the
// three viscous weights, of which B_F0 and B_F2 are the outer two.
enum { B_G0, B_G1, B_K0, B_K1, B_LIN, B_COT2, B_M, B_HM, B_WP, B_F0, B_FS, B_F2, NB };
// per cell of a scalar line: off-diagonal, diagonal and off-diagonal weights per
// 1/(rho_0 + rho_1) (their sum is zero), advection factor
enum { S_W0, S_W1, S_W2, S_Q, NS };
struct Tabs {
  float* b[3];       // block lines along r (nr entries), theta (nr nt), phi (nr nt, one entry a line)
  float* s[3][2];    // scalar lines along r (nr, both kinds the same), theta (kind 1: (nr+1) nt; kind 2: nr nt),
                     // phi (one entry a line; kind 1: (nr+1) nt, kind 2: nr (nt+1))
};
inline size_t tabs_floats(int nr, int nt) {
  const size_t n2 = (size_t)nr * nt, nr2 = (size_t)(nr + 1) * nt, nt2 = (size_t)nr * (nt + 1);
  return NB * (nr + 2 * n2) + NS * (nr + 2 * nr2 + n2 + nt2);
}
inline Tabs tabs_of(float* p, int nr, int nt) {
  const size_t n2 = (size_t)nr * nt, nr2 = (size_t)(nr + 1) * nt;
  Tabs T;
  T.b[0] = p; p += (size_t)NB * nr;
  T.b[1] = p; p += NB * n2;
  T.b[2] = p; p += NB * n2;
  T.s[0][0] = T.s[0][1] = p; p += (size_t)NS * nr;
  T.s[1][0] = p; p += NS * nr2;
  T.s[1][1] = p; p += NS * n2;
  T.s[2][0] = p; p += NS * nr2;
  T.s[2][1] = p;
  return T;
}

struct Args {
  Geo<float> g;
  Coef<float> c;
  CF<float> ub, rhs;
  MF<float> x;                      // increments (update = 0)
  int update, norms;                // phi: uk = base + x; accumulate the squares of x
  CF<double> base;
  MF<double> uk;
  double* acc;
  Tabs T;
  float h, hgm, hgm1, hvp2, hmu2;   // tau/2 and its products with gamma, gamma - 1, 2 mu (gamma - 1), 2 mu
  float gm1, iRg;
  float* scr;                       // per block: 12 (block lines; 21 cyclic) or 2 (scalar; 3) rows of 32 floats a cell
  int nb0, nb1;                     // blocks of the block lines, and of kind 1
  int* flag;
};

template <int D> __device__ __forceinline__ int len(const Geo<float>& g) { return D == 0 ? g.nr : g.nt; }
// flat index of centre m of the line (a, b), and of its faces along D
template <int D> __device__ __forceinline__ int ic_of(const Geo<float>& g, int a, int b, int m) {
  return D == 0 ? IC(g, m, a, b) : IC(g, a, m, b);
}
template <int D> __device__ __forceinline__ int fx_of(const Geo<float>& g, int a, int b, int m) {
  return D == 0 ? IRf(g, m, a, b) : ITf(g, a, m, b);
}

struct Th { float Pb, Tb, rho, be; };
template <typename Consts>
__device__ __forceinline__ Th thermo(const Consts& A, int i, float pp, float Tp) {
  Th t;
  t.Pb = A.g.pcen[i] + pp;
  t.Tb = A.g.Tcen[i] + Tp;
  t.rho = t.Pb * A.iRg * __fdividef(1.f, t.Tb);
  t.be = A.gm1 * t.Tb * __fdividef(1.f, t.Pb);
  return t;
}

// The p- and T-rows of a cell from the values it reads (q0, q1: its table entry; th:
// its thermodynamics; ulo, uhi: Ubar's u_D on its faces; the gradients; s1, s2: the
// cross sums): their p and T columns below (Ab), at (Bb) and above (Cb), their u
// columns of the face below (in Ab) and above (in Bb).
template <int D, typename Consts>
__device__ __forceinline__ void form_cell(const Consts& A, const float4& q0, const float4& q1, const Th& th, float ulo,
                                          float uhi, float grr, float gtt, float gpp, float s1, float s2, float* Ab,
                                          float* Bb, float* Cb) {
  const float G0 = q0.x, G1 = q0.y, K0 = q0.z, K1 = q0.w, LIN = q1.x, COT2 = q1.y, MD = q1.z, HM = q1.w;
  const float t3 = (grr + gtt + gpp) * (1.f / 3.f);
  const float vT = A.hmu2 * th.be, hbe = A.h * th.be;
  const float ap = fmaf(A.hvp2, t3, A.hgm * th.Pb), aT = fmaf(vT, t3, A.hgm1 * th.Tb);
  const float adv = A.h * HM * 0.5f * (ulo + uhi);
  const float lin = (D == 0 ? gtt + gpp : D == 1 ? fmaf(gpp, COT2, -s1) : fmaf(s2, COT2, s1)) * LIN;
  const float m0 = (D == 0 ? grr : D == 1 ? gtt : gpp) * MD, vs = lin + m0, vu = lin - m0;
  Ab[0] = -adv; Ab[1] = A.hgm1 * K0; Ab[2] = fmaf(-ap, G0, A.hvp2 * vs);
  Ab[4] = fmaf(hbe, K0, -adv); Ab[5] = fmaf(-aT, G0, vT * vs);
  Cb[0] = adv; Cb[1] = A.hgm1 * K1; Cb[4] = fmaf(hbe, K1, adv);
  Bb[0] = 1.f; Bb[1] = -(Ab[1] + Cb[1]); Bb[2] = fmaf(ap, G1, A.hvp2 * vu);
  Bb[4] = 1.f - (Ab[4] + Cb[4]); Bb[5] = fmaf(aT, G1, vT * vu);
  // the T column's row sums, 0 and 1, hold exactly: where conduction makes the
  // entries large, their rounding would otherwise act on smooth fields
  Cb[1] = -Bb[1] - Ab[1];
  Cb[4] = (1.f - Bb[4]) - Ab[4];
  Bb[3] = Bb[7] = 0.f;
}
// The row of a face between two cells whose densities add up to rs (q2: its table
// entry, HM: its direction's half metric factor, u: Ubar's u_D on it; y: its
// right-hand side): u on the face below, on it and above; returns the weight of p
// above (below: minus that).  The whole row is divided by the sum of its u weights, 1
// + h FS / rs, so that they add up to 1 and hold that exactly, as in the T column (the
// sum itself is lost in the last bits of weights of some thousand where the row is stiff).
template <typename Consts>
__device__ __forceinline__ float form_face(const Consts& A, const float4& q2, float HM, float rs, float u, float* f, float* y) {
  const float i = __fdividef(1.f, fmaf(A.h, q2.z, rs)), hv = A.h * i, r = rs * i, av = A.h * u * HM * r;
  f[0] = fmaf(hv, q2.y, -av);
  f[1] = 1.f - (f[0] + fmaf(hv, q2.w, av));
  f[2] = (1.f - f[1]) - f[0];
  *y *= r;
  return hv * q2.x;
}
// The blocks of a cell with its face m + 1 (rho1: the density beyond it; face: it is
// an unknown) and its right-hand side y.
template <int D, typename Consts>
__device__ __forceinline__ void form(const Consts& A, const float4& q0, const float4& q1, const float4& q2, const Th& th,
                                     float rho1, bool face, float ulo, float uhi, float grr, float gtt, float gpp, float s1,
                                     float s2, float* Ab, float* Bb, float* Cb, float* y) {
  form_cell<D>(A, q0, q1, th, ulo, uhi, grr, gtt, gpp, s1, s2, Ab, Bb, Cb);
  if (face) {
    float f[3];
    const float wp = form_face(A, q2, q1.w, th.rho + rho1, uhi, f, y + 2);
    Ab[8] = f[0];
    Bb[6] = -wp; Bb[8] = f[1];
    Cb[6] = wp; Cb[8] = f[2];
  } else {                                              // the last cell of a walled line
    Ab[8] = 0.f;
    Bb[6] = 0.f; Bb[8] = 1.f;
    Cb[6] = Cb[8] = 0.f;
  }
}
// The blocks of a cell with its face m (q2: that face's entry; rho0: the density
// below it), in the order of an elimination from the line's upper end: L couples to
// the cell above, U to the one below.  L, B, U have the zeros of form's A, B, C.
template <int D, typename Consts>
__device__ __forceinline__ void form_down(const Consts& A, const float4& q0, const float4& q1, const float4& q2, const Th& th,
                                          float rho0, float ulo, float uhi, float grr, float gtt, float gpp, float s1,
                                          float s2, float* L, float* B, float* U, float* y) {
  float a[9], c[9], f[3];
  form_cell<D>(A, q0, q1, th, ulo, uhi, grr, gtt, gpp, s1, s2, a, B, c);
  L[0] = c[0]; L[1] = c[1]; L[2] = B[2]; L[4] = c[4]; L[5] = B[5];
  B[2] = a[2]; B[5] = a[5];
  U[0] = a[0]; U[1] = a[1]; U[4] = a[4];
  const float wp = form_face(A, q2, q1.w, th.rho + rho0, ulo, f, y + 2);
  L[8] = f[2];
  B[6] = wp; B[8] = f[1];
  U[6] = -wp; U[8] = f[0];
}

template <typename R>
__device__ __forceinline__ void inverse_or_nan(const R* S, R* I, int* bad) {
  if (!inv3(S, I)) {
    *bad |= FLAG_SINGULAR;
#pragma unroll
    for (int q = 0; q < 9; q++) I[q] = R(NAN);
  }
}

// The row of a scalar line's cell (w: its table entry, rs, us: the sums of the two
// centres' densities and advecting velocities): below, at, above, with the sum 1
// exact as in the block lines' rows.
__device__ __forceinline__ float3 form_scalar(float h, const float4& w, float rs, float us) {
  const float hv = __fdividef(h, rs), adv = h * us * w.w, a = fmaf(hv, w.x, -adv), b = 1.f - (a + fmaf(hv, w.z, adv));
  return make_float3(a, b, (1.f - b) - a);
}

// One cell of a side's elimination: (E, g[, H]) from its blocks and the cell
// before's.  first: the side's first cell.  REV (the bottom side of a cyclic line):
// from form's blocks with A and C in each other's place.
template <bool REV, bool CYC>
__device__ __forceinline__ void cell_step(float* Ab, float* Bb, float* Cb, float* y, bool first, float* E, float* gv,
                                          float* H, int* bad) {
  const float* L = REV ? Cb : Ab;
  const float* Un = REV ? Ab : Cb;
  constexpr unsigned ML = REV ? M_C : M_A, MU = REV ? M_A : M_C;
  if (!CYC && first) { Bb[0] += L[0]; Bb[1] += L[1]; Bb[4] += L[4]; }   // zero-gradient ghosts of p and T
  float Hs[9];
  if (!first) {
    sub_mul<ML, 3>(L, E, Bb);
    sub_mul<ML, 1>(L, gv, y);
  }
  if (CYC) {
#pragma unroll
    for (int q = 0; q < 9; q++) Hs[q] = 0.f;
    if (first) {
#pragma unroll
      for (int q = 0; q < 9; q++) if (ML >> q & 1) Hs[q] = L[q];   // couples to the ring's last cell
    } else {
      sub_mul<ML, 3>(L, H, Hs);
    }
  }
  float Si[9];
  inverse_or_nan(Bb, Si, bad);
  mul_sparse<MU>(Si, Un, E);
  mv(Si, y, gv);
  if (CYC) mul_sparse<M_ALL>(Si, Hs, H);
}

// The p- and T-rows of a walled line's middle cell, and their right-hand sides.
struct Mid { float a[9], b[9], c[9], y[2]; };

// Where the sides of a walled line meet: the middle cell's p and T (z[0], z[1]) and u
// on its faces, below (z[2]) and above (z[3]), from its rows and what the sides left:
// (p, T, u) of the cell below (its u the middle cell's lower face) is gt - Et (p, T,
// u above), of the cell above gb - Eb (p, T, u below).
__device__ __forceinline__ void meet(const float* Et, const float* gt, const float* Eb, const float* gb, const Mid& M,
                                     float* z, int* bad) {
  // u below over (p, T), u above eliminated: pv v = vr - vp p - vt T
  const float vp = fmaf(-Et[8], Eb[6], Et[6]), vt = fmaf(-Et[8], Eb[7], Et[7]), vr = fmaf(-Et[8], gb[2], gt[2]),
              pv = fmaf(-Et[8], Eb[8], 1.f), iv = __fdividef(1.f, pv);
  float P[2], T[2], R[2];
#pragma unroll
  for (int r = 0; r < 2; r++) {
    float V = M.a[3 * r + 2], W = M.b[3 * r + 2];
    P[r] = r ? 0.f : M.b[0];
    T[r] = M.b[3 * r + 1];
    R[r] = M.y[r];
#pragma unroll
    for (int k = 0; k < 2; k++) {      // the p and T of the cells below and above
      if (r > k) continue;             // (no p in the T-row)
      const float a = -M.a[3 * r + k], c = -M.c[3 * r + k];
      P[r] = fmaf(a, Et[3 * k], P[r]); T[r] = fmaf(a, Et[3 * k + 1], T[r]);
      W = fmaf(a, Et[3 * k + 2], W); R[r] = fmaf(a, gt[k], R[r]);
      P[r] = fmaf(c, Eb[3 * k], P[r]); T[r] = fmaf(c, Eb[3 * k + 1], T[r]);
      V = fmaf(c, Eb[3 * k + 2], V); R[r] = fmaf(c, gb[k], R[r]);
    }
    P[r] = fmaf(-W, Eb[6], P[r]); T[r] = fmaf(-W, Eb[7], T[r]); V = fmaf(-W, Eb[8], V); R[r] = fmaf(-W, gb[2], R[r]);
    const float f = V * iv;
    P[r] = fmaf(-f, vp, P[r]); T[r] = fmaf(-f, vt, T[r]); R[r] = fmaf(-f, vr, R[r]);
  }
  const float iT = __fdividef(1.f, T[1]), f = T[0] * iT, pp = fmaf(-f, P[1], P[0]);
  if (pv == 0.f || T[1] == 0.f || pp == 0.f || !isfinite(pv) || !isfinite(T[1]) || !isfinite(pp)) *bad |= FLAG_SINGULAR;
  z[0] = __fdividef(fmaf(-f, R[1], R[0]), pp);
  z[1] = fmaf(-P[1], z[0], R[1]) * iT;
  z[2] = fmaf(-vt, z[1], fmaf(-vp, z[0], vr)) * iv;
  z[3] = fmaf(-Eb[8], z[2], fmaf(-Eb[7], z[1], fmaf(-Eb[6], z[0], gb[2])));
}

// Values a lane will need some cells ahead go to its own words of a ring in shared
// memory by asynchronous 4-byte copies (128 bytes a warp and value), so that the
// loads of several cells are in flight without registers (block lines along r of
// 128 x 256 x 256: 296 us with one cell ahead in registers, 235 with the ring; what
// bounds it now is L2 traffic, 2.4 GB at 10 TB/s, 96 of its 150 bytes a cell the
// factors).  Every lane reads only what it copied itself, so its
// own wait is enough; a group is committed per cell, empty past the end.
__device__ __forceinline__ void cpa(float* dst, const float* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cpa_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cpa_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// (measured with r and theta sweeps of 128 x 256 x 256: 4 and 8 cells 334 and 376
// us; 3 and 6 326 and 400; 6 and 12, which leave fewer blocks an SM, 362 and 397)
constexpr int FWD = 4, BACK = 8;     // cells ahead in the elimination, in the substitution
constexpr int RING = BACK * 12 > FWD * 10 ? BACK * 12 : FWD * 10;   // 32-float rows of a warp's ring (block lines)
enum { V_P, V_T, V_GRR, V_GTT, V_GPP, V_R0, V_R4, V_U, V_RU, V_S1, NV };

// Elimination of one side's cnt cells along r or theta: SIDE 0 from the first cell,
// each with its face m + 1, SIDE 1 from the last, each with its face m.  The cell after
// them is the middle one; SIDE 0 leaves its rows.  ring: this lane's column of the warp's ring.
template <int D, int SIDE>
__device__ __forceinline__ void eliminate(const Args& A, int a, int b, int n, int cnt, float* ring, float* scr, float* E,
                                          float* gv, Mid* mid, int* bad) {
  const Geo<float>& g = A.g;
  auto cell = [&](int s) { return SIDE ? n - 1 - s : s; };
  auto bgi = [&](int m) { return D == 0 ? m : a; };      // radial index of cell m
  auto row = [&](int m) { return reinterpret_cast<const float4*>(A.T.b[D] + (size_t)NB * (D == 0 ? m : a * g.nt + m)); };
  // the cells of this side and the middle one, each with the face not seen yet
  auto issue = [&](int s) {
    if (s <= cnt) {
      const int m = cell(s), c = ic_of<D>(g, a, b, m), f = fx_of<D>(g, a, b, SIDE ? m : m + 1);
      float* w = ring + (s % FWD) * (NV * 32);
      cpa(w + V_P * 32, A.ub.f[0] + c); cpa(w + V_T * 32, A.ub.f[4] + c);
      cpa(w + V_GRR * 32, A.c.grr + c); cpa(w + V_GTT * 32, A.c.gtt + c); cpa(w + V_GPP * 32, A.c.gpp + c);
      cpa(w + V_R0 * 32, A.rhs.f[0] + c); cpa(w + V_R4 * 32, A.rhs.f[4] + c);
      cpa(w + V_U * 32, A.ub.f[1 + D] + f); cpa(w + V_RU * 32, A.rhs.f[1 + D] + f);
      if (D == 1) cpa(w + V_S1 * 32, A.c.srt + c);
    }
    cpa_commit();
  };
#pragma unroll
  for (int s = 0; s < FWD; s++) issue(s);
  float uf = A.ub.f[1 + D][fx_of<D>(g, a, b, SIDE ? n : 0)];
  cpa_wait<FWD - 1>();
  Th th = thermo(A, bgi(cell(0)), ring[V_P * 32], ring[V_T * 32]);
  for (int s = 0; s < cnt; s++) {
    const int m = cell(s);
    const float4 q0 = row(m)[0], q1 = row(m)[1], q2 = row(SIDE ? m - 1 : m)[2];
    cpa_wait<FWD - 2>();                                  // cells s and s + 1 have arrived
    const float* w = ring + (s % FWD) * (NV * 32);
    const float* w1 = ring + ((s + 1) % FWD) * (NV * 32);
    const Th t1 = thermo(A, bgi(cell(s + 1)), w1[V_P * 32], w1[V_T * 32]);
    const float u = w[V_U * 32], grr = w[V_GRR * 32], gtt = w[V_GTT * 32], gpp = w[V_GPP * 32],
                s1 = D == 1 ? w[V_S1 * 32] : 0.f;
    float y[3] = {w[V_R0 * 32], w[V_R4 * 32], w[V_RU * 32]}, Ab[9], Bb[9], Cb[9];
    if (SIDE) form_down<D>(A, q0, q1, q2, th, t1.rho, u, uf, grr, gtt, gpp, s1, 0.f, Ab, Bb, Cb, y);
    else form<D>(A, q0, q1, q2, th, t1.rho, true, uf, u, grr, gtt, gpp, s1, 0.f, Ab, Bb, Cb, y);
    cell_step<false, false>(Ab, Bb, Cb, y, s == 0, E, gv, nullptr, bad);
    issue(s + FWD);
    uf = u;
    th = t1;
    float* sp = scr + (size_t)m * (12 * 32);
#pragma unroll
    for (int q = 0; q < 9; q++) sp[q * 32] = E[q];
#pragma unroll
    for (int q = 0; q < 3; q++) sp[(9 + q) * 32] = gv[q];
  }
  if (SIDE == 0) {
    const float* w = ring + (cnt % FWD) * (NV * 32);      // (arrived with cell cnt - 1)
    form_cell<D>(A, row(cnt)[0], row(cnt)[1], th, uf, w[V_U * 32], w[V_GRR * 32], w[V_GTT * 32], w[V_GPP * 32],
                 D == 1 ? w[V_S1 * 32] : 0.f, 0.f, mid->a, mid->b, mid->c);
    mid->y[0] = w[V_R0 * 32];
    mid->y[1] = w[V_R4 * 32];
  }
  cpa_wait<0>();
}

constexpr int NEX = 15;   // rows the sides of a walled block line exchange

// 32 block lines of direction D, adjacent in phi: warp 0 the top side, warp 1 the bottom
template <int D>
__device__ __forceinline__ void block_lines(const Args& A, float (*ex)[32], float (*rings)[32], int blk, int* bad) {
  const Geo<float>& g = A.g;
  const int n = len<D>(g), lane = threadIdx.x & 31, side = threadIdx.x >> 5;
  const int nl = (D == 0 ? g.nt : g.nr) * g.np, l0 = blk * 32 + lane;
  const bool valid = l0 < nl;
  const int line = valid ? l0 : nl - 1, a = line / g.np, b = line - a * g.np;
  const int q = n / 2, cnt = side ? n - 1 - q : q;        // the middle cell; this side's cells
  float* scr = A.scr + (size_t)blk * n * (12 * 32) + lane;
  float* ring = &rings[side * RING][lane];
  float E[9], gv[3], x[3];
  Mid mid;
  int sing = 0;
  if (side == 0) {
    eliminate<D, 0>(A, a, b, n, cnt, ring, scr, E, gv, &mid, &sing);
  } else {
    eliminate<D, 1>(A, a, b, n, cnt, ring, scr, E, gv, nullptr, &sing);
#pragma unroll
    for (int k = 0; k < 9; k++) ex[k][lane] = E[k];
#pragma unroll
    for (int k = 0; k < 3; k++) ex[9 + k][lane] = gv[k];
  }
  __syncthreads();   // (also orders the factors' stores before their copies back)
  auto cell = [&](int s) { return side ? n - 1 - s : s; };
  // the factors of cell cnt - 1 - t of this side
  auto issue = [&](int t) {
    if (t < cnt) {
      const float* sp = scr + (size_t)cell(cnt - 1 - t) * (12 * 32);
      float* w = ring + (t % BACK) * (12 * 32);
#pragma unroll
      for (int k = 0; k < 12; k++) cpa(w + k * 32, sp + k * 32);
    }
    cpa_commit();
  };
#pragma unroll 1
  for (int t = 0; t < BACK; t++) issue(t);
  if (side == 0) {
    float Eb[9], gb[3], z[4];
#pragma unroll
    for (int k = 0; k < 9; k++) Eb[k] = ex[k][lane];
#pragma unroll
    for (int k = 0; k < 3; k++) gb[k] = ex[9 + k][lane];
    meet(E, gv, Eb, gb, mid, z, &sing);
    ex[12][lane] = z[0]; ex[13][lane] = z[1]; ex[14][lane] = z[2];
    x[0] = z[0]; x[1] = z[1]; x[2] = z[3];
    if (valid) {
      const int c = ic_of<D>(g, a, b, q);
      A.x.f[0][c] = x[0];
      A.x.f[4][c] = x[1];
      A.x.f[1 + D][fx_of<D>(g, a, b, 0)] = 0.f;
      A.x.f[1 + D][fx_of<D>(g, a, b, n)] = 0.f;
    }
  }
  __syncthreads();
  if (side) { x[0] = ex[12][lane]; x[1] = ex[13][lane]; x[2] = ex[14][lane]; }
  for (int t = 0; t < cnt; t++) {
    const int m = cell(cnt - 1 - t);
    cpa_wait<BACK - 1>();
    const float* w = ring + (t % BACK) * (12 * 32);
    float e[9], v[3];
#pragma unroll
    for (int k = 0; k < 9; k++) e[k] = w[k * 32];
#pragma unroll
    for (int k = 0; k < 3; k++) v[k] = w[(9 + k) * 32];
    sub_mul<M_ALL, 1>(e, x, v);
#pragma unroll
    for (int k = 0; k < 3; k++) x[k] = v[k];
    issue(t + BACK);
    // the cell's factors are dead: drop their 12 lines from L2 unwritten
    __syncwarp();
    if (lane < 12)
      asm volatile("discard.global.L2 [%0], 128;" ::"l"(scr - lane + (size_t)m * (12 * 32) + lane * 32) : "memory");
    if (valid) {
      const int c = ic_of<D>(g, a, b, m);
      A.x.f[0][c] = x[0];
      A.x.f[4][c] = x[1];
      A.x.f[1 + D][fx_of<D>(g, a, b, side ? m : m + 1)] = x[2];
    }
  }
  cpa_wait<0>();
  if (valid) *bad |= sing;
}

constexpr int SFWD = 8, SBACK = 16, SRING = SBACK * 2 > SFWD * 5 ? SBACK * 2 : SFWD * 5;

// 32 transverse scalar lines of component CC along D, the same way (slot: their
// place in the scratch, after the block lines')
template <int D, int KIND>
__device__ __forceinline__ void scalar_lines(const Args& A, float (*ex)[32], float (*rings)[32], int blk, int slot, int* bad) {
  const Geo<float>& g = A.g;
  constexpr int CC = trans_comp(D, KIND);
  const int n = len<D>(g), lane = threadIdx.x & 31, side = threadIdx.x >> 5;
  // lines (a, b): a = 1.. for the component normal to a's direction; b = 1.. (0..
  // when periodic) for u_phi
  const int a0 = CC == 2 ? 0 : 1, b0 = CC == 2 && !g.per ? 1 : 0, nb = g.np - b0;
  const int nl = ((D == 0 ? g.nt : g.nr) - a0) * nb, l0 = blk * 32 + lane;
  const bool valid = l0 < nl;
  const int line = valid ? l0 : nl - 1, a = line / nb + a0, b = line % nb + b0;
  const int h = (n + 1) / 2, cnt = side ? n - h : h;
  float* scr = A.scr + (size_t)A.nb0 * n * (12 * 32) + (size_t)slot * n * (2 * 32) + lane;
  float* ring = &rings[side * SRING][lane];
  const float* rhs = A.rhs.f[1 + CC];
  const float* ua = D == 0 ? A.c.uc0 : A.c.uc1;
  auto cell = [&](int s) { return side ? n - 1 - s : s; };
  const int bm = CC == 2 ? (b > 0 ? b - 1 : g.np - 1) : b;   // b = 0 only on a periodic line
  auto fx = [&](int m) {
    const int i = D == 0 ? m : a, j = D == 0 ? a : m;
    return CC == 0 ? IRf(g, i, j, b) : CC == 1 ? ITf(g, i, j, b) : IPf(g, i, j, b);
  };
  auto c1 = [&](int m) { return D == 0 ? IC(g, m, a, b) : IC(g, a, m, b); };
  auto c0 = [&](int m) {
    const int i = D == 0 ? m : a, j = D == 0 ? a : m;
    return CC == 0 ? IC(g, i - 1, j, b) : CC == 1 ? IC(g, i, j - 1, b) : IC(g, i, j, bm);
  };
  auto issue = [&](int s) {
    if (s < cnt) {
      const int m = cell(s), p = c0(m), q = c1(m);
      float* w = ring + (s % SFWD) * (5 * 32);
      cpa(w, A.c.rho + p); cpa(w + 32, A.c.rho + q);
      cpa(w + 64, ua + p); cpa(w + 96, ua + q);
      cpa(w + 128, rhs + fx(m));
    }
    cpa_commit();
  };
#pragma unroll 1
  for (int s = 0; s < SFWD; s++) issue(s);
  float e = 0.f, gy = 0.f;
  int sing = 0;
  for (int s = 0; s < cnt; s++) {
    const int m = cell(s);
    const float4 w = reinterpret_cast<const float4*>(A.T.s[D][KIND - 1])[D == 0 ? m : a * g.nt + m];
    cpa_wait<SFWD - 1>();
    const float* v = ring + (s % SFWD) * (5 * 32);
    const float3 k = form_scalar(A.h, w, v[0] + v[32], v[64] + v[96]);
    const float r = v[128], am = k.x, cm = k.z;
    float bmid = k.y;
    issue(s + SFWD);
    if (m == 0) bmid -= am;                               // no-slip ghosts
    if (m == n - 1) bmid -= cm;
    const float lo = side ? cm : am, up = side ? am : cm;
    const float den = s ? fmaf(-lo, e, bmid) : bmid;
    if (den == 0.f || !isfinite(den)) sing |= FLAG_SINGULAR;
    const float id = __fdividef(1.f, den);
    gy = (s ? fmaf(-lo, gy, r) : r) * id;
    e = up * id;
    if (s + 1 < cnt) {
      float* sp = scr + (size_t)m * 64;
      sp[0] = e;
      sp[32] = gy;
    }
  }
  ex[side * 2][lane] = e;
  ex[side * 2 + 1][lane] = gy;
  __syncthreads();
  cpa_wait<0>();
  auto back = [&](int t) {   // the factors of cell cnt - 2 - t of this side
    if (t < cnt - 1) {
      const float* sp = scr + (size_t)cell(cnt - 2 - t) * 64;
      float* w = ring + (t % SBACK) * 64;
      cpa(w, sp);
      cpa(w + 32, sp + 32);
    }
    cpa_commit();
  };
#pragma unroll 1
  for (int t = 0; t < SBACK; t++) back(t);
  float x;
  {
    const float ep = ex[(1 - side) * 2][lane], gp = ex[(1 - side) * 2 + 1][lane], den = fmaf(-e, ep, 1.f);
    if (den == 0.f || !isfinite(den)) sing |= FLAG_SINGULAR;
    x = __fdividef(fmaf(-e, gp, gy), den);
  }
  for (int s = cnt - 1; s >= 0; s--) {
    const int m = cell(s);
    if (s < cnt - 1) {
      const int t = cnt - 2 - s;
      cpa_wait<SBACK - 1>();
      const float* w = ring + (t % SBACK) * 64;
      x = fmaf(-w[0], x, w[32]);
      back(t + SBACK);
      __syncwarp();
      if (lane < 2) asm volatile("discard.global.L2 [%0], 128;" ::"l"(scr - lane + (size_t)m * 64 + lane * 32) : "memory");
    }
    if (valid) {
      A.x.f[1 + CC][fx(m)] = x;
      const int i = D == 0 ? m : a, j = D == 0 ? a : m;
      // the wall faces next to the first and last line
      if (CC == 0 && a == 1) A.x.f[1][IRf(g, 0, j, b)] = 0.f;
      if (CC == 0 && a == g.nr - 1) A.x.f[1][IRf(g, g.nr, j, b)] = 0.f;
      if (CC == 1 && a == 1) A.x.f[2][ITf(g, i, 0, b)] = 0.f;
      if (CC == 1 && a == g.nt - 1) A.x.f[2][ITf(g, i, g.nt, b)] = 0.f;
      if (CC == 2 && !g.per && b == 1) A.x.f[3][IPf(g, i, j, 0)] = 0.f;
      if (CC == 2 && !g.per && b == g.np - 1) A.x.f[3][IPf(g, i, j, g.np)] = 0.f;
    }
  }
  if (valid) *bad |= sing;
}

// ---------------------------------------------------------------- phi lines
// A phi line is contiguous, so the lanes of a warp (32 lines) read addresses np
// apart: each lane takes its line in groups of 4 cells with 16-byte loads (VEC:
// np a multiple of 4; single loads otherwise), the next group in flight while
// the current one is eliminated.  The bottom side starts at a multiple of 4 cells, so
// that each side's groups are whole, or past the half of a line too short for that:
// the bottom side of a ring holds the last of the others, whose coupling to X is made
// there, the middle cell of a walled line lies in one group with the cell below it.
// Cyclic lines keep their last cell X out and carry three more columns H (x = y -
// Z X), like the FP64 mode's (sph_fp64_lines.cuh).  X's own system and every x = y -
// Z X are FP64, as in the one-thread-per-line solver: y and Z X cancel where the
// ring is stiff, and the increment reaches the FP64 state unrounded.

// the first cell of the bottom side of N cells (3 and more); a walled line's middle cell
// is the one before
__device__ __forceinline__ int phi_split(int N) {
  const int c = ((N + 1) / 2 + 3) & ~3;
  return c < N ? c : N / 2 + 1;
}

// (the rows are addressed from their first element: the bounds-checked build looks at
// the range [m0, m1) of a row of lim values that an access takes)
__device__ __forceinline__ void row_checked(int f, int m0, int m1, int lim) {
#ifdef SPH_CHECKED
  if (m1 > m0) { checked(f, 0, 0, m0, 1, 1, lim, 0); checked(f, 0, 0, m1 - 1, 1, 1, lim, 0); }
#endif
}
template <bool VEC>
__device__ __forceinline__ void load4(const float* f, int m0, int lim, float* o) {
  row_checked(0, m0, VEC ? m0 + 4 : m0 + 1, lim);
  if (VEC) {
    const float4 v = *reinterpret_cast<const float4*>(f + m0);
    o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
  } else {
#pragma unroll
    for (int q = 0; q < 4; q++) o[q] = m0 + q < lim ? f[m0 + q] : 0.f;
  }
}

struct Grp { float p[4], T[4], grr[4], gtt[4], gpp[4], s1[4], s2[4], r0[4], r4[4], u[4], ru[4]; };

// Elimination of one side's cells [lo, hi).  Cyclic: each with its face m + 1, from
// cell 0 (SIDE 0) or N - 1 (SIDE 1).  Walled: SIDE 1 takes each cell with its face m,
// and SIDE 0 leaves the rows of its last cell, the middle one, in mid.
template <int SIDE, bool CYC, bool VEC>
__device__ __forceinline__ void eliminate_phi(const Args& A, int i, int j, int N, int lo, int hi, float* scr, float* E,
                                              float* gv, float* H, Mid* mid, int* bad) {
  const Geo<float>& g = A.g;
  const int n = g.np, nf = g.npf, ic = IC(g, i, j, 0), fc = IPf(g, i, j, 0);
  constexpr int W = CYC ? 21 : 12;
  constexpr bool DOWN = SIDE && !CYC;
  auto load = [&](int m0, Grp& r) {
    if (m0 < n) {
      load4<VEC>(A.ub.f[0] + ic, m0, n, r.p); load4<VEC>(A.ub.f[4] + ic, m0, n, r.T);
      load4<VEC>(A.c.grr + ic, m0, n, r.grr); load4<VEC>(A.c.gtt + ic, m0, n, r.gtt); load4<VEC>(A.c.gpp + ic, m0, n, r.gpp);
      load4<VEC>(A.c.srp + ic, m0, n, r.s1); load4<VEC>(A.c.stp + ic, m0, n, r.s2);
      load4<VEC>(A.rhs.f[0] + ic, m0, n, r.r0); load4<VEC>(A.rhs.f[4] + ic, m0, n, r.r4);
    }
    if (m0 < nf) {
      load4<VEC && CYC>(A.ub.f[3] + fc, m0, nf, r.u);
      load4<VEC && CYC>(A.rhs.f[3] + fc, m0, nf, r.ru);
    }
  };
  const float4* tb = reinterpret_cast<const float4*>(A.T.b[2] + (size_t)NB * (i * g.nt + j));
  const float4 q0 = tb[0], q1 = tb[1], q2 = tb[2];
  int gr = SIDE ? (hi - 1) / 4 : 0;
  const int ge = SIDE ? lo / 4 : (hi - 1) / 4;
  Grp c, nx;
  load(4 * gr, c);
  // carried along: Ubar's u on the face shared with the cell before; its right-hand
  // side and density (the ring's bottom side); the cell's own thermodynamics (else)
  float uc = SIDE ? A.ub.f[3][IPf(g, i, j, N)] : c.u[0], rc = 0.f, rho = 1.f;
  Th th;
  if (SIDE) {
    th = thermo(A, i, A.ub.f[0][IC(g, i, j, n - 1)], A.ub.f[4][IC(g, i, j, n - 1)]);
    rho = th.rho;
    if (CYC) rc = A.rhs.f[3][IPf(g, i, j, N)];
  } else {
    th = thermo(A, i, c.p[0], c.T[0]);
  }
  bool first = true;
  for (;;) {
    const bool more = gr != ge;
    // (a side's last group still reads the cell after it: its p, T and u)
    if (SIDE ? (DOWN ? gr > 0 : more) : 4 * (gr + 1) < (n > nf ? n : nf)) load(4 * (SIDE ? gr - 1 : gr + 1), nx);
#pragma unroll
    for (int z = 0; z < 4; z++) {
      const int q = SIDE ? 3 - z : z, m = 4 * gr + q;
      if (m < lo || m >= hi) continue;
      float y[3], Ab[9], Bb[9], Cb[9];
      y[0] = c.r0[q];
      y[1] = c.r4[q];
      if (DOWN) {
        const Th t1 = thermo(A, i, q > 0 ? c.p[q > 0 ? q - 1 : 0] : nx.p[3], q > 0 ? c.T[q > 0 ? q - 1 : 0] : nx.T[3]);
        y[2] = c.ru[q];
        form_down<2>(A, q0, q1, q2, th, t1.rho, c.u[q], uc, c.grr[q], c.gtt[q], c.gpp[q], c.s1[q], c.s2[q], Ab, Bb, Cb, y);
        uc = c.u[q];
        th = t1;
      } else if (SIDE) {
        th = thermo(A, i, c.p[q], c.T[q]);
        y[2] = rc;
        form<2>(A, q0, q1, q2, th, rho, true, c.u[q], uc, c.grr[q], c.gtt[q], c.gpp[q], c.s1[q], c.s2[q], Ab, Bb, Cb, y);
        uc = c.u[q];
        rc = c.ru[q];
        rho = th.rho;
      } else {
        const int qn = q < 3 ? q + 1 : 0;
        const float un = q < 3 ? c.u[qn] : nx.u[0];
        Th t1 = th;
        if (m + 1 < n) t1 = thermo(A, i, q < 3 ? c.p[qn] : nx.p[0], q < 3 ? c.T[qn] : nx.T[0]);
        y[2] = q < 3 ? c.ru[qn] : nx.ru[0];
        form<2>(A, q0, q1, q2, th, t1.rho, true, uc, un, c.grr[q], c.gtt[q], c.gpp[q], c.s1[q], c.s2[q], Ab, Bb, Cb, y);
        uc = un;
        th = t1;
      }
      if (!CYC && !SIDE && m == hi - 1) {                 // the middle cell
#pragma unroll
        for (int k = 0; k < 6; k++) { mid->a[k] = Ab[k]; mid->b[k] = Bb[k]; mid->c[k] = Cb[k]; }
        mid->y[0] = y[0];
        mid->y[1] = y[1];
        continue;
      }
      cell_step<SIDE && CYC, CYC>(Ab, Bb, Cb, y, first, E, gv, H, bad);
      first = false;
      if (!CYC || (SIDE ? m > lo : m < hi - 1)) {
        float* sp = scr + (size_t)m * (W * 32);
#pragma unroll
        for (int e = 0; e < 9; e++) sp[e * 32] = E[e];
#pragma unroll
        for (int e = 0; e < 3; e++) sp[(9 + e) * 32] = gv[e];
        if (CYC)
#pragma unroll
          for (int e = 0; e < 9; e++) sp[(12 + e) * 32] = H[e];
      }
    }
    if (!more) break;
    gr += SIDE ? -1 : 1;
    c = nx;
  }
}

// an integer test for FP64 values, whose compares take the FP64 pipe
__device__ __forceinline__ bool finite_(float v) { return isfinite(v); }
__device__ __forceinline__ bool finite_(double v) { return ((unsigned)__double2hiint(v) & 0x7ff00000u) != 0x7ff00000u; }

// cells [m0, m1) of one group of a line's field: x (update = 0) or uk = base + x;
// v[q] belongs to index m0 - m0 % 4 + q.  V: float, or double on cyclic lines,
// whose increment reaches the state unrounded.
template <bool VEC, typename V>
__device__ __forceinline__ void emit4(const Args& A, int f, int at, int m0, int m1, const V* v, SqSum<float>& ss, int* bad) {
  const int g0 = m0 & ~3;
  row_checked(f & 3, at + m0, at + m1, A.g.nt * (f == 3 ? A.g.nr * A.g.npf : (A.g.nr + (f == 1)) * A.g.np) + (f == 2 ? A.g.nr * A.g.np : 0));
  if (!A.update) {
    float* x = A.x.f[f] + at;
    if (VEC && m1 - m0 == 4) {
      *reinterpret_cast<float4*>(x + g0) = make_float4((float)v[0], (float)v[1], (float)v[2], (float)v[3]);
    } else {
#pragma unroll
      for (int q = 0; q < 4; q++) if (g0 + q >= m0 && g0 + q < m1) x[g0 + q] = (float)v[q];
    }
    return;
  }
  const double* b = A.base.f[f] + at + g0;
  double* u = A.uk.f[f] + at + g0;
#pragma unroll
  for (int q = 0; q < 4; q++)
    if (g0 + q >= m0 && g0 + q < m1) {
      if (!finite_(v[q])) *bad |= FLAG_NONFINITE;
      if (A.norms) ss.add(f, (float)v[q]);
    }
  if (VEC && m1 - m0 == 4) {
    const double2 b0 = reinterpret_cast<const double2*>(b)[0], b1 = reinterpret_cast<const double2*>(b)[1];
    reinterpret_cast<double2*>(u)[0] = make_double2(b0.x + f2d(v[0]), b0.y + f2d(v[1]));
    reinterpret_cast<double2*>(u)[1] = make_double2(b1.x + f2d(v[2]), b1.y + f2d(v[3]));
  } else {
    double w[4];
#pragma unroll
    for (int q = 0; q < 4; q++) if (g0 + q >= m0 && g0 + q < m1) w[q] = b[q] + f2d(v[q]);
#pragma unroll
    for (int q = 0; q < 4; q++) if (g0 + q >= m0 && g0 + q < m1) u[q] = w[q];
  }
}
__device__ __forceinline__ void emit_wall(const Args& A, int f, int idx) {
  if (A.update) A.uk.f[f][idx] = A.base.f[f][idx];
  else A.x.f[f][idx] = 0.f;
}
// cells [m0, m1) of one group of a cyclic block line: p, T, and u on their faces m + 1
template <bool VEC>
__device__ __forceinline__ void emit_cells(const Args& A, int i, int j, int m0, int m1, const double (*v)[4],
                                           SqSum<float>& ss, int* bad) {
  const Geo<float>& g = A.g;
  const int n = g.np, ic = IC(g, i, j, 0), fc = IPf(g, i, j, 0);
  emit4<VEC>(A, 0, ic, m0, m1, v[0], ss, bad);
  emit4<VEC>(A, 4, ic, m0, m1, v[1], ss, bad);
  const bool last = m1 == n;           // the last cell's face m + 1 is the ring's first
  emit4<false>(A, 3, fc + 1, m0, last ? m1 - 1 : m1, v[2], ss, bad);
  if (last) emit4<false>(A, 3, fc + 1 - n, n - 1, n, v[2], ss, bad);
}

// 32 walled block lines (i, j) along phi
template <bool VEC>
__device__ __forceinline__ void block_lines_phi_walled(const Args& A, float (*ex)[32], int blk, SqSum<float>& ss, int* bad) {
  const Geo<float>& g = A.g;
  const int n = g.np, lane = threadIdx.x & 31, side = threadIdx.x >> 5;
  const int nl = g.nr * g.nt, l0 = blk * 32 + lane;
  const bool valid = l0 < nl;
  const int line = valid ? l0 : nl - 1, i = line / g.nt, j = line - i * g.nt;
  // the sides' cells, the middle one the top side's last
  const int c = phi_split(n), lo = side ? c : 0, hi = side ? n : c;
  const int ic = IC(g, i, j, 0), fc = IPf(g, i, j, 0);
  float* scr = A.scr + (size_t)blk * n * (12 * 32) + lane;
  float E[9], gv[3], x[3];
  Mid mid;
  int sing = 0;
  if (side == 0) {
    eliminate_phi<0, false, VEC>(A, i, j, n, lo, hi, scr, E, gv, nullptr, &mid, &sing);
  } else {
    eliminate_phi<1, false, VEC>(A, i, j, n, lo, hi, scr, E, gv, nullptr, nullptr, &sing);
#pragma unroll
    for (int k = 0; k < 9; k++) ex[k][lane] = E[k];
#pragma unroll
    for (int k = 0; k < 3; k++) ex[9 + k][lane] = gv[k];
  }
  __syncthreads();
  if (side == 0) {
    float Eb[9], gb[3], z[4];
#pragma unroll
    for (int k = 0; k < 9; k++) Eb[k] = ex[k][lane];
#pragma unroll
    for (int k = 0; k < 3; k++) gb[k] = ex[9 + k][lane];
    meet(E, gv, Eb, gb, mid, z, &sing);
    ex[12][lane] = z[0]; ex[13][lane] = z[1]; ex[14][lane] = z[2];
    x[0] = z[0]; x[1] = z[1]; x[2] = z[3];
    if (valid) {
      emit_wall(A, 3, IPf(g, i, j, 0));
      emit_wall(A, 3, IPf(g, i, j, n));
    }
  }
  __syncthreads();
  if (side) { x[0] = ex[12][lane]; x[1] = ex[13][lane]; x[2] = ex[14][lane]; }
  // substitution outwards, group by group
  const int dir = side ? 1 : -1, m_in = side ? lo : hi - 2;   // the first cell with factors
  {
    float En[9], gn[3], out[3][4];
    auto fetch = [&](int m) {
      const float* sp = scr + (size_t)m * (12 * 32);
#pragma unroll
      for (int k = 0; k < 9; k++) En[k] = sp[k * 32];
#pragma unroll
      for (int k = 0; k < 3; k++) gn[k] = sp[(9 + k) * 32];
    };
    fetch(m_in);
    int gr = (side ? lo : hi - 1) / 4;
    const int ge = (side ? hi - 1 : lo) / 4;
    for (;;) {
#pragma unroll
      for (int z = 0; z < 4; z++) {
        const int q = side ? z : 3 - z, m = 4 * gr + q;
        if (m < lo || m >= hi) continue;
        if (m != c - 1) {
          float e[9], v[3];
#pragma unroll
          for (int k = 0; k < 9; k++) e[k] = En[k];
#pragma unroll
          for (int k = 0; k < 3; k++) v[k] = gn[k];
          if (side ? m < hi - 1 : m > lo) fetch(m + dir);
          sub_mul<M_ALL, 1>(e, x, v);
#pragma unroll
          for (int k = 0; k < 3; k++) x[k] = v[k];
        }
        // (a side-dependent index would put the array in local memory)
#pragma unroll
        for (int k = 0; k < 3; k++) {
          if (side) out[k][z] = x[k];
          else out[k][3 - z] = x[k];
        }
      }
      if (valid) {
        const int m0 = 4 * gr > lo ? 4 * gr : lo, m1 = 4 * gr + 4 < hi ? 4 * gr + 4 : hi;
        emit4<VEC>(A, 0, ic, m0, m1, out[0], ss, bad);
        emit4<VEC>(A, 4, ic, m0, m1, out[1], ss, bad);
        // u on the faces m (bottom), m + 1 (top: the middle cell's is the bottom's)
        if (side) emit4<false>(A, 3, fc, m0, m1, out[2], ss, bad);
        else emit4<false>(A, 3, fc + 1, m0, m1 < c - 1 ? m1 : c - 1, out[2], ss, bad);
      }
      // the group's factors are dead: drop their lines from L2 unwritten
      __syncwarp();
      for (int k = lane; k < 4 * 12; k += 32)
        if (4 * gr + k / 12 >= lo && 4 * gr + k / 12 < hi)
          asm volatile("discard.global.L2 [%0], 128;" ::"l"(scr - lane + (size_t)(4 * gr * 12 + k) * 32) : "memory");
      if (gr == ge) break;
      gr += dir;
    }
  }
  if (valid) *bad |= sing;
}

// 32 cyclic block lines (i, j) along phi
template <bool VEC>
__device__ __forceinline__ void block_lines_phi_ring(const Args& A, float (*ex)[32], int blk, SqSum<float>& ss, int* bad) {
  const Geo<float>& g = A.g;
  const int n = g.np, N = n - 1, lane = threadIdx.x & 31, side = threadIdx.x >> 5;
  const int nl = g.nr * g.nt, l0 = blk * 32 + lane;
  const bool valid = l0 < nl;
  const int line = valid ? l0 : nl - 1, i = line / g.nt, j = line - i * g.nt;
  const int c = phi_split(N), lo = side ? c : 0, hi = side ? N : c;
  constexpr int W = 21;
  float* scr = A.scr + (size_t)blk * n * (W * 32) + lane;
  float E[9], gv[3], H[9];
  int sing = 0;
  if (side == 0) eliminate_phi<0, true, VEC>(A, i, j, N, lo, hi, scr, E, gv, H, nullptr, &sing);
  else eliminate_phi<1, true, VEC>(A, i, j, N, lo, hi, scr, E, gv, H, nullptr, &sing);
  {
    float* mine = &ex[side * W][lane];
#pragma unroll
    for (int q = 0; q < 9; q++) mine[q * 32] = E[q];
#pragma unroll
    for (int q = 0; q < 3; q++) mine[(9 + q) * 32] = gv[q];
#pragma unroll
    for (int q = 0; q < 9; q++) mine[(12 + q) * 32] = H[q];
  }
  __syncthreads();
  float x[3], Z[9];
  {
    const float* o = &ex[(1 - side) * W][lane];
    float Ep[9], gp[3], M[9], Mi[9];
#pragma unroll
    for (int q = 0; q < 9; q++) { Ep[q] = o[q * 32]; M[q] = q % 4 == 0 ? 1.f : 0.f; }
#pragma unroll
    for (int q = 0; q < 3; q++) gp[q] = o[(9 + q) * 32];
    sub_mul<M_ALL, 3>(E, Ep, M);
    sub_mul<M_ALL, 1>(E, gp, gv);
    inverse_or_nan(M, Mi, &sing);
    mv(Mi, gv, x);
    float Hp[9];
#pragma unroll
    for (int q = 0; q < 9; q++) Hp[q] = o[(12 + q) * 32];
    sub_mul<M_ALL, 3>(E, Hp, H);
    mul_sparse<M_ALL>(Mi, H, Z);
  }
  // substitution outwards; y and Z stay in the factors' place until the ring is closed
  const int ms = side ? lo : hi - 1, dir = side ? 1 : -1;   // the side's meeting cell, outwards
  {
    float En[9], gn[3], Hn[9];
    auto fetch = [&](int m) {
      const float* sp = scr + (size_t)m * (W * 32);
#pragma unroll
      for (int q = 0; q < 9; q++) { En[q] = sp[q * 32]; Hn[q] = sp[(12 + q) * 32]; }
#pragma unroll
      for (int q = 0; q < 3; q++) gn[q] = sp[(9 + q) * 32];
    };
    if (hi - lo >= 2) fetch(ms + dir);
    for (int m = ms; side ? m < hi : m >= lo; m += dir) {
      if (m != ms) {
        float e[9], v[3], w[9];
#pragma unroll
        for (int k = 0; k < 9; k++) { e[k] = En[k]; w[k] = Hn[k]; }
#pragma unroll
        for (int k = 0; k < 3; k++) v[k] = gn[k];
        if (side ? m < hi - 1 : m > lo) fetch(m + dir);
        sub_mul<M_ALL, 1>(e, x, v);
        sub_mul<M_ALL, 3>(e, Z, w);
#pragma unroll
        for (int k = 0; k < 3; k++) x[k] = v[k];
#pragma unroll
        for (int k = 0; k < 9; k++) Z[k] = w[k];
      }
      float* sp = scr + (size_t)m * (W * 32);
#pragma unroll
      for (int k = 0; k < 9; k++) sp[k * 32] = Z[k];
#pragma unroll
      for (int k = 0; k < 3; k++) sp[(9 + k) * 32] = x[k];
    }
  }
  // the ring's last cell: (B - C Z_0 - A Z_{N-1}) X = r - C y_0 - A y_{N-1}
  __syncthreads();
  float* mine = &ex[side * W][lane];
#pragma unroll
  for (int q = 0; q < 9; q++) mine[q * 32] = Z[q];
#pragma unroll
  for (int q = 0; q < 3; q++) mine[(9 + q) * 32] = x[q];
  __syncthreads();
  const int ic = IC(g, i, j, 0), fc = IPf(g, i, j, 0), e = IC(g, i, j, n - 1);
  const float4* tb = reinterpret_cast<const float4*>(A.T.b[2] + (size_t)NB * (i * g.nt + j));
  const Th th = thermo(A, i, A.ub.f[0][e], A.ub.f[4][e]), t0 = thermo(A, i, A.ub.f[0][ic], A.ub.f[4][ic]);
  float Ab[9], Bb[9], Cb[9], r[3] = {A.rhs.f[0][e], A.rhs.f[4][e], A.rhs.f[3][fc]};
  form<2>(A, tb[0], tb[1], tb[2], th, t0.rho, true, A.ub.f[3][IPf(g, i, j, n - 1)], A.ub.f[3][fc], A.c.grr[e], A.c.gtt[e],
          A.c.gpp[e], A.c.srp[e], A.c.stp[e], Ab, Bb, Cb, r);
  double L[9], B[9], Bi[9], X[3], y[3] = {r[0], r[1], r[2]};
#pragma unroll
  for (int q = 0; q < 9; q++) B[q] = Bb[q];
#pragma unroll
  for (int w = 0; w < 2; w++) {      // cell 0 lies with the top side, cell N - 1 with the bottom
    const float* o = &ex[w * W][lane];
    double Zw[9], yw[3];
#pragma unroll
    for (int q = 0; q < 9; q++) { Zw[q] = o[q * 32]; L[q] = (w ? M_A : M_C) >> q & 1 ? (w ? Ab : Cb)[q] : 0.f; }
#pragma unroll
    for (int q = 0; q < 3; q++) yw[q] = o[(9 + q) * 32];
    if (w) { sub_mul<M_A, 3>(L, Zw, B); sub_mul<M_A, 1>(L, yw, y); }
    else { sub_mul<M_C, 3>(L, Zw, B); sub_mul<M_C, 1>(L, yw, y); }
  }
  inverse_or_nan(B, Bi, &sing);
  mv(Bi, y, X);
  for (int m0 = lo; m0 < hi; m0 = (m0 & ~3) + 4) {
    const int m1 = (m0 & ~3) + 4 < hi ? (m0 & ~3) + 4 : hi;
    double out[3][4];
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int m = (m0 & ~3) + q;
      if (m < m0 || m >= m1) continue;
      const float* sp = scr + (size_t)m * (W * 32);
      double Zm[9], v[3];
#pragma unroll
      for (int k = 0; k < 9; k++) Zm[k] = f2d(sp[k * 32]);
#pragma unroll
      for (int k = 0; k < 3; k++) v[k] = f2d(sp[(9 + k) * 32]);
      sub_mul<M_ALL, 1>(Zm, X, v);
#pragma unroll
      for (int k = 0; k < 3; k++) out[k][q] = v[k];
    }
    if (valid) emit_cells<VEC>(A, i, j, m0, m1, out, ss, bad);
    __syncwarp();
    for (int k = lane; k < (m1 - m0) * W; k += 32)
      asm volatile("discard.global.L2 [%0], 128;" ::"l"(scr - lane + ((size_t)m0 * W + k) * 32) : "memory");
  }
  if (side == 0 && valid) {
    double out[3][4];
#pragma unroll
    for (int q = 0; q < 4; q++)
#pragma unroll
      for (int k = 0; k < 3; k++) out[k][q] = X[k];
    emit_cells<VEC>(A, i, j, n - 1, n, out, ss, bad);
  }
  if (valid) *bad |= sing;
}

template <bool CYC, bool VEC>
__device__ __forceinline__ void block_lines_phi(const Args& A, float (*ex)[32], int blk, SqSum<float>& ss, int* bad) {
  if constexpr (CYC) block_lines_phi_ring<VEC>(A, ex, blk, ss, bad);
  else block_lines_phi_walled<VEC>(A, ex, blk, ss, bad);
}

// 32 transverse scalar lines along phi: component 0 (KIND 1, r-faces 1..nr-1) or 1
// (KIND 2, theta-faces 1..nt-1)
template <int KIND, bool CYC, bool VEC>
__device__ __forceinline__ void scalar_lines_phi(const Args& A, float (*ex)[32], int blk, int slot, SqSum<float>& ss,
                                                 int* bad) {
  const Geo<float>& g = A.g;
  constexpr int CC = KIND - 1, W = CYC ? 3 : 2;
  const int n = g.np, N = CYC ? n - 1 : n, lane = threadIdx.x & 31, side = threadIdx.x >> 5;
  const int nj = CC == 1 ? g.nt - 1 : g.nt, nl = (CC == 0 ? g.nr - 1 : g.nr) * nj, l0 = blk * 32 + lane;
  const bool valid = l0 < nl;
  const int line = valid ? l0 : nl - 1, i = line / nj + (CC == 0), j = line % nj + (CC == 1);
  const int c = phi_split(N), lo = side ? c : 0, hi = side ? N : c;
  float* scr = A.scr + (size_t)A.nb0 * n * ((CYC ? 21 : 12) * 32) + (size_t)slot * n * (W * 32) + lane;
  const int p0 = CC == 0 ? IC(g, i - 1, j, 0) : IC(g, i, j - 1, 0), p1 = IC(g, i, j, 0);
  const int fx = CC == 0 ? IRf(g, i, j, 0) : ITf(g, i, j, 0);
  const float4 w = reinterpret_cast<const float4*>(A.T.s[2][CC])[CC == 0 ? i * g.nt + j : i * (g.nt + 1) + j];
  struct G5 { float a[4], b[4], u[4], v[4], r[4]; };
  auto load = [&](int m0, G5& q) {
    load4<VEC>(A.c.rho + p0, m0, n, q.a); load4<VEC>(A.c.rho + p1, m0, n, q.b);
    load4<VEC>(A.c.uc2 + p0, m0, n, q.u); load4<VEC>(A.c.uc2 + p1, m0, n, q.v);
    load4<VEC>(A.rhs.f[1 + CC] + fx, m0, n, q.r);
  };
  float e = 0.f, gy = 0.f, hz = 0.f;
  int sing = 0;
  // one cell of the side's elimination; S: which side, a compile-time constant
  auto step = [&](auto S, const G5& q5, int q, int m, bool first) {
    constexpr int SIDE = decltype(S)::value;
    const float3 k = form_scalar(A.h, w, q5.a[q] + q5.b[q], q5.u[q] + q5.v[q]);
    const float am = k.x, cm = k.z;
    float bm = k.y;
    if (!CYC && m == 0) bm -= am;                         // no-slip ghosts
    if (!CYC && m == n - 1) bm -= cm;
    const float L = SIDE ? cm : am, U = SIDE ? am : cm;
    const float den = first ? bm : fmaf(-L, e, bm);
    if (den == 0.f || !isfinite(den)) sing |= FLAG_SINGULAR;
    const float id = __fdividef(1.f, den);
    gy = (first ? q5.r[q] : fmaf(-L, gy, q5.r[q])) * id;
    if (CYC) hz = (first ? L : -L * hz) * id;
    e = U * id;
    if (SIDE ? m > lo : m < hi - 1) {
      float* sp = scr + (size_t)m * (W * 32);
      sp[0] = e;
      sp[32] = gy;
      if (CYC) sp[64] = hz;
    }
  };
  {
    G5 cg, nx;
    int gr = side ? (hi - 1) / 4 : 0;
    const int ge = side ? lo / 4 : (hi - 1) / 4;
    load(4 * gr, cg);
    bool first = true;
    for (;;) {
      const bool more = gr != ge;
      if (more) load(4 * (side ? gr - 1 : gr + 1), nx);
#pragma unroll
      for (int z = 0; z < 4; z++) {
        const int m = 4 * gr + (side ? 3 - z : z);
        if (m < lo || m >= hi) continue;
        if (side) step(std::integral_constant<int, 1>(), cg, 3 - z, m, first);
        else step(std::integral_constant<int, 0>(), cg, z, m, first);
        first = false;
      }
      if (!more) break;
      gr += side ? -1 : 1;
      cg = nx;
    }
  }
  ex[side * 3][lane] = e;
  ex[side * 3 + 1][lane] = gy;
  ex[side * 3 + 2][lane] = hz;
  __syncthreads();
  float x, Z = 0.f;
  {
    const float ep = ex[(1 - side) * 3][lane], gp = ex[(1 - side) * 3 + 1][lane], den = fmaf(-e, ep, 1.f);
    if (den == 0.f || !isfinite(den)) sing |= FLAG_SINGULAR;
    const float id = __fdividef(1.f, den);
    x = fmaf(-e, gp, gy) * id;
    if (CYC) Z = fmaf(-e, ex[(1 - side) * 3 + 2][lane], hz) * id;
  }
  // the wall faces beside the first and last line of the component
  auto wall = [&](int m0, int m1, bool lowest, bool highest) {
    for (int m = m0; m < m1; m++) {
      if (lowest) emit_wall(A, 1 + CC, CC == 0 ? IRf(g, 0, j, m) : ITf(g, i, 0, m));
      if (highest) emit_wall(A, 1 + CC, CC == 0 ? IRf(g, g.nr, j, m) : ITf(g, i, g.nt, m));
    }
  };
  const bool wl = CC == 0 ? i == 1 : j == 1, wh = CC == 0 ? i == g.nr - 1 : j == g.nt - 1;
  const int ms = side ? lo : hi - 1, dir = side ? 1 : -1;
  {
    float en = 0.f, gn = 0.f, hn = 0.f, out[4];
    auto fetch = [&](int m) {
      const float* sp = scr + (size_t)m * (W * 32);
      en = sp[0];
      gn = sp[32];
      if (CYC) hn = sp[64];
    };
    if (hi - lo >= 2) fetch(ms + dir);
    int gr = ms / 4;
    const int ge = (side ? hi - 1 : lo) / 4;
    for (;;) {
#pragma unroll
      for (int z = 0; z < 4; z++) {
        const int m = 4 * gr + (side ? z : 3 - z);
        if (m < lo || m >= hi) continue;
        if (m != ms) {
          const float e_ = en, g_ = gn, h_ = hn;
          if (side ? m < hi - 1 : m > lo) fetch(m + dir);
          x = fmaf(-e_, x, g_);
          if (CYC) Z = fmaf(-e_, Z, h_);
        }
        if (CYC) {
          float* sp = scr + (size_t)m * (W * 32);
          sp[0] = Z;
          sp[32] = x;
        } else {
          if (side) out[z] = x;
          else out[3 - z] = x;
        }
      }
      if (!CYC) {
        if (valid) {
          const int m0 = 4 * gr > lo ? 4 * gr : lo, m1 = 4 * gr + 4 < hi ? 4 * gr + 4 : hi;
          emit4<VEC>(A, 1 + CC, fx, m0, m1, out, ss, bad);
          if (wl || wh) wall(m0, m1, wl, wh);
        }
        __syncwarp();
        if (lane < 4 * W && 4 * gr + lane / W >= lo && 4 * gr + lane / W < hi)
          asm volatile("discard.global.L2 [%0], 128;" ::"l"(scr - lane + (size_t)(4 * gr * W + lane) * 32) : "memory");
      }
      if (gr == ge) break;
      gr += dir;
    }
  }
  if (CYC) {
    __syncthreads();
    ex[side * 3][lane] = Z;
    ex[side * 3 + 1][lane] = x;
    __syncthreads();
    const int m = n - 1;
    const float3 k = form_scalar(A.h, w, A.c.rho[p0 + m] + A.c.rho[p1 + m], A.c.uc2[p0 + m] + A.c.uc2[p1 + m]);
    const double am = k.x, cm = k.z;
    const double den = fma(-cm, (double)ex[0][lane], fma(-am, (double)ex[3][lane], (double)k.y));
    if (den == 0.0 || !finite_(den)) sing |= FLAG_SINGULAR;
    const double X = fma(-cm, (double)ex[1][lane], fma(-am, (double)ex[4][lane], (double)A.rhs.f[1 + CC][fx + m])) / den;
    for (int m0 = lo; m0 < hi; m0 = (m0 & ~3) + 4) {
      const int m1 = (m0 & ~3) + 4 < hi ? (m0 & ~3) + 4 : hi;
      double out[4];
#pragma unroll
      for (int q = 0; q < 4; q++) {
        const int k = (m0 & ~3) + q;
        if (k < m0 || k >= m1) continue;
        const float* sp = scr + (size_t)k * (W * 32);
        out[q] = fma(-f2d(sp[0]), X, f2d(sp[32]));
      }
      if (valid) {
        emit4<VEC>(A, 1 + CC, fx, m0, m1, out, ss, bad);
        if (wl || wh) wall(m0, m1, wl, wh);
      }
    }
    if (side == 0 && valid) {
      const double out[4] = {X, X, X, X};
      emit4<VEC>(A, 1 + CC, fx, n - 1, n, out, ss, bad);
      if (wl || wh) wall(n - 1, n, wl, wh);
    }
  }
  if (valid) *bad |= sing;
}

}  // namespace lines2
