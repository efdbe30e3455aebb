// sph_noalloc.cu -- a batched 3x3-block tridiagonal line solver that allocates no
// device memory.
//
// Some callers cannot call cudaMalloc: code that runs while a memory pool must
// not grow, inside a host that forbids runtime allocation after start-up, or in
// plug-ins that only receive device pointers from their host.  For them this
// file provides one entry point, sph_block_thomas_noalloc, which runs the same
// block Thomas elimination the line sweeps use (forward elimination with the
// block adjugate, no pivoting between blocks, back substitution) on line systems
// the caller has assembled.  Its elimination scratch (C'_m and d'_m, 12 doubles
// per block) lives in the file-scope array below instead of a cudaMalloc'd
// buffer.  The array is part of the library image: every GPU that loads the
// library holds it (SPH_NOALLOC_MAX_BLOCKS * 12 doubles, 12.6 MB) until the
// process exits.
#include <cuda_runtime.h>
#include <math.h>

#include "../../include/sph.h"

#define NOALLOC_MAX_DEVICES 64

static __device__ __align__(256) double g_noalloc_scratch[(size_t)SPH_NOALLOC_MAX_BLOCKS * 12];

// Device address of the array on each device, looked up once per device: in
// host code the symbol's name is only a host-side stand-in, not an address.
static double* s_scratch[NOALLOC_MAX_DEVICES];
static int s_nsm[NOALLOC_MAX_DEVICES];   // and its SMs

static __device__ __forceinline__ bool inv3_na(const double* S, double* I) {
  double c00 = S[4] * S[8] - S[5] * S[7];
  double c01 = S[5] * S[6] - S[3] * S[8];
  double c02 = S[3] * S[7] - S[4] * S[6];
  double det = S[0] * c00 + S[1] * c01 + S[2] * c02;
  if (det == 0.0 || !isfinite(det)) return false;
  double id = 1.0 / det;
  I[0] = c00 * id; I[3] = c01 * id; I[6] = c02 * id;
  I[1] = (S[2] * S[7] - S[1] * S[8]) * id;
  I[4] = (S[0] * S[8] - S[2] * S[6]) * id;
  I[7] = (S[1] * S[6] - S[0] * S[7]) * id;
  I[2] = (S[1] * S[5] - S[2] * S[4]) * id;
  I[5] = (S[2] * S[3] - S[0] * S[5]) * id;
  I[8] = (S[0] * S[4] - S[1] * S[3]) * id;
  return true;
}

// One thread per line.  Blocks of line l, cell m start at ((l*n + m)*9); the
// scratch is interleaved by line, [(m*12 + q)*nlines + l], so a warp's accesses
// are contiguous.
__global__ void k_block_thomas_noalloc(int nlines, int n, const double* __restrict__ A, const double* __restrict__ B,
                                       const double* __restrict__ C, const double* __restrict__ d,
                                       double* __restrict__ x, double* __restrict__ scr) {
  int l = blockIdx.x * blockDim.x + threadIdx.x;
  if (l >= nlines) return;
  double Cp[9], dp[3];
  for (int m = 0; m < n; m++) {
    long b = ((long)l * n + m);
    const double* Am = A + 9 * b;
    const double* Bm = B + 9 * b;
    const double* Cm = C + 9 * b;
    const double* dm = d + 3 * b;
    double S[9], y[3];
    if (m == 0) {
      for (int q = 0; q < 9; q++) S[q] = Bm[q];
      for (int q = 0; q < 3; q++) y[q] = dm[q];
    } else {
      for (int r = 0; r < 3; r++) {
        for (int q = 0; q < 3; q++)
          S[r * 3 + q] = Bm[r * 3 + q] - (Am[r * 3] * Cp[q] + Am[r * 3 + 1] * Cp[3 + q] + Am[r * 3 + 2] * Cp[6 + q]);
        y[r] = dm[r] - (Am[r * 3] * dp[0] + Am[r * 3 + 1] * dp[1] + Am[r * 3 + 2] * dp[2]);
      }
    }
    double Si[9];
    if (!inv3_na(S, Si)) {   // zero pivot: the whole line becomes NaN
      for (long q = 0; q < 3L * n; q++) x[3L * l * n + q] = NAN;
      return;
    }
    bool last = (m == n - 1);
    for (int r = 0; r < 3; r++) {
      for (int q = 0; q < 3; q++)
        Cp[r * 3 + q] = last ? 0.0 : Si[r * 3] * Cm[q] + Si[r * 3 + 1] * Cm[3 + q] + Si[r * 3 + 2] * Cm[6 + q];
      dp[r] = Si[r * 3] * y[0] + Si[r * 3 + 1] * y[1] + Si[r * 3 + 2] * y[2];
    }
    if (!last) {
      double* s = scr + (long)m * 12 * nlines + l;
      for (int q = 0; q < 9; q++) s[(long)q * nlines] = Cp[q];
      for (int q = 0; q < 3; q++) s[(long)(9 + q) * nlines] = dp[q];
    }
  }
  double xs[3] = {dp[0], dp[1], dp[2]};
  double* xo = x + 3 * ((long)l * n + (n - 1));
  xo[0] = xs[0]; xo[1] = xs[1]; xo[2] = xs[2];
  for (int m = n - 2; m >= 0; m--) {
    const double* s = scr + (long)m * 12 * nlines + l;
    double Cq[9], dq[3], xn[3];
    for (int q = 0; q < 9; q++) Cq[q] = s[(long)q * nlines];
    for (int q = 0; q < 3; q++) dq[q] = s[(long)(9 + q) * nlines];
    for (int r = 0; r < 3; r++) xn[r] = dq[r] - (Cq[r * 3] * xs[0] + Cq[r * 3 + 1] * xs[1] + Cq[r * 3 + 2] * xs[2]);
    xs[0] = xn[0]; xs[1] = xn[1]; xs[2] = xn[2];
    xo = x + 3 * ((long)l * n + m);
    xo[0] = xs[0]; xo[1] = xs[1]; xo[2] = xs[2];
  }
}

// Few lines: 16 lanes per line, two lines per warp.  A FP64 instruction of a warp
// takes 64 cycles of its SM quarter however many lanes are active, so one
// thread per line leaves a serial chain of ~120 of them per block on a few
// warps.  Here lane 4 r + q holds element (r, q) of [C'_m | d'_m] (3 x 4; lanes 12-15
// repeat row 2) and every product of the same elimination, in the same order,
// is one element per lane, its operands exchanged by shuffles: 17 FP64
// instructions a block.  1024 lines of 128 blocks: 661 -> 146 us.
__device__ __forceinline__ double from(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }

__global__ void __launch_bounds__(32) k_block_thomas_split(int nlines, int n, const double* __restrict__ A,
                                                           const double* __restrict__ B, const double* __restrict__ C,
                                                           const double* __restrict__ d, double* __restrict__ x,
                                                           double* __restrict__ scr) {
  const int lane = threadIdx.x, g0 = lane & 16, e = lane & 15, q = e & 3, r = e >> 2 < 3 ? e >> 2 : 2;
  const int l0 = blockIdx.x * 2 + (lane >> 4);
  const bool valid = l0 < nlines;
  const long l = valid ? l0 : nlines - 1;
  // element (a, b) of the 3 x 3 (or 3 x 4) array spread over the line's lanes
  auto at = [&](double v, int a, int b) { return from(v, g0 + 4 * a + b); };
  const int r1 = (r + 1) % 3, r2 = (r + 2) % 3, q3 = q < 3 ? q : 0, q1 = (q3 + 1) % 3, q2 = (q3 + 2) % 3;
  double an[3], cn[3], bn;
  auto fetch = [&](int m) {
    const long b = l * n + m;
#pragma unroll
    for (int z = 0; z < 3; z++) {
      an[z] = m > 0 ? A[9 * b + 3 * r + z] : 0.0;
      cn[z] = q < 3 && m < n - 1 ? C[9 * b + 3 * z + q] : 0.0;
    }
    bn = q < 3 ? B[9 * b + 3 * r + q] : d[3 * b + r];
  };
  bool bad = false;
  double v = 0.0;   // element (r, q) of [C' | d'] of the block before
  fetch(0);
  for (int m = 0; m < n; m++) {
    const double a0 = an[0], a1 = an[1], a2 = an[2], c0 = cn[0], c1 = cn[1], c2 = cn[2];
    double t = bn;
    if (m + 1 < n) fetch(m + 1);
    if (m > 0) t = t - fma(a2, at(v, 2, q), fma(a1, at(v, 1, q), a0 * at(v, 0, q)));
    // adj(S): element (r, q) is the cofactor of (q, r), column q's rows r1, r2 ... of S
    const double s11 = at(t, q1, r1), s22 = at(t, q2, r2), s12 = at(t, q1, r2), s21 = at(t, q2, r1);
    const double adj = fma(s11, s22, -(s12 * s21));
    const double det = fma(at(t, 0, 2), at(adj, 2, 0), fma(at(t, 0, 1), at(adj, 1, 0), at(t, 0, 0) * at(adj, 0, 0)));
    const unsigned hi = (unsigned)__double2hiint(det) & 0x7fffffffu;
    if (hi >= 0x7ff00000u || (hi | (unsigned)__double2loint(det)) == 0u) bad = true;   // zero or non-finite pivot
    const double u0 = q < 3 ? c0 : 0.0, u1 = q < 3 ? c1 : 0.0, u2 = q < 3 ? c2 : 0.0;
    const double y0 = at(t, 0, 3), y1 = at(t, 1, 3), y2 = at(t, 2, 3);
    // (the inverse before it meets the right-hand side, as one thread per line does: adj(S)
    // alone has the square of S's scale, and its product may leave FP64's range)
    const double inv = adj * (1.0 / det);
    v = fma(at(inv, r, 2), q < 3 ? u2 : y2, fma(at(inv, r, 1), q < 3 ? u1 : y1, at(inv, r, 0) * (q < 3 ? u0 : y0)));
    if (m < n - 1 && valid && e < 12) scr[(l * n + m) * 12 + e] = v;
  }
  __syncwarp();
  double xs[3];
#pragma unroll
  for (int z = 0; z < 3; z++) xs[z] = at(v, z, 3);
  double en[4];
  auto back = [&](int m) {
    const double* s = scr + (l * n + m) * 12 + 4 * r;
#pragma unroll
    for (int z = 0; z < 4; z++) en[z] = s[z];
  };
  if (n >= 2) back(n - 2);
  for (int m = n - 1; m >= 0; m--) {
    if (m < n - 1) {
      const double e0 = en[0], e1 = en[1], e2 = en[2], gq = en[3];
      if (m > 0) back(m - 1);
      const double mine = gq - fma(e2, xs[2], fma(e1, xs[1], e0 * xs[0]));
#pragma unroll
      for (int z = 0; z < 3; z++) xs[z] = at(mine, z, 0);
    }
    if (valid && q == 0 && e < 12) x[3 * (l * n + m) + r] = bad ? NAN : r == 0 ? xs[0] : r == 1 ? xs[1] : xs[2];
  }
}

// Per-device set-up, with that device current: its SMs, the device address of the array.
static int noalloc_setup(int dev) {
  if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) return SPH_ERR_ARG;
  if (s_scratch[dev]) return SPH_OK;
  void* p = NULL;
  if (cudaDeviceGetAttribute(&s_nsm[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return SPH_ERR_CUDA;
  if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return SPH_ERR_CUDA;
  s_scratch[dev] = (double*)p;
  return SPH_OK;
}

extern "C" int sph_block_thomas_noalloc(int nlines, int n, const double* A, const double* B, const double* C,
                                        const double* d, double* x, void* stream) {
  if (nlines < 1 || n < 1 || !A || !B || !C || !d || !x) return SPH_ERR_ARG;
  if ((long long)nlines * (long long)n > (long long)SPH_NOALLOC_MAX_BLOCKS) return SPH_ERR_ARG;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return SPH_ERR_CUDA;
  int e = noalloc_setup(dev);
  if (e != SPH_OK) return e;
  cudaStream_t st = (cudaStream_t)stream;
  // the lane-split form needs 17 FP64 instructions a block on nlines / 2 warps, one
  // thread per line about 120 on nlines / 32: the split's time grows with the lines
  // once they fill the SM quarters (8 lines an SM) and reaches the other's near 47 an
  // SM (us, 16 blocks a line, 152 SMs: 6144 lines 74 against 82, 7168 80 against 82, 8192
  // 92 against 83)
  if (nlines <= 47 * s_nsm[dev]) {
    k_block_thomas_split<<<(nlines + 1) / 2, 32, 0, st>>>(nlines, n, A, B, C, d, x, s_scratch[dev]);
  } else {
    int threads = 32;
    int blocks = (nlines + threads - 1) / threads;
    k_block_thomas_noalloc<<<blocks, threads, 0, st>>>(nlines, n, A, B, C, d, x, s_scratch[dev]);
  }
  return cudaGetLastError() == cudaSuccess ? SPH_OK : SPH_ERR_CUDA;
}
