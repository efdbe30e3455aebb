// sph_blk3.cuh -- products with the sparse 3x3 blocks of a line row (p, T, u):
// the lower block A sees no p in the T row and only u in the u row, the upper
// block C sees no u in the p and T rows, no p in the T row, no T in the u row.
// A mask has bit 3r+q set where entry (r, q) may be nonzero; the zeros are
// skipped at compile time (a compiler may not: 0 * x is not 0 for every x).
#pragma once

namespace blk3 {

constexpr unsigned M_A = 0x137, M_C = 0x153, M_B = 0x177, M_ALL = 0x1ff;   // A: 012 45 8; C: 01 4 6 8; B: 012 45 6 8
// the mask of the transposed block
__host__ __device__ constexpr unsigned mt(unsigned m) {
  unsigned o = 0;
  for (int r = 0; r < 3; r++)
    for (int q = 0; q < 3; q++)
      if (m >> (3 * r + q) & 1) o |= 1u << (3 * q + r);
  return o;
}

__device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }

// S (3 x NCOL) -= L E over L's nonzero entries
template <unsigned M, int NCOL, typename R>
__device__ __forceinline__ void sub_mul(const R* L, const R* E, R* S) {
#pragma unroll
  for (int r = 0; r < 3; r++)
#pragma unroll
    for (int k = 0; k < 3; k++)
      if (M >> (3 * r + k) & 1)
#pragma unroll
        for (int q = 0; q < NCOL; q++) S[r * NCOL + q] = fma_(-L[3 * r + k], E[k * NCOL + q], S[r * NCOL + q]);
}
// Z = X U over U's nonzero entries (3 x 3)
template <unsigned M, typename R>
__device__ __forceinline__ void mul_sparse(const R* X, const R* U, R* Z) {
#pragma unroll
  for (int q = 0; q < 3; q++)
#pragma unroll
    for (int r = 0; r < 3; r++) {
      R v = R(0);
      bool first = true;
#pragma unroll
      for (int k = 0; k < 3; k++)
        if (M >> (3 * k + q) & 1) {
          v = first ? X[3 * r + k] * U[3 * k + q] : fma_(X[3 * r + k], U[3 * k + q], v);
          first = false;
        }
      Z[3 * r + q] = v;
    }
}
template <typename R>
__device__ __forceinline__ void mv(const R* X, const R* y, R* z) {
#pragma unroll
  for (int r = 0; r < 3; r++) z[r] = fma_(X[3 * r + 2], y[2], fma_(X[3 * r + 1], y[1], X[3 * r] * y[0]));
}

}  // namespace blk3
