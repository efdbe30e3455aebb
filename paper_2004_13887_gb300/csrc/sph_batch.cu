// sph_batch.cu -- batched launches over a batch of independent problems of
// different sizes (sph_batch_capture_fused): every stage of the scheme's
// iteration (Section 2.2: the midpoint state and frozen coefficients of eq.
// chapter3mainsd, the right-hand side of eq. spl1, the line solves of eqs.
// spl1-spl3) runs as ONE launch over all problems, not one per problem.
//
// A launch reads an instance descriptor table (one entry per problem: its
// grid, coefficient planes, state and work buffers -- what the single-problem
// kernels take as parameters) and a block map (per block: which problem, and
// which tile or line group of it).  A block copies its problem's descriptor
// into shared memory and runs the same device code as the single-problem
// kernel on that tile or line group, so a batched step computes what
// per-problem steps compute (to FP32 rounding: the code is compiled into other
// kernels, where the compiler may contract other multiply-adds).  The sweeps
// launch once per line layout
// (lines of the same length and lane layout share a kernel instantiation),
// the layouts side by side on separate streams.  Everything is recorded into
// one CUDA graph of an even number of steps, like sph_batch_capture.
#include <cuda_runtime.h>
#include <stdlib.h>
#include <string.h>

#include <vector>

#include "../../include/sph.h"
#include "sph_kernels.cuh"
#include "sph_host.cuh"

namespace fused {

// the tile of a stencil launch: tk x tj x ti points (phi, theta, r) per block
// of 128 threads, gx x gy tiles in the phi x theta plane, n tiles in all
struct Tile { int tk, tj, ti, gx, gy, n; };

// Consecutive tiles of one problem a block of a stencil launch takes (one
// descriptor load for all of them), and the blocks per SM the coefficient and
// right-hand-side kernels are compiled for (48 and 72 registers a thread): the
// descriptor in shared memory costs registers that at the single-problem
// kernels' 40 and 56 spill.  Measured, ms a step of the 64-instance ensemble: 1 tile
// 49.1, 4 tiles 45.8, 8 tiles 45.5; right-hand side, ms a pass of 12 problems: 4
// blocks 16.25, 5 16.00, 6 15.67, 7 15.62, 8 15.75, 9 16.20 (four launches' worth
// of rows in one, a thread a row: 16.96).
#ifndef FUSED_TILES
#define FUSED_TILES 8
#endif
constexpr int TILES = FUSED_TILES;
#ifndef FUSED_MINB_COEF
#define FUSED_MINB_COEF 10
#endif
#ifndef FUSED_MINB_RHS
#define FUSED_MINB_RHS 7
#endif

struct StenTab {   // a stencil stage of a problem
  s32::Args A;
  Tile t;
};

struct LineTab {
  SweepArgs<float> S;
  int ng1;    // line groups of the first transverse kind (the scalar launch)
  int pad;
};

// dst = src for a descriptor (8-byte words, the whole block), then a barrier
template <typename T>
__device__ __forceinline__ void load_args(T& dst, const T& src) {
  static_assert(sizeof(T) % 8 == 0, "descriptors are whole 8-byte words");
  const unsigned long long* s = reinterpret_cast<const unsigned long long*>(&src);
  unsigned long long* d = reinterpret_cast<unsigned long long*>(&dst);
  for (int w = threadIdx.x; w < (int)(sizeof(T) / 8); w += blockDim.x) d[w] = s[w];
  __syncthreads();
}

// point (i, j, k) of this thread in tile b of a launch with tile shape t
struct Pt { int i, j, k, i0, j0; };
__device__ __forceinline__ Pt point_of(const Tile& t, int b) {
  const int bx = b % t.gx, r = b / t.gx, by = r % t.gy, bz = r / t.gy;
  const int tid = threadIdx.x, tx = tid % t.tk, r2 = tid / t.tk, ty = r2 % t.tj, tz = r2 / t.tj;
  Pt p;
  p.i0 = bz * t.ti;
  p.j0 = by * t.tj;
  p.i = p.i0 + tz;
  p.j = p.j0 + ty;
  p.k = bx * t.tk + tx;
  return p;
}

// Ubar and D of one chunk of one field of one problem: map = (problem, field,
// first pair, pairs), the pairs of 16-byte loads as in k_avg; the chunk that
// ends the field also takes an odd last element.
__global__ void __launch_bounds__(256) k_avg_f(const AvgArgs<float>* tab, const int4* map) {
  const int4 m = map[blockIdx.x];
  const AvgArgs<float>& A = tab[m.x];
  const int f = m.y;
  const double* __restrict__ a = A.a[f];
  const double* __restrict__ b = A.b[f];
  float* __restrict__ o = A.o[f];
  float* __restrict__ lo = A.lo[f];
  float* __restrict__ d = A.d[f];
  const long n = A.n[f];
  const int same = A.same;
  for (int r = threadIdx.x; r < m.w; r += blockDim.x) {
    const long t = (long)m.z + r;
    double2 x = reinterpret_cast<const double2*>(a)[t];
    if (same) {
      split1(x.x, o, lo, 2 * t);
      split1(x.y, o, lo, 2 * t + 1);
    } else {
      double2 y = reinterpret_cast<const double2*>(b)[t];
      avg1(x.x, y.x, o, lo, d, 2 * t);
      avg1(x.y, y.y, o, lo, d, 2 * t + 1);
    }
  }
  if ((n & 1) && (long)m.z + m.w == (n >> 1) && threadIdx.x == 0) {
    if (same) split1(a[n - 1], o, lo, n - 1);
    else avg1(a[n - 1], b[n - 1], o, lo, d, n - 1);
  }
}

// the coefficient stage over the tiles of every problem
__global__ void __launch_bounds__(128, FUSED_MINB_COEF) k_coef_f(const StenTab* tab, const int2* map) {
  __shared__ StenTab S;
  const int2 m = map[blockIdx.x];
  load_args(S, tab[m.x]);
  const Geo<float>& g = S.A.g;
  const int b1 = min(m.y + TILES, S.t.n);
  for (int b = m.y; b < b1; b++) {
    const Pt p = point_of(S.t, b);
    const bool inner = tile_inner_at(g, p.i0, p.j0, S.t.ti, S.t.tj);
    if (p.k >= g.np || p.j >= g.nt || p.i >= g.nr) continue;
    const s32::Loc L = s32::loc_of(g, p.i, p.j, p.k);
    if (inner) s32::coef<0>(S.A, L);
    else s32::coef<1>(S.A, L);
  }
}

// the right-hand side over the tiles of every problem
__global__ void __launch_bounds__(128, FUSED_MINB_RHS) k_rhs_f(const StenTab* tab, const int2* map) {
  __shared__ StenTab S;
  __shared__ float own[s32::NO][128];
  const int2 m = map[blockIdx.x];
  load_args(S, tab[m.x]);
  const int b1 = min(m.y + TILES, S.t.n);
  for (int b = m.y; b < b1; b++) {
    const Pt p = point_of(S.t, b);
    s32::rhs_cell<false>(S.A, p.i, p.j, p.k, tile_inner_at(S.A.g, p.i0, p.j0, S.t.ti, S.t.tj), &own[0][threadIdx.x]);
  }
}

// the iteration residual's sums of squares of every problem, zeroed
__global__ void k_zero_acc_f(double* const* acc, int n) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < 5 * n) acc[q / 5][q % 5] = 0.0;
}

// block lines of one layout over every problem that has it: map = (entry of
// the layout's table, line group)
template <int D, int P, int L, int CB>
__global__ void __launch_bounds__(CB / P, 512 * P / CB) k_lines_blk_f(const LineTab* tab, const int2* map) {
  __shared__ SweepArgs<float> S;
  const int2 m = map[blockIdx.x];
  load_args(S, tab[m.x].S);
  lines::lines_blk<D, P, L, CB>(S, m.y);
}

// both transverse kinds of one layout over every problem that has it: groups
// [0, ng1) of an entry are of the first kind, the rest of the second
template <int D, int P, int L, int CB>
__global__ void __launch_bounds__(CB / P, 65536 * P / (CB * 48)) k_lines_sca_f(const LineTab* tab, const int2* map) {
  __shared__ SweepArgs<float> S;
  const int2 m = map[blockIdx.x];
  load_args(S, tab[m.x].S);
  const int ng1 = tab[m.x].ng1;
  if (m.y < ng1) lines::lines_sca<D, P, L, CB, 1>(S, m.y);
  else lines::lines_sca<D, P, L, CB, 2>(S, m.y - ng1);
}

// The r- (D = 0) and theta-lines (1) of every problem, 32 lines a block
// (sph_lines2.cuh): one launch for the block lines and one for the scalar lines over
// all problems; map = (problem, block of its launch).
template <int D>
__global__ void __launch_bounds__(64, LINES2_MINB) k_l2_blk_f(const lines2::Args* tab, const int2* map) {
  __shared__ lines2::Args S;
  __shared__ float ex[lines2::NEX][32];
  __shared__ float rings[2 * lines2::RING][32];
  const int2 m = map[blockIdx.x];
  load_args(S, tab[m.x]);
  int bad = 0;
  lines2::block_lines<D>(S, ex, rings, m.y, &bad);
  if (bad) atomicOr(S.flag, bad);
}
template <int D>
__global__ void __launch_bounds__(64) k_l2_sca_f(const lines2::Args* tab, const int2* map) {
  __shared__ lines2::Args S;
  __shared__ float ex[4][32];
  __shared__ float rings[2 * lines2::SRING][32];
  const int2 m = map[blockIdx.x];
  load_args(S, tab[m.x]);
  int bad = 0;
  if (m.y < S.nb1) lines2::scalar_lines<D, 1>(S, ex, rings, m.y, m.y, &bad);
  else lines2::scalar_lines<D, 2>(S, ex, rings, m.y - S.nb1, m.y, &bad);
  if (bad) atomicOr(S.flag, bad);
}

}  // namespace fused

// ============================================================== host side

namespace {

template <typename R> CF<R> cf5(R* const* p) { CF<R> r; for (int f = 0; f < 5; f++) r.f[f] = p[f]; return r; }
template <typename R> MF<R> mf5(R* const* p) { MF<R> r; for (int f = 0; f < 5; f++) r.f[f] = p[f]; return r; }

// host staging of the tables and maps: pieces at 256-byte offsets of one
// device buffer
struct Blob {
  std::vector<char> h;
  size_t put(const void* p, size_t n) {
    size_t off = (h.size() + 255) & ~(size_t)255;
    h.resize(off + (n ? n : 1));
    if (n) memcpy(h.data() + off, p, n);
    return off;
  }
  template <typename T> size_t put(const std::vector<T>& v) { return put(v.data(), v.size() * sizeof(T)); }
};

// the stencil tile of a context over an nk x nj x ni box
fused::Tile tile_of(const sph_ctx* c, int nk, int nj, int ni, int* blocks) {
  fused::Tile t;
  t.tj = c->tile_j;
  t.ti = c->tile_i;
  t.tk = 128 / (t.tj * t.ti);
  t.gx = (nk + t.tk - 1) / t.tk;
  t.gy = (nj + t.tj - 1) / t.tj;
  t.n = t.gx * t.gy * ((ni + t.ti - 1) / t.ti);
  *blocks = t.n;
  return t;
}

// the shared-memory attributes of a layout's batched kernels (per device, before any capture)
template <int D, int P, int L>
int attr_f() {
  constexpr int CB = lines_cb(D, L * P);
  static unsigned long long done = 0;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return SPH_ERR_CUDA;
  const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
  if (done & bit) return SPH_OK;
  const int smb = lines::NFB * lines::Shape<P, L, CB>::FS * (int)sizeof(float);
  const int sms = lines::NFS * lines::Shape<P, L, CB>::FS * (int)sizeof(float);
  if (cudaFuncSetAttribute(fused::k_lines_blk_f<D, P, L, CB>, cudaFuncAttributeMaxDynamicSharedMemorySize, smb) !=
          cudaSuccess ||
      cudaFuncSetAttribute(fused::k_lines_sca_f<D, P, L, CB>, cudaFuncAttributeMaxDynamicSharedMemorySize, sms) !=
          cudaSuccess)
    return SPH_ERR_CUDA;
  done |= bit;
  return SPH_OK;
}

template <int D, int P, int L>
void launch_f(const fused::LineTab* tab, const int2* mb, int nb, const int2* ms, int ns, cudaStream_t s1,
              cudaStream_t s2) {
  constexpr int CB = lines_cb(D, L * P);
  using SH = lines::Shape<P, L, CB>;
  const size_t smb = (size_t)lines::NFB * SH::FS * sizeof(float);
  const size_t sms = (size_t)lines::NFS * SH::FS * sizeof(float);
  if (nb > 0) fused::k_lines_blk_f<D, P, L, CB><<<nb, SH::NT, smb, s1>>>(tab, mb);
  if (ns > 0) fused::k_lines_sca_f<D, P, L, CB><<<ns, SH::NT, sms, s2>>>(tab, ms);
}

// one layout's attributes (attr) or launches, dispatched on (P, L)
template <int D>
int layout_f(int P, int L, bool attr, const fused::LineTab* tab, const int2* mb, int nb, const int2* ms, int ns,
             cudaStream_t s1, cudaStream_t s2) {
#define SPH_LAYOUT_F(p, l)                           \
  if (P == p && L == l) {                            \
    if (attr) return attr_f<D, p, l>();              \
    launch_f<D, p, l>(tab, mb, nb, ms, ns, s1, s2); \
    return SPH_OK;                                   \
  }
  SPH_LINES_EACH_PL(SPH_LAYOUT_F)
#undef SPH_LAYOUT_F
  if constexpr (D == 2) {
    if (P == 8 && L == 64) { if (attr) return attr_f<D, 8, 64>(); launch_f<D, 8, 64>(tab, mb, nb, ms, ns, s1, s2); return SPH_OK; }
    if (P == 8 && L == 128) { if (attr) return attr_f<D, 8, 128>(); launch_f<D, 8, 128>(tab, mb, nb, ms, ns, s1, s2); return SPH_OK; }
  }
  return SPH_ERR_ARG;
}

int layout_any(int D, int P, int L, bool attr, const fused::LineTab* tab, const int2* mb, int nb, const int2* ms,
               int ns, cudaStream_t s1, cudaStream_t s2) {
  if (D == 0) return layout_f<0>(P, L, attr, tab, mb, nb, ms, ns, s1, s2);
  if (D == 1) return layout_f<1>(P, L, attr, tab, mb, nb, ms, ns, s1, s2);
  return layout_f<2>(P, L, attr, tab, mb, nb, ms, ns, s1, s2);
}

// the problems of one batch whose lines along d share a layout (P, L)
struct Layout {
  int d, P, L;
  std::vector<int> q;                 // problems (batch indices)
  size_t tab[2][2];                   // LineTab arrays per (step parity, later iteration)
  size_t mb, ms;                      // block maps
  int nb, ns;                         // blocks of the block-line and scalar-line launches
};

}  // namespace

void batch_fused_free(sph_batch* b) {
  if (!b) return;
  if (b->ftab) {
    cudaStreamSynchronize(b->st);
    cudaFree(b->ftab);
    b->ftab = NULL;
  }
  for (int q = 0; q < b->fstreams; q++) {
    cudaStreamDestroy(b->fst[q]);
    cudaEventDestroy(b->fjoin[q]);
  }
  if (b->fstreams) cudaEventDestroy(b->ffork);
  b->fstreams = 0;
}

// n side streams wait for what the batch stream holds so far / the batch
// stream waits for them (stream-ordered, so the capture records the edges)
static int ffork(sph_batch* b, int n) {
  if (cudaEventRecord(b->ffork, b->st) != cudaSuccess) return SPH_ERR_CUDA;
  for (int q = 0; q < n; q++)
    if (cudaStreamWaitEvent(b->fst[q], b->ffork, 0) != cudaSuccess) return SPH_ERR_CUDA;
  return SPH_OK;
}
static int fjoin(sph_batch* b, int n) {
  for (int q = 0; q < n; q++)
    if (cudaEventRecord(b->fjoin[q], b->fst[q]) != cudaSuccess || cudaStreamWaitEvent(b->st, b->fjoin[q], 0) != cudaSuccess)
      return SPH_ERR_CUDA;
  return SPH_OK;
}

extern "C" int sph_batch_capture_fused(sph_batch* b, double dt, int n_iter, int steps) {
  if (!b || !(dt > 0) || n_iter < 1 || steps < 2 || (steps & 1)) return SPH_ERR_ARG;
  const int n = b->n;
  for (int q = 0; q < n; q++) {
    const sph_ctx* c = b->c[q];
    if (c->prof || c->prec != SPH_PREC_MIXED || c->hasbc || c->d32.g.hasw || c->line_solver == SPH_LINES_THOMAS)
      return SPH_ERR_ARG;
    for (int d = 0; d < 3; d++)
      if (!lines_ok(c, d)) return SPH_ERR_ARG;
  }
  // work the contexts have queued (state uploads) is finished before the
  // tables are built and the graph is first replayed on the batch stream
  for (int q = 0; q < n; q++)
    if (cudaStreamSynchronize(b->c[q]->st) != cudaSuccess) return SPH_ERR_CUDA;
  if (b->exec) {
    cudaStreamSynchronize(b->st);
    cudaGraphExecDestroy(b->exec);
    b->exec = NULL;
  }
  if (b->graph) { cudaGraphDestroy(b->graph); b->graph = NULL; }
  if (b->ftab) { cudaFree(b->ftab); b->ftab = NULL; }
  if (!b->fstreams) {
    if (cudaEventCreateWithFlags(&b->ffork, cudaEventDisableTiming) != cudaSuccess) return SPH_ERR_CUDA;
    for (int q = 0; q < SPH_FUSED_STREAMS; q++) {
      if (cudaStreamCreateWithFlags(&b->fst[q], cudaStreamNonBlocking) != cudaSuccess ||
          cudaEventCreateWithFlags(&b->fjoin[q], cudaEventDisableTiming) != cudaSuccess) {
        b->fstreams = q + 1;  // batch_fused_free destroys what was made (a failed create leaves a null handle)
        batch_fused_free(b);
        return SPH_ERR_CUDA;
      }
      b->fstreams = q + 1;
    }
  }

  Blob blob;
  // ---- averaging: tables per (step parity, later iteration), one map
  std::vector<AvgArgs<float>> avg[2][2];
  std::vector<int4> mavg;
  // ---- stencil stages
  std::vector<fused::StenTab> coef(n);
  std::vector<fused::StenTab> rhs[2][2];
  std::vector<int2> msten;
  std::vector<double*> accs(n);
  for (int p = 0; p < 2; p++)
    for (int it = 0; it < 2; it++) {
      avg[p][it].resize(n);
      rhs[p][it].resize(n);
    }
  for (int q = 0; q < n; q++) {
    sph_ctx* c = b->c[q];
    Bufs<float>& B = c->d32;
    const Geo<double>& g = c->d64.g;
    accs[q] = c->acc;
    for (int p = 0; p < 2; p++)
      for (int it = 0; it < 2; it++) {
        const int cur = c->cur ^ p;
        double* const* un = c->U[cur];
        double* const* uk = it ? c->U[1 - cur] : un;
        AvgArgs<float>& A = avg[p][it][q];
        memset(&A, 0, sizeof A);
        A.same = !it;
        for (int f = 0; f < 5; f++) {
          A.a[f] = un[f]; A.b[f] = uk[f]; A.o[f] = B.Ub[f]; A.lo[f] = B.UbLo[f]; A.d[f] = B.Db[f];
          A.n[f] = (long)c->nf[f];
        }
        fused::StenTab& R = rhs[p][it][q];
        memset(&R, 0, sizeof R);
        s32_fill(c, cf5(B.Ub), dt, &R.A);
        R.A.hasD = it;
      }
    int nb;
    fused::Tile tc = tile_of(c, g.np, g.nt, g.nr, &nb);
    fused::StenTab& C = coef[q];
    memset(&C, 0, sizeof C);
    s32_fill(c, cf5(B.Ub), dt, &C.A);
    C.t = tc;
    for (int p = 0; p < 2; p++)
      for (int it = 0; it < 2; it++) rhs[p][it][q].t = tc;
    // a block per fused::TILES consecutive tiles of the problem
    for (int k = 0; k < nb; k += fused::TILES) msten.push_back(make_int2(q, k));
    for (int f = 0; f < 5; f++) {
      const long pairs = (long)c->nf[f] >> 1;
      for (long s = 0; s < pairs || (s == 0 && pairs == 0); s += 1024)
        mavg.push_back(make_int4(q, f, (int)s, (int)(pairs - s < 1024 ? pairs - s : 1024)));
    }
  }
  // ---- line layouts of each direction
  std::vector<Layout> lay;
  std::vector<fused::LineTab> ltab[64][2][2];   // per layout (at most 3 x 15 exist)
  std::vector<int2> lmb[64], lms[64];
  // r and theta: the lines of all problems, whatever their lengths, in one pair of
  // launches where the batch has enough of them to fill the SMs.  A problem's own
  // choice among the partitioned layouts then counts for its phi lines alone: a pair of
  // launches for every layout chosen costs what the layouts gain (the ensemble of 64, 4
  // of 45 grids with the one-warp layout: 33.33 ms a step with their own launches, 33.28
  // without; 12 instances 7.16 against 7.05).
  bool two[3] = {false, false, false};
  std::vector<lines2::Args> l2tab[2];
  std::vector<int2> l2b[2], l2s[2];
  for (int d = 0; d < 2; d++) {
    long lines = 0;
    for (int q = 0; q < n; q++) {
      const Geo<double>& g = b->c[q]->d64.g;
      lines += (long)(d == 0 ? g.nt : g.nr) * g.np;
    }
    two[d] = lines >= LINES2_MIN;
    for (int q = 0; q < n && two[d]; q++) {
      sph_ctx* c = b->c[q];
      Bufs<float>& B = c->d32;
      lines2::Args A;
      int nb0, ns;
      lines2_fill(c, d, dt, cf5(B.Ub), cf5(d == 1 ? B.X1 : B.Rb), mf5(d == 1 ? B.Rb : B.X1), &A, &nb0, &ns);
      l2tab[d].push_back(A);
      for (int k = 0; k < nb0; k++) l2b[d].push_back(make_int2(q, k));
      for (int k = 0; k < ns; k++) l2s[d].push_back(make_int2(q, k));
    }
  }
  for (int d = 0; d < 3; d++)
    for (int q = 0; q < n && !two[d]; q++) {
      sph_ctx* c = b->c[q];
      const Geo<double>& g = c->d64.g;
      const int len = d == 0 ? g.nr : d == 1 ? g.nt : g.np;
      int P = 0, L = 0;
      lines_pl(c->line_solver, d, len, &P, &L);
      int li = -1;
      for (int z = 0; z < (int)lay.size(); z++)
        if (lay[z].d == d && lay[z].P == P && lay[z].L == L) li = z;
      if (li < 0) {
        if (lay.size() >= 64) return SPH_ERR_ARG;
        Layout Ly;
        Ly.d = d; Ly.P = P; Ly.L = L; Ly.nb = Ly.ns = 0; Ly.mb = Ly.ms = 0;
        lay.push_back(Ly);
        li = (int)lay.size() - 1;
      }
      Layout& Ly = lay[li];
      const int e = (int)Ly.q.size();
      Ly.q.push_back(q);
      const int CB = lines_cb(d, len), NW = CB / len, NWW = CB / P / 32;
      Bufs<float>& B = c->d32;
      int ng[3] = {0, 0, 0};
      for (int p = 0; p < 2; p++)
        for (int it = 0; it < 2; it++) {
          const int cur = c->cur ^ p;
          double* const* un = c->U[cur];
          double* const* uk = it ? c->U[1 - cur] : un;
          fused::LineTab T;
          memset(&T, 0, sizeof T);
          SweepArgs<float>& S = T.S;
          S.g = B.g; S.P = c->P; S.c = B.c; S.ub = cf5(B.Ub); S.d = d; S.h = (float)(0.5 * dt);
          S.rhs = cf5(d == 1 ? B.X1 : B.Rb);
          S.x = mf5(d == 1 ? B.Rb : B.X1);
          S.update = d == 2;
          S.base = cf5(uk);
          S.uk = mf5(c->U[1 - cur]);
          S.scr = B.scr; S.acc = c->acc; S.flag = c->flag;
          line_layout(g, d, S);
          lines2_rows(c, d, dt, &S);
          S.norms = 1;
          for (int k = 0; k < 3; k++) ng[k] = lines_groups(S, k, NW);
          T.ng1 = ng[1];
          ltab[li][p][it].push_back(T);
        }
      // one factor slot per warp of the block-line launch (as in the single-problem path)
      if ((size_t)ng[0] * NWW * 32 * lines::slot_floats(P) > c->nscr) return SPH_ERR_ARG;
      for (int k = 0; k < ng[0]; k++) lmb[li].push_back(make_int2(e, k));
      for (int k = 0; k < ng[1] + ng[2]; k++) lms[li].push_back(make_int2(e, k));
    }
  // ---- one device buffer
  size_t oavg[2][2], orhs[2][2];
  for (int p = 0; p < 2; p++)
    for (int it = 0; it < 2; it++) {
      oavg[p][it] = blob.put(avg[p][it]);
      orhs[p][it] = blob.put(rhs[p][it]);
    }
  const size_t ocoef = blob.put(coef), omavg = blob.put(mavg), omsten = blob.put(msten), oacc = blob.put(accs);
  size_t ol2[2], ol2b[2], ol2s[2];
  for (int d = 0; d < 2; d++) { ol2[d] = blob.put(l2tab[d]); ol2b[d] = blob.put(l2b[d]); ol2s[d] = blob.put(l2s[d]); }
  for (size_t z = 0; z < lay.size(); z++) {
    for (int p = 0; p < 2; p++)
      for (int it = 0; it < 2; it++) lay[z].tab[p][it] = blob.put(ltab[z][p][it]);
    lay[z].mb = blob.put(lmb[z]);
    lay[z].ms = blob.put(lms[z]);
    lay[z].nb = (int)lmb[z].size();
    lay[z].ns = (int)lms[z].size();
  }
  if (cudaMalloc(&b->ftab, blob.h.size()) != cudaSuccess) { cudaGetLastError(); b->ftab = NULL; return SPH_ERR_NOMEM; }
  if (cudaMemcpy(b->ftab, blob.h.data(), blob.h.size(), cudaMemcpyHostToDevice) != cudaSuccess) return SPH_ERR_CUDA;
  char* base = (char*)b->ftab;
  for (size_t z = 0; z < lay.size(); z++)
    if (int e = layout_any(lay[z].d, lay[z].P, lay[z].L, true, NULL, NULL, 0, NULL, 0, NULL, NULL)) return e;
  // ---- the graph: `steps` steps of every problem
  for (int q = 0; q < n; q++) { b->cur[q] = b->c[q]->cur; b->nlaunch[q] = 0; }
  long long nk = 0;
  if (cudaStreamBeginCapture(b->st, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return SPH_ERR_CUDA;
  int err = SPH_OK;
  for (int s = 0; s < steps && !err; s++) {
    const int p = s & 1;
    for (int it = 0; it < n_iter && !err; it++) {
      const int il = it > 0;
      fused::k_avg_f<<<(unsigned)mavg.size(), 256, 0, b->st>>>((const AvgArgs<float>*)(base + oavg[p][il]),
                                                               (const int4*)(base + omavg));
      fused::k_coef_f<<<(unsigned)msten.size(), 128, 0, b->st>>>((const fused::StenTab*)(base + ocoef),
                                                                (const int2*)(base + omsten));
      nk += 2;
      const fused::StenTab* rt = (const fused::StenTab*)(base + orhs[p][il]);
      fused::k_rhs_f<<<(unsigned)msten.size(), 128, 0, b->st>>>(rt, (const int2*)(base + omsten));
      nk++;
      for (int d = 0; d < 3 && !err; d++) {
        if (d == 2 && it == n_iter - 1) {
          fused::k_zero_acc_f<<<(5 * n + 255) / 256, 256, 0, b->st>>>((double* const*)(base + oacc), n);
          nk++;
        }
        if (two[d]) {
          if ((err = ffork(b, 1))) break;
          const lines2::Args* lt = (const lines2::Args*)(base + ol2[d]);
          const int2 *mb = (const int2*)(base + ol2b[d]), *ms = (const int2*)(base + ol2s[d]);
          const unsigned nb = (unsigned)l2b[d].size(), ns = (unsigned)l2s[d].size();
          if (d == 0) {
            fused::k_l2_blk_f<0><<<nb, 64, 0, b->st>>>(lt, mb);
            fused::k_l2_sca_f<0><<<ns, 64, 0, b->fst[0]>>>(lt, ms);
          } else {
            fused::k_l2_blk_f<1><<<nb, 64, 0, b->st>>>(lt, mb);
            fused::k_l2_sca_f<1><<<ns, 64, 0, b->fst[0]>>>(lt, ms);
          }
          nk += 2;
          err = fjoin(b, 1);
          continue;
        }
        int used = 0;
        for (size_t z = 0; z < lay.size(); z++) used += lay[z].d == d ? 2 : 0;
        used = used < SPH_FUSED_STREAMS ? used : SPH_FUSED_STREAMS;
        if ((err = ffork(b, used))) break;
        int slot = 0;
        for (size_t z = 0; z < lay.size() && !err; z++) {
          const Layout& Ly = lay[z];
          if (Ly.d != d) continue;
          cudaStream_t s1 = b->fst[slot % SPH_FUSED_STREAMS], s2 = b->fst[(slot + 1) % SPH_FUSED_STREAMS];
          slot += 2;
          err = layout_any(d, Ly.P, Ly.L, false, (const fused::LineTab*)(base + Ly.tab[p][il]),
                           (const int2*)(base + Ly.mb), Ly.nb, (const int2*)(base + Ly.ms), Ly.ns, s1, s2);
          nk += (Ly.nb > 0) + (Ly.ns > 0);
        }
        if (!err) err = fjoin(b, used);
      }
      if (!err && cudaGetLastError() != cudaSuccess) err = SPH_ERR_CUDA;
    }
  }
  cudaGraph_t gr = NULL;
  cudaError_t ce = cudaStreamEndCapture(b->st, &gr);
  if (!err && ce != cudaSuccess) err = SPH_ERR_CUDA;
  if (!err && cudaGraphInstantiate(&b->exec, gr, 0) != cudaSuccess) err = SPH_ERR_CUDA;
  if (err) {
    if (gr) cudaGraphDestroy(gr);
    b->exec = NULL;
    cudaGetLastError();
    return err;
  }
  b->graph = gr;
  b->nlaunch[0] = nk;  // the batched kernels are shared: counted once, on the first problem
  return SPH_OK;
}

#ifdef SPH_CHECKED
int bounds_take_batch(int* h) {
  int z[5] = {0, 0, 0, 0, 0};
  if (cudaMemcpyFromSymbol(h, g_bounds, 5 * sizeof(int)) != cudaSuccess ||
      cudaMemcpyToSymbol(g_bounds, z, sizeof z) != cudaSuccess)
    return SPH_ERR_CUDA;
  return SPH_OK;
}
#endif
