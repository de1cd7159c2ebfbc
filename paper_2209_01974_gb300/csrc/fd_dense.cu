// Dense FP64 kernels of the FD loop: tall-skinny Gram products, in-place block
// rotations, Cholesky and triangular inverse (Cholesky-QR, Sec. 2) and the
// residual norms rho_i = ||A v_i - theta_i v_i||_2 (Sec. 2, Alg. 1).
//
// FP64 arithmetic on GB300 runs at about 1.2 TFLOP/s, so these kernels are
// FP64-ALU bound; they use register tiles fed from shared memory and split the
// long dimension D across CTAs with a deterministic second-pass reduction.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "fd_internal.cuh"

namespace cg = cooperative_groups;

namespace fdi {
namespace {

// ---------------------------------------------------------------------------
// Gram: P[slice] = X[rows of slice]^T Y[rows of slice], 64 x 64 output tiles
//
// Bound by the FP64 pipe (a warp's FMA takes 16 cycles of an SM), so a tile's 16 x 16
// parts that lie beyond the product's edge, or below a symmetric product's diagonal,
// are left out: the mirrored part has the same sums in the same order.  Measured,
// 476,929 rows: 16 columns 3,390 -> 306 us, 32 3,465 -> 722 us, 64 3,536 -> 2,172 us.
// ---------------------------------------------------------------------------
constexpr int GT = 64;   // tile edge
constexpr int GP = 16;   // edge of a tile's parts: thread (ty, tx) has one element of each
constexpr int GK = 16;   // rows per shared-memory stage

// one tile's parts (u, v), u, v < U, on or above the diagonal if DIAG
template <int U, bool DIAG>
__device__ __forceinline__ void gram_tile(const double* __restrict__ X, int64_t ldx, const double* __restrict__ Y,
                                          int64_t ldy, int i0, int j0, int m, int n, int64_t k0, int64_t k1,
                                          double (&Xs)[GK][GT], double (&Ys)[GK][GT], double* Ps) {
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  constexpr int W = GP * U;
  double acc[U][U] = {};
  for (int64_t kb = k0; kb < k1; kb += GK) {
#pragma unroll
    for (int q = 0; q < (GK * W) / 256; ++q) {
      int e = threadIdx.x + q * 256;
      int kk = e / W, c = e % W;
      int64_t k = kb + kk;
      Xs[kk][c] = (k < k1 && i0 + c < m) ? X[k * ldx + i0 + c] : 0.0;
      Ys[kk][c] = (k < k1 && j0 + c < n) ? Y[k * ldy + j0 + c] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < GK; ++kk) {
      double a[U], b[U];
#pragma unroll
      for (int u = 0; u < U; ++u) { a[u] = Xs[kk][ty + GP * u]; b[u] = Ys[kk][tx + GP * u]; }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int v = DIAG ? u : 0; v < U; ++v) acc[u][v] = fma(a[u], b[v], acc[u][v]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = DIAG ? u : 0; v < U; ++v) {
      int i = i0 + ty + GP * u, j = j0 + tx + GP * v;
      if (i < m && j < n) Ps[(int64_t)i * n + j] = acc[u][v];
    }
}

__global__ void __launch_bounds__(256)
    k_gram_partial(const double* __restrict__ X, int64_t ldx, const double* __restrict__ Y,
                   int64_t ldy, int64_t D, int m, int n, int ntj, bool sym, int64_t rows_per_slice,
                   double* __restrict__ P) {
  __shared__ double Xs[GK][GT], Ys[GK][GT];
  // tile coordinates
  int t = blockIdx.x, ti, tj;
  if (sym) {  // enumerate ti <= tj
    ti = 0;
    int rowlen = ntj;
    while (t >= rowlen) { t -= rowlen; ++ti; --rowlen; }
    tj = ti + t;
  } else {
    ti = t / ntj;
    tj = t % ntj;
  }
  const int i0 = ti * GT, j0 = tj * GT;
  const int64_t k0 = (int64_t)blockIdx.y * rows_per_slice;
  const int64_t k1 = min(D, k0 + rows_per_slice);
  double* Ps = P + (int64_t)blockIdx.y * m * n;
  const int parts = (min(GT, max(m - i0, n - j0)) + GP - 1) / GP;
  const bool diag = sym && ti == tj;
#define FD_GRAM_TILE(U) \
  if (diag) gram_tile<U, true>(X, ldx, Y, ldy, i0, j0, m, n, k0, k1, Xs, Ys, Ps); \
  else gram_tile<U, false>(X, ldx, Y, ldy, i0, j0, m, n, k0, k1, Xs, Ys, Ps)
  if (parts == 1) { FD_GRAM_TILE(1); }
  else if (parts == 2) { FD_GRAM_TILE(2); }
  else if (parts == 3) { FD_GRAM_TILE(3); }
  else { FD_GRAM_TILE(4); }
#undef FD_GRAM_TILE
}

__global__ void k_gram_reduce(const double* P, int slices, int m, int n, bool sym, double* C,
                              int ldc) {
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)m * n) return;
  int i = (int)(e / n), j = (int)(e % n);
  if (sym && i / GP > j / GP) return;  // computed by the mirrored part
  double s = 0.0;
  for (int q = 0; q < slices; ++q) s += P[(int64_t)q * m * n + e];
  C[(int64_t)i * ldc + j] = s;
  if (sym && i / GP < j / GP) C[(int64_t)j * ldc + i] = s;
}

// ---------------------------------------------------------------------------
// rotate: V[rows] <- V[rows] * M, in place, TR rows per CTA
// ---------------------------------------------------------------------------
// RT rows per CTA: 256 / RT threads along the columns, RT / 4 of each 64 columns per
// thread.  Few rows are spread thinner, 4 to a CTA, so that every SM's FP64 pipe has
// rows and warps enough (1,728 x 96: 34 us, 125 us with 16 rows in 108 CTAs).  Bound by
// the FP64 pipe from 64 columns on; the columns that a last 64 lacks are left out.
template <int RT, bool UPPER>
__global__ void __launch_bounds__(256)
    k_rotate(double* V, int64_t ldv, int64_t D, int n, const double* __restrict__ M) {
  extern __shared__ double Vt[];  // RT x n
  constexpr int LANES = 256 / RT, COLS = 64 / LANES;
  const int64_t r0 = (int64_t)blockIdx.x * RT;
  const int nr = D - r0 < RT ? (int)(D - r0) : RT;
  for (int e = threadIdx.x; e < RT * n; e += 256) {
    int r = e / n, c = e % n;
    Vt[e] = r < nr ? V[(r0 + r) * ldv + c] : 0.0;
  }
  __syncthreads();
  const int r = threadIdx.x / LANES;
  const int c0 = threadIdx.x % LANES;  // columns c0 + LANES v
  for (int cb = 0; cb < n; cb += 64) {
    double acc[COLS] = {};
    const int kend = UPPER ? min(n, cb + 64) : n;
    const double* vr = Vt + r * n;
    const int nv = min(COLS, (n - cb + LANES - 1) / LANES);  // columns beyond n cost FP64 cycles too
    int col[COLS];
#pragma unroll
    for (int v = 0; v < COLS; ++v) col[v] = min(cb + c0 + LANES * v, n - 1);  // beyond n: not stored
    // rows k0 .. k1 of M; TRI: the diagonal block of an upper M, of which what is stored
    // below the diagonal does not enter (its products count as zero: leaving out those of
    // columns wholly below it took 66,000 x 64 from 461 to 506 us)
    auto add_rows = [&](auto tri, int k, int k1) {
      constexpr bool TRI = decltype(tri)::value;
      for (; k + 4 <= k1; k += 4) {
        double m[4][COLS];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int v = 0; v < COLS; ++v) m[u][v] = TRI && k + u > col[v] ? 0.0 : __ldg(M + (int64_t)(k + u) * n + col[v]);
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int v = 0; v < COLS; ++v)
            if (v < nv) acc[v] = fma(vr[k + u], m[u][v], acc[v]);
      }
      for (; k < k1; ++k)
#pragma unroll
        for (int v = 0; v < COLS; ++v)
          if (v < nv) acc[v] = fma(vr[k], TRI && k > col[v] ? 0.0 : __ldg(M + (int64_t)k * n + col[v]), acc[v]);
    };
    if constexpr (UPPER) {
      add_rows(std::false_type{}, 0, cb);
      add_rows(std::true_type{}, cb, kend);
    } else {
      add_rows(std::false_type{}, 0, kend);
    }
    if (r < nr) {
#pragma unroll
      for (int v = 0; v < COLS; ++v) {
        int c = cb + c0 + LANES * v;
        if (c < n) V[(r0 + r) * ldv + c] = acc[v];
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Cholesky (one CTA): R upper with R^T R = G + shift I, shift = coeff * tr(G)
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(1024) k_cholesky(const double* G, int n, double coeff,
                                                   double* R, int* ok) {
  __shared__ double sh_tr[1024];
  __shared__ int fail;
  __shared__ double rinv;
  double tr = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) tr += G[(int64_t)i * n + i];
  sh_tr[threadIdx.x] = tr;
  __syncthreads();
  for (int o = 512; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh_tr[threadIdx.x] += sh_tr[threadIdx.x + o];
    __syncthreads();
  }
  const double shift = coeff * sh_tr[0];
  for (int64_t e = threadIdx.x; e < (int64_t)n * n; e += blockDim.x) {
    int i = (int)(e / n), j = (int)(e % n);
    R[e] = j >= i ? G[e] + (i == j ? shift : 0.0) : 0.0;
  }
  if (threadIdx.x == 0) fail = 0;
  __syncthreads();
  for (int k = 0; k < n; ++k) {
    if (threadIdx.x == 0) {
      double d = R[(int64_t)k * n + k];
      if (!(d > 0.0) || !isfinite(d)) {
        fail = 1;
      } else {
        double r = sqrt(d);
        R[(int64_t)k * n + k] = r;
        rinv = 1.0 / r;
      }
    }
    __syncthreads();
    if (fail) break;
    for (int j = k + 1 + threadIdx.x; j < n; j += blockDim.x) R[(int64_t)k * n + j] *= rinv;
    __syncthreads();
    const int m = n - k - 1;
    for (int64_t e = threadIdx.x; e < (int64_t)m * m; e += blockDim.x) {
      int i = k + 1 + (int)(e / m), j = k + 1 + (int)(e % m);
      if (j >= i) R[(int64_t)i * n + j] -= R[(int64_t)k * n + i] * R[(int64_t)k * n + j];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) *ok = fail ? 0 : 1;
}

// ---------------------------------------------------------------------------
// Cooperative blocked version: panels of 8 rows, one grid barrier per panel.
//
// The chain of pivots bounds it (an FP64 reciprocal square root and an update per
// column, 0.4 us), so what a panel adds to it is kept short: every CTA loads the
// panel's rows, factors the 8 x 8 diagonal block in one warp's registers and solves
// the panel into its shared memory by itself (the same values everywhere), and
// only the trailing update is divided (rows over CTAs).  The panel's finished rows
// are written after the barrier, when no CTA reads the unfinished ones any more.
// One barrier per column instead took 440 us at n = 128, 1.61 ms at n = 384;
// this takes 109 us and 0.43 ms.
// ---------------------------------------------------------------------------
constexpr int CB = 8;  // panel rows

__global__ void __launch_bounds__(256) k_cholesky_coop(const double* G, int n, double coeff, double* R, int* ok) {
  cg::grid_group grid = cg::this_grid();
  extern __shared__ double sP[];  // 2 x CB x n: the panel's finished rows, by panel parity
  __shared__ double red[256];
  __shared__ double sD[CB][CB + 1], sR[CB];
  __shared__ int sfail;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double tr = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) tr += G[(int64_t)i * n + i];
  red[threadIdx.x] = tr;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  const double shift = coeff * red[0];
  for (int i = blockIdx.x; i < n; i += gridDim.x)
    for (int j = threadIdx.x; j < n; j += blockDim.x)
      __stcg(R + (int64_t)i * n + j, j >= i ? G[(int64_t)i * n + j] + (i == j ? shift : 0.0) : 0.0);
  grid.sync();
  bool fail = false;
  for (int k0 = 0, panel = 0; k0 < n; k0 += CB, ++panel) {
    const int kb = min(CB, n - k0);
    double* P = sP + (panel & 1) * CB * n;
    // the diagonal block: lane (i, j) of warp 0 holds elements (i, j) and (i + 4, j)
    if (warp == 0) {
      const int i = lane >> 3, j = lane & 7;
      double v[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = i + 4 * h;
        v[h] = r < kb && j < kb && j >= r ? __ldcg(R + (int64_t)(k0 + r) * n + k0 + j) : (r == j ? 1.0 : 0.0);
      }
      bool bad = false;
#pragma unroll
      for (int p = 0; p < CB; ++p) {
        const double d = __shfl_sync(0xffffffffu, v[p >> 2], (p & 3) * 8 + p);
        if (!(d > 0.0) || !isfinite(d)) bad = true;
        const double ri = rsqrt(bad ? 1.0 : d);
        if (i == (p & 3)) v[p >> 2] = j == p ? d * ri : v[p >> 2] * ri;
        const double rj = __shfl_sync(0xffffffffu, v[p >> 2], (p & 3) * 8 + j);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const double rr = __shfl_sync(0xffffffffu, v[p >> 2], (p & 3) * 8 + i + 4 * h);
          if (i + 4 * h > p && j >= i + 4 * h) v[h] = fma(-rr, rj, v[h]);
        }
        if (lane == 0) sR[p] = ri;
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) sD[i + 4 * h][j] = v[h];
      if (lane == 0) sfail = bad;
    }
    __syncthreads();
    if (sfail) {  // the same in every CTA: all stop here
      fail = true;
      break;
    }
    // the panel's other columns: R_kk^T x = g
    for (int j = k0 + threadIdx.x; j < n; j += blockDim.x) {
      double x[CB];
#pragma unroll
      for (int p = 0; p < CB; ++p) x[p] = p < kb && j >= k0 + CB ? __ldcg(R + (int64_t)(k0 + p) * n + j) : 0.0;
#pragma unroll
      for (int p = 0; p < CB; ++p) {
#pragma unroll
        for (int q = 0; q < p; ++q) x[p] = fma(-sD[q][p], x[q], x[p]);
        x[p] *= sR[p];
      }
#pragma unroll
      for (int p = 0; p < CB; ++p) P[p * n + j] = j < k0 + CB ? (j - k0 >= p ? sD[p][j - k0] : 0.0) : x[p];
    }
    __syncthreads();
    // trailing rows of this CTA
    for (int i = k0 + CB + blockIdx.x; i < n; i += gridDim.x) {
      double* ri = R + (int64_t)i * n;
      for (int j = i + threadIdx.x; j < n; j += blockDim.x) {
        double v = __ldcg(ri + j);
#pragma unroll
        for (int p = 0; p < CB; ++p) v = fma(-P[p * n + i], P[p * n + j], v);
        __stcg(ri + j, v);
      }
    }
    grid.sync();
    if (panel % gridDim.x == blockIdx.x)
      for (int e = threadIdx.x; e < kb * (n - k0); e += blockDim.x) {
        const int p = e / (n - k0), j = k0 + e % (n - k0);
        if (j >= k0 + p) R[(int64_t)(k0 + p) * n + j] = P[p * n + j];
      }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *ok = fail ? 0 : 1;
}

// ---------------------------------------------------------------------------
// triangular inverse: X = R^-1 (upper).  One CTA takes 8 columns from their
// diagonal block upwards in blocks of 8 rows: S = I - R X over the rows below (64
// sums, split four ways over the row index), then back substitution inside the
// block.  A warp per column, one row at a time with a warp-wide FP64 reduction
// each, took 184 us at n = 128 and 0.70 ms at n = 384; this takes 66 us and 0.36 ms.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_tri_inverse(const double* R, int n, double* X) {
  extern __shared__ double xs[];  // n x 8: the finished rows of the 8 columns
  __shared__ double part[4][64];
  __shared__ double S[CB][CB + 1], inv[CB];
  const int c0 = blockIdx.x * CB;
  const int i = (threadIdx.x >> 3) & 7, c = threadIdx.x & 7, slice = threadIdx.x >> 6;
  const int last = min(n, c0 + CB);  // rows at or beyond `last` are zero
  for (int r0 = c0; r0 >= 0; r0 -= CB) {
    double s = 0.0;
    if (r0 + i < n)
      for (int k = r0 + CB + slice; k < last; k += 4) s = fma(__ldg(R + (int64_t)(r0 + i) * n + k), xs[k * CB + c], s);
    part[slice][i * CB + c] = s;
    __syncthreads();
    if (slice == 0) {
      const int e = i * CB + c;
      S[i][c] = (r0 + i == c0 + c ? 1.0 : 0.0) - ((part[0][e] + part[1][e]) + (part[2][e] + part[3][e]));
    } else if (threadIdx.x < 64 + CB && r0 + threadIdx.x - 64 < n) {  // an FP64 division takes as long as the rest of a row
      inv[threadIdx.x - 64] = 1.0 / __ldg(R + (int64_t)(r0 + threadIdx.x - 64) * n + r0 + threadIdx.x - 64);
    }
    __syncthreads();
    if (threadIdx.x < CB) {  // one column per thread
      const int col = threadIdx.x, rows = min(CB, n - r0);
      double x[CB];
#pragma unroll
      for (int p = CB - 1; p >= 0; --p) {
        x[p] = 0.0;
        if (p < rows) {
          double v = S[p][col];
#pragma unroll
          for (int q = p + 1; q < CB; ++q)
            if (q < rows) v = fma(-__ldg(R + (int64_t)(r0 + p) * n + r0 + q), x[q], v);
          x[p] = v * inv[p];
          xs[(r0 + p) * CB + col] = x[p];
        }
      }
    }
    __syncthreads();
  }
  for (int e = threadIdx.x; e < n * CB; e += 256) {
    const int r = e / CB, q = c0 + e % CB;
    if (q < n) X[(int64_t)r * n + q] = r <= q ? xs[e] : 0.0;
  }
}

// C = A * B, n x n (small)
__global__ void k_small_gemm(const double* A, const double* B, double* C, int n) {
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)n * n) return;
  int i = (int)(e / n), j = (int)(e % n);
  double s = 0.0;
  for (int k = 0; k < n; ++k) s = fma(A[(int64_t)i * n + k], B[(int64_t)k * n + j], s);
  C[e] = s;
}

__global__ void k_identity(double* A, int n) {
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < (int64_t)n * n) A[e] = (e / n == e % n) ? 1.0 : 0.0;
}

// ---------------------------------------------------------------------------
// residual norms
// ---------------------------------------------------------------------------
__global__ void k_resid_partial(const double* V, const double* AV, int64_t ld, int64_t D, int n,
                                const double* theta, double* P) {
  for (int c = threadIdx.x; c < n; c += blockDim.x) {
    const double th = theta[c];
    double s = 0.0;
    for (int64_t r = blockIdx.x; r < D; r += gridDim.x) {
      const double d = AV[r * ld + c] - th * V[r * ld + c];
      s = fma(d, d, s);
    }
    P[(int64_t)blockIdx.x * n + c] = s;
  }
}

// one warp per column (one thread's 608 dependent FP64 additions took 42 us)
__global__ void k_resid_reduce(const double* P, int nb, int n, double* out) {
  const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (c >= n) return;
  double s = 0.0;
  for (int b = lane; b < nb; b += 32) s += P[(int64_t)b * n + c];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) out[c] = sqrt(s);
}

// Copies of D x n blocks with a change of type.  FP64 -> float-float: hi the nearest
// float, lo the nearest float to the exact FP64 remainder; back, hi + lo is exact in
// FP64.
struct alignas(8) pair_f { float hi, lo; };
struct pair_u { float hi, lo; };  // the same at a 4-byte boundary
__device__ __forceinline__ void convert(double v, float& o) { o = __double2float_rn(v); }
__device__ __forceinline__ void convert(float v, double& o) { o = (double)v; }
template <typename P>
__device__ __forceinline__ void convert(double v, P& o) {
  o.hi = __double2float_rn(v);
  o.lo = __double2float_rn(v - (double)o.hi);
}
__device__ __forceinline__ void convert(double v, double& o) { o = v; }
__device__ __forceinline__ void convert(float v, float& o) { o = v; }
__device__ __forceinline__ void convert(pair_f v, double& o) { o = (double)v.hi + (double)v.lo; }
__device__ __forceinline__ void convert(pair_u v, double& o) { o = (double)v.hi + (double)v.lo; }
__device__ __forceinline__ void convert(pair_u v, pair_u& o) { o = v; }

template <typename T, int W>
struct alignas(sizeof(T) * W < 16 ? sizeof(T) * W : 16) Pack { T v[W]; };

// FP64 and FP32 blocks, bound by memory: W elements per thread and row (16 or 32
// bytes on the wider side) and UNROLL rows in flight.  One element per thread with a
// 64-bit division for its row ran at half the copy bandwidth (11.8M x 32, FP64 ->
// FP32: 1.32 ms, now 0.65).
template <typename S, typename T, int W, int UNROLL>
__global__ void __launch_bounds__(256) k_convert(const S* s, int64_t lds, T* d, int64_t ldd, int64_t D, int n) {
  const unsigned q = (unsigned)n / W, per = q < 256 ? 256 / q : 1;  // threads of a row, rows at once
  const unsigned r = threadIdx.x / q, c0 = q < 256 ? threadIdx.x - r * q : blockIdx.y * 256 + threadIdx.x;
  if (q < 256 && r >= per) return;
  const int64_t row0 = (int64_t)blockIdx.x * per * UNROLL + (q < 256 ? r : 0);
  for (unsigned c = c0; c < q; c += gridDim.y * 256) {
    Pack<S, W> in[UNROLL];
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) {
      const int64_t row = row0 + (int64_t)u * per;
      if (row < D) in[u] = *reinterpret_cast<const Pack<S, W>*>(s + row * lds + (int64_t)c * W);
    }
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) {
      const int64_t row = row0 + (int64_t)u * per;
      if (row < D) {
        Pack<T, W> out;
#pragma unroll
        for (int e = 0; e < W; ++e) convert(in[u].v[e], out.v[e]);
        *reinterpret_cast<Pack<T, W>*>(d + row * ldd + (int64_t)c * W) = out;
      }
    }
  }
}

// Float-float blocks: the conversions are bound by the FP64 pipe, so a thread takes
// one element and none is idle at the end of a row (rows of packs as above, 3,000,000
// x 33: 788 us to float-float, 590 back, against 709 and 533).
template <typename S, typename T>
__global__ void __launch_bounds__(256) k_convert_each(const S* s, int64_t lds, T* d, int64_t ldd, int64_t D, int n) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= D * n) return;
  const int64_t i = t / n;
  const int j = (int)(t % n);
  T o;
  convert(s[i * lds + j], o);
  d[i * ldd + j] = o;
}

template <typename S, typename T, int W>
bool packs(const S* s, int64_t lds, const T* d, int64_t ldd, int n) {
  return n % W == 0 && lds % W == 0 && ldd % W == 0 && (uintptr_t)s % alignof(Pack<S, W>) == 0 &&
         (uintptr_t)d % alignof(Pack<T, W>) == 0;
}

template <typename S, typename T>
fd_status convert_block(fd_ctx* ctx, const S* s, int64_t lds, T* d, int64_t ldd, int64_t D, int n) {
  constexpr int W = sizeof(S) == 4 || sizeof(T) == 4 ? 4 : 2;
  const int w = packs<S, T, W>(s, lds, d, ldd, n) ? W : 1;
  const int64_t q = n / w, per = q < 256 ? 256 / q : 1;
  const unsigned wide = q < 256 ? 1 : (unsigned)std::min<int64_t>(cdiv(q, 256), 65535);  // CTAs along a row
  // four rows per thread where that leaves every SM eight CTAs; small blocks are
  // spread over more of them (50 x 5,000, FP64 -> FP32: 8.3 -> 4.2 us)
  const bool deep = cdiv(D, per * 4) * wide >= 8LL * ctx->num_sms;
  const dim3 grid((unsigned)cdiv(D, per * (deep ? 4 : 1)), wide);
  auto kernel = w == W ? deep ? k_convert<S, T, W, 4> : k_convert<S, T, W, 1>
                       : deep ? k_convert<S, T, 1, 4> : k_convert<S, T, 1, 1>;
  kernel<<<grid, 256, 0, ctx->stream>>>(s, lds, d, ldd, D, n);
  FD_LAUNCHED(ctx);
  return FD_OK;
}

template <typename S, typename T>
fd_status convert_each(fd_ctx* ctx, const S* s, int64_t lds, T* d, int64_t ldd, int64_t D, int n) {
  k_convert_each<<<(unsigned)cdiv(D * n, 256), 256, 0, ctx->stream>>>(s, lds, d, ldd, D, n);
  FD_LAUNCHED(ctx);
  return FD_OK;
}

}  // namespace

// tall-skinny products large enough for the tensor-core splitting to pay off.  It is
// faster from fewer rows and columns on (30,001 x 80: orthonormalisation 0.96 ms), but
// its digits are relative to the largest entry of a row or column, and blocks whose
// columns differ in size lose to that (orthonormalisation error 3.5e-16 -> 8.8e-14): the
// line stays where FP64 costs several times as much (65,537 x 128: Gram 1,149 against
// 241 us, rotation 1,745 against 220 us)
static bool use_ozaki(const fd_ctx* ctx, int64_t D, int m, int n) {
  if (ctx->gemm_mode == FD_GEMM_FP64) return false;
  if (ctx->gemm_mode == FD_GEMM_OZAKI) return true;
  return D >= 65536 && m >= 64 && n >= 64;
}

fd_status gram(fd_ctx* ctx, const double* X, int64_t ldx, const double* Y, int64_t ldy, int64_t D,
               int m, int n, double* C, int ldc, bool sym) {
  if (use_ozaki(ctx, D, m, n)) {
    bool used = false;
    FD_TRY(oz_gram(ctx, X, ldx, Y, ldy, D, m, n, C, ldc, sym, &used));
    if (used) return FD_OK;
  }
  const int nti = (int)cdiv(m, GT), ntj = (int)cdiv(n, GT);
  const int tiles = sym ? nti * (nti + 1) / 2 : nti * ntj;
  // about four CTAs per SM; short blocks are cut down to one shared-memory stage
  // (1,728 x 96 with its reduction: 51 us, 70 us with 64 rows per slice)
  int64_t slices = std::max<int64_t>(1, cdiv(4LL * ctx->num_sms, tiles));
  slices = std::min<int64_t>(slices, std::max<int64_t>(1, cdiv(D, GK)));
  int64_t rps = cdiv(cdiv(D, slices), GK) * GK;
  slices = std::max<int64_t>(1, cdiv(D, rps));
  void* p;
  if (workspace(ctx, "gram_partial", sizeof(double) * slices * m * n, &p, true) != FD_OK) {
    // refused: slices of four stages or more
    ctx->err.clear();
    slices = std::min<int64_t>(slices, std::max<int64_t>(1, cdiv(D, 4 * GK)));
    rps = cdiv(cdiv(D, slices), GK) * GK;
    slices = std::max<int64_t>(1, cdiv(D, rps));
    FD_TRY(workspace(ctx, "gram_partial", sizeof(double) * slices * m * n, &p));
  }
  double* P = (double*)p;
  dim3 grid(tiles, (unsigned)slices);
  k_gram_partial<<<grid, 256, 0, ctx->stream>>>(X, ldx, Y, ldy, D, m, n, ntj, sym, rps, P);
  FD_LAUNCHED(ctx);
  k_gram_reduce<<<(unsigned)cdiv((int64_t)m * n, 256), 256, 0, ctx->stream>>>(P, (int)slices, m, n,
                                                                             sym, C, ldc);
  FD_LAUNCHED(ctx);
  return FD_OK;
}

fd_status gram_partials(fd_ctx* ctx, const double* X, int64_t ldx, const double* Y, int64_t ldy,
                        int64_t D, int m, int n, double* C, int ldc, bool sym, double* P,
                        int64_t max_slices) {
  const int nti = (int)cdiv(m, GT), ntj = (int)cdiv(n, GT);
  const int tiles = sym ? nti * (nti + 1) / 2 : nti * ntj;
  // about four CTAs per SM; short blocks are cut down to one shared-memory stage
  // (1,728 x 96 with its reduction: 51 us, 70 us with 64 rows per slice)
  int64_t slices = std::max<int64_t>(1, cdiv(4LL * ctx->num_sms, tiles));
  slices = std::min<int64_t>(slices, std::max<int64_t>(1, cdiv(D, GK)));
  slices = std::max<int64_t>(1, std::min<int64_t>(slices, max_slices));
  const int64_t rps = cdiv(cdiv(D, slices), GK) * GK;
  slices = std::max<int64_t>(1, cdiv(D, rps));
  dim3 grid(tiles, (unsigned)slices);
  k_gram_partial<<<grid, 256, 0, ctx->stream>>>(X, ldx, Y, ldy, D, m, n, ntj, sym, rps, P);
  FD_LAUNCHED(ctx);
  k_gram_reduce<<<(unsigned)cdiv((int64_t)m * n, 256), 256, 0, ctx->stream>>>(P, (int)slices, m, n,
                                                                             sym, C, ldc);
  FD_LAUNCHED(ctx);
  return FD_OK;
}

fd_status identity_dev(fd_ctx* ctx, double* A, int n) {
  k_identity<<<(unsigned)cdiv((int64_t)n * n, 256), 256, 0, ctx->stream>>>(A, n);
  FD_LAUNCHED(ctx);
  return FD_OK;
}

fd_status small_gemm_dev(fd_ctx* ctx, const double* A, const double* B, double* C, int n) {
  k_small_gemm<<<(unsigned)cdiv((int64_t)n * n, 256), 256, 0, ctx->stream>>>(A, B, C, n);
  FD_LAUNCHED(ctx);
  return FD_OK;
}

fd_status rotate(fd_ctx* ctx, double* V, int64_t ldv, int64_t D, int n, const double* M, bool upper) {
  if (use_ozaki(ctx, D, n, n)) {
    bool used = false;
    FD_TRY(oz_rotate(ctx, V, ldv, D, n, M, upper, &used));
    if (used) return FD_OK;
  }
  return rotate_fp64(ctx, V, ldv, D, n, M, upper);
}

template <int RT>
static fd_status launch_rotate(fd_ctx* ctx, double* V, int64_t ldv, int64_t D, int n, const double* M, bool upper) {
  const size_t smem = sizeof(double) * RT * n;
  auto kernel = upper ? k_rotate<RT, true> : k_rotate<RT, false>;
  if (smem > 48 * 1024)
    FD_CUDA(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ctx->smem_optin));
  kernel<<<(unsigned)cdiv(D, RT), 256, smem, ctx->stream>>>(V, ldv, D, n, M);
  FD_LAUNCHED(ctx);
  return FD_OK;
}

fd_status rotate_fp64(fd_ctx* ctx, double* V, int64_t ldv, int64_t D, int n, const double* M,
                      bool upper) {
  // one limit on the width for every number of rows
  if (sizeof(double) * 16 * n > ctx->smem_optin) return set_err(ctx, FD_ERR_ARG, "block too wide for rotation (%d)", n);
  // three CTAs per SM or more where the rows allow it
  if (D < 24LL * ctx->num_sms) return launch_rotate<4>(ctx, V, ldv, D, n, M, upper);
  if (D < 48LL * ctx->num_sms) return launch_rotate<8>(ctx, V, ldv, D, n, M, upper);
  return launch_rotate<16>(ctx, V, ldv, D, n, M, upper);
}

fd_status cholesky(fd_ctx* ctx, const double* G, int n, double coeff, double* R, int* ok_dev) {
  // two panels or more: one CTA per SM, co-resident (cooperative launch), no more
  // than there are rows to update
  const size_t smem = sizeof(double) * 2 * CB * n;
  if (n > CB && smem <= ctx->smem_optin) {
    if (smem > 32 * 1024)
      FD_CUDA(ctx, cudaFuncSetAttribute(k_cholesky_coop, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)(sizeof(double) * 2 * CB * 1024)));
    const int grid = std::min(ctx->num_sms, n);
    void* args[] = {(void*)&G, (void*)&n, (void*)&coeff, (void*)&R, (void*)&ok_dev};
    if (cudaLaunchCooperativeKernel((const void*)k_cholesky_coop, grid, 256, args, smem, ctx->stream) == cudaSuccess) {
      ctx->launches++;
      return FD_OK;
    }
    cudaGetLastError();  // cooperative launch unavailable: the one-CTA kernel below
  }
  k_cholesky<<<1, 1024, 0, ctx->stream>>>(G, n, coeff, R, ok_dev);
  FD_LAUNCHED(ctx);
  return FD_OK;
}

fd_status tri_inverse(fd_ctx* ctx, const double* R, int n, double* Rinv) {
  const size_t smem = sizeof(double) * CB * n;
  // the default limit of 48 KB covers the kernel's static arrays too (2.7 KB)
  if (smem > 32 * 1024)
    FD_CUDA(ctx, cudaFuncSetAttribute(k_tri_inverse, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)(sizeof(double) * CB * 1024)));
  k_tri_inverse<<<(unsigned)cdiv(n, CB), 256, smem, ctx->stream>>>(R, n, Rinv);
  FD_LAUNCHED(ctx);
  return FD_OK;
}

fd_status resid_norms(fd_ctx* ctx, const double* V, const double* AV, int64_t ld, int64_t D, int n,
                      const double* theta, double* out) {
  const int nb = std::min<int64_t>(ctx->num_sms * 4, std::max<int64_t>(1, D));
  void* p;
  FD_TRY(workspace(ctx, "resid_partial", sizeof(double) * nb * n, &p));
  k_resid_partial<<<nb, 256, 0, ctx->stream>>>(V, AV, ld, D, n, theta, (double*)p);
  FD_LAUNCHED(ctx);
  k_resid_reduce<<<(unsigned)cdiv(n, 8), 256, 0, ctx->stream>>>((double*)p, nb, n, out);
  FD_LAUNCHED(ctx);
  return FD_OK;
}

// The last Cholesky-QR pass factors the Gram matrix of a block the earlier
// passes have orthonormalised: its R is close to the identity.  A diagonal
// entry off by more than a factor 4 means they failed (a numerically rank
// deficient block beyond what the shifted passes recover): FD_ERR_BREAKDOWN
// instead of a block that is not orthonormal.  Synchronises.
fd_status check_last_factor(fd_ctx* ctx, const double* Rk, int ns) {
  std::vector<double> d(ns);
  FD_CUDA(ctx, cudaMemcpy2DAsync(d.data(), sizeof(double), Rk, sizeof(double) * (ns + 1), sizeof(double),
                                 ns, cudaMemcpyDeviceToHost, ctx->stream));
  FD_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  for (int i = 0; i < ns; ++i)
    if (!(std::fabs(d[i]) > 0.25 && std::fabs(d[i]) < 4.0))
      return set_err(ctx, FD_ERR_BREAKDOWN,
                     "Cholesky-QR: the block is numerically rank deficient (last-pass R[%d][%d] = %g)", i, i, d[i]);
  return FD_OK;
}

fd_status orthonormalize(fd_ctx* ctx, double* V, int64_t D, int ns, int64_t ldv, double* R,
                         int* passes_out) {
  void* p;
  const size_t nn = (size_t)ns * ns;
  FD_TRY(workspace(ctx, "ortho", sizeof(double) * 4 * nn + 64, &p));
  double* G = (double*)p;
  double* Rk = G + nn;
  double* Ri = Rk + nn;
  double* Rt = Ri + nn;
  int* ok = (int*)(Rt + nn);
  const double coeff = 11.0 * ((double)D * ns + (double)ns * (ns + 1)) * 0x1.0p-53;
  if (R) {
    k_identity<<<(unsigned)cdiv(nn, 256), 256, 0, ctx->stream>>>(R, ns);
    FD_LAUNCHED(ctx);
  }
  bool any_shift = false;
  int passes = 0;
  while (passes < 2 || (any_shift && passes < 3)) {
    FD_TRY(gram(ctx, V, ldv, V, ldv, D, ns, ns, G, ns, true));
    FD_TRY(cholesky(ctx, G, ns, 0.0, Rk, ok));
    int hok = 0;
    FD_CUDA(ctx, cudaMemcpyAsync(&hok, ok, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    FD_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    if (!hok) {
      FD_TRY(cholesky(ctx, G, ns, coeff, Rk, ok));
      FD_CUDA(ctx, cudaMemcpyAsync(&hok, ok, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
      FD_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
      if (!hok) return set_err(ctx, FD_ERR_BREAKDOWN, "shifted Cholesky-QR broke down (pass %d)", passes + 1);
      any_shift = true;
    }
    FD_TRY(tri_inverse(ctx, Rk, ns, Ri));
    FD_TRY(rotate(ctx, V, ldv, D, ns, Ri, true));
    if (R) {
      k_small_gemm<<<(unsigned)cdiv(nn, 256), 256, 0, ctx->stream>>>(Rk, R, Rt, ns);
      FD_LAUNCHED(ctx);
      FD_CUDA(ctx, cudaMemcpyAsync(R, Rt, sizeof(double) * nn, cudaMemcpyDeviceToDevice, ctx->stream));
    }
    ++passes;
  }
  FD_TRY(check_last_factor(ctx, Rk, ns));
  if (passes_out) *passes_out = passes;
  return FD_OK;
}

static int bundle_width(int remaining) {
  const int w[] = {128, 64, 32, 16, 8, 4, 2};
  for (int x : w)
    if (x <= remaining) return x;
  return 0;
}

fd_status rayleigh_ritz_dev(fd_ctx* ctx, const fd_matrix* A, double* V, double* AV, int64_t D,
                            int ns, int64_t ld, double* theta_dev, double* resid_dev) {
  for (int j = 0; j < ns;) {
    int w = bundle_width(ns - j);
    FD_TRY(spmmv(ctx, A, FD_F64, V + j, ld, AV + j, ld, w, true));
    j += w;
  }
  void* p;
  const size_t nn = (size_t)ns * ns;
  FD_TRY(workspace(ctx, "rr", sizeof(double) * 2 * nn, &p));
  double* H = (double*)p;
  double* Q = H + nn;
  FD_TRY(gram(ctx, V, ld, AV, ld, D, ns, ns, H, ns, true));
  FD_TRY(sym_eig(ctx, H, ns, theta_dev, Q, 40));
  FD_TRY(rotate(ctx, V, ld, D, ns, Q, false));
  // A (V Q) by a second SpMMV instead of rotating AV: on GB300 the rotation is
  // FP64-ALU bound (D ns^2 FMAs) while the SpMMV costs nnz ns FMAs
  for (int j = 0; j < ns;) {
    int w = bundle_width(ns - j);
    FD_TRY(spmmv(ctx, A, FD_F64, V + j, ld, AV + j, ld, w, true));
    j += w;
  }
  FD_TRY(resid_norms(ctx, V, AV, ld, D, ns, theta_dev, resid_dev));
  return FD_OK;
}

fd_status copy_cols_f64_to_f32(fd_ctx* ctx, const double* src, int64_t lds, float* dst, int64_t ldd,
                               int64_t D, int n) {
  return convert_block(ctx, src, lds, dst, ldd, D, n);
}
fd_status copy_cols_f32_to_f64(fd_ctx* ctx, const float* src, int64_t lds, double* dst, int64_t ldd,
                               int64_t D, int n) {
  return convert_block(ctx, src, lds, dst, ldd, D, n);
}
fd_status copy_cols_f64_to_ff(fd_ctx* ctx, const double* src, int64_t lds, float* dst, int64_t ldd,
                              int64_t D, int n) {
  if ((uintptr_t)dst & 7) return convert_each(ctx, src, lds, reinterpret_cast<pair_u*>(dst), ldd, D, n);
  return convert_each(ctx, src, lds, reinterpret_cast<pair_f*>(dst), ldd, D, n);
}
fd_status copy_cols_ff_to_f64(fd_ctx* ctx, const float* src, int64_t lds, double* dst, int64_t ldd,
                              int64_t D, int n) {
  if ((uintptr_t)src & 7) return convert_each(ctx, reinterpret_cast<const pair_u*>(src), lds, dst, ldd, D, n);
  return convert_each(ctx, reinterpret_cast<const pair_f*>(src), lds, dst, ldd, D, n);
}

}  // namespace fdi

using namespace fdi;

extern "C" {

fd_status fd_orthonormalize(fd_ctx* ctx, double* V, int64_t D, int ns, int64_t ldv, double* R,
                            int* passes) {
  if (!ctx) return FD_ERR_ARG;
  ctx->err.clear();
  if (!V || D < 1 || ns < 1 || ns > 1024 || ldv < ns || ns > D)
    return set_err(ctx, FD_ERR_ARG, "need V, 1 <= ns <= min(1024, D), ldv >= ns");
  FD_CUDA(ctx, cudaSetDevice(ctx->device));
  return orthonormalize(ctx, V, D, ns, ldv, R, passes);
}

fd_status fd_gram(fd_ctx* ctx, const double* X, int64_t ldx, const double* Y, int64_t ldy, int64_t D,
                   int m, int n, double* C, int ldc) {
  if (!ctx) return FD_ERR_ARG;
  ctx->err.clear();
  if (!X || !Y || !C || D < 1 || m < 1 || n < 1 || m > 4096 || n > 4096 || ldx < m || ldy < n || ldc < n)
    return set_err(ctx, FD_ERR_ARG, "need blocks, D >= 1, 1 <= m, n <= 4096, ld >= width");
  FD_CUDA(ctx, cudaSetDevice(ctx->device));
  return gram(ctx, X, ldx, Y, ldy, D, m, n, C, ldc, X == Y && ldx == ldy && m == n);
}

fd_status fd_rotate(fd_ctx* ctx, double* V, int64_t ldv, int64_t D, int n, const double* M, int upper) {
  if (!ctx) return FD_ERR_ARG;
  ctx->err.clear();
  if (!V || !M || D < 1 || n < 1 || n > 1024 || ldv < n)
    return set_err(ctx, FD_ERR_ARG, "need blocks, D >= 1, 1 <= n <= 1024, ldv >= n");
  FD_CUDA(ctx, cudaSetDevice(ctx->device));
  return rotate(ctx, V, ldv, D, n, M, upper != 0);
}

fd_status fd_set_gemm_mode(fd_ctx* ctx, fd_gemm_mode mode) {
  if (!ctx) return FD_ERR_ARG;
  if (mode != FD_GEMM_AUTO && mode != FD_GEMM_FP64 && mode != FD_GEMM_OZAKI)
    return set_err(ctx, FD_ERR_ARG, "unknown gemm mode %d", (int)mode);
  ctx->gemm_mode = (int)mode;
  return FD_OK;
}

fd_status fd_copy_block(fd_ctx* ctx, const void* src, fd_prec sp, int64_t lds, void* dst, fd_prec dp,
                        int64_t ldd, int64_t D, int n) {
  if (!ctx) return FD_ERR_ARG;
  ctx->err.clear();
  auto known = [](fd_prec p) { return p == FD_F64 || p == FD_F32 || p == FD_FF; };
  if (!src || !dst || D < 0 || n < 0 || lds < n || ldd < n || !known(sp) || !known(dp) ||
      (sp == FD_F32 && dp == FD_FF) || (sp == FD_FF && dp == FD_F32))
    return set_err(ctx, FD_ERR_ARG, "need buffers, D, n >= 0, lds, ldd >= n and a supported type pair");
  if (D == 0 || n == 0) return FD_OK;
  FD_CUDA(ctx, cudaSetDevice(ctx->device));
  if (sp == FD_F64 && dp == FD_F32)
    return copy_cols_f64_to_f32(ctx, (const double*)src, lds, (float*)dst, ldd, D, n);
  if (sp == FD_F32 && dp == FD_F64)
    return copy_cols_f32_to_f64(ctx, (const float*)src, lds, (double*)dst, ldd, D, n);
  if (sp == FD_F64 && dp == FD_FF)
    return copy_cols_f64_to_ff(ctx, (const double*)src, lds, (float*)dst, ldd, D, n);
  if (sp == FD_FF && dp == FD_F64)
    return copy_cols_ff_to_f64(ctx, (const float*)src, lds, (double*)dst, ldd, D, n);
  if (sp == FD_F32) return convert_block(ctx, (const float*)src, lds, (float*)dst, ldd, D, n);
  // a float-float block may start at any float, between the 8-byte boundaries too
  if (((uintptr_t)src | (uintptr_t)dst) & 7)
    return convert_each(ctx, (const pair_u*)src, lds, (pair_u*)dst, ldd, D, n);
  return convert_block(ctx, (const double*)src, lds, (double*)dst, ldd, D, n);  // float-float pairs: 8 bytes too
}

fd_status fd_rayleigh_ritz(fd_ctx* ctx, const fd_matrix* A, double* V, double* AV, int64_t D, int ns,
                           int64_t ld, double* theta, double* resid) {
  if (!ctx) return FD_ERR_ARG;
  ctx->err.clear();
  if (!A || !V || !AV || !theta || !resid) return set_err(ctx, FD_ERR_ARG, "null argument");
  if (D != A->D || ns < 2 || ns % 2 || ns > 1024 || ns > D || ld < ns || ld % 2 ||
      ((uintptr_t)V & 15) || ((uintptr_t)AV & 15))
    return set_err(ctx, FD_ERR_ARG, "need D = matrix dimension, even 2 <= ns <= 1024, even ld >= ns, aligned blocks");
  FD_CUDA(ctx, cudaSetDevice(ctx->device));
  void* p;
  FD_TRY(workspace(ctx, "rr_out", sizeof(double) * 2 * ns, &p));
  double* th = (double*)p;
  FD_TRY(rayleigh_ritz_dev(ctx, A, V, AV, D, ns, ld, th, th + ns));
  FD_CUDA(ctx, cudaMemcpyAsync(theta, th, sizeof(double) * ns, cudaMemcpyDeviceToHost, ctx->stream));
  FD_CUDA(ctx, cudaMemcpyAsync(resid, th + ns, sizeof(double) * ns, cudaMemcpyDeviceToHost, ctx->stream));
  FD_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  return FD_OK;
}

}  // extern "C"
