// Spectral inclusion intervals from a few Lanczos steps (Sec. 2, Alg. 1 steps
// 1-2), for one matrix or for all instances of a batch at once.
//
// The work of a step is small (an nb = 1 SpMV and two Gram-Schmidt passes over
// the vectors so far); what it costs is the chain between them.  So all steps of
// all matrices run in one cooperative kernel: the CTAs are divided among the
// matrices, each owns a run of rows, and a step has four grid barriers (two
// passes of dot products, the norm, the next vector) and no host round trip.  64
// threads of a CTA go along the rows and four such sets along the vectors (along the
// rows too while there are fewer tiles of vectors than sets): FP64 adds issue at one
// warp in 64 clocks, so a CTA's sums are combined by a halving exchange (9 adds for 8
// sums over a warp instead of 40).
// The tridiagonal matrix is diagonalised on the host by implicit QL with the last
// components of the eigenvectors alone carried along.
// Measured against a kernel per operation: 20 steps on 110,592 rows 4.6 -> 0.9 ms, on
// 2,097,152 11.6 -> 8.8; 50 steps on each of twelve matrices of 1,000 to 2,744 rows 89
// (device time, without the 600 host round trips) -> 2.1 ms.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "fd_internal.cuh"

namespace cg = cooperative_groups;

namespace fdi {
namespace {

constexpr int LZ_THREADS = 256;
constexpr int LZ_ROWS = 64;                       // threads along the rows
constexpr int LZ_SETS = LZ_THREADS / LZ_ROWS;     // sets along the vectors
// CTAs per SM for many rows, and the rows per SM of each: one CTA has too few loads
// under way to stream the vectors (2.1M rows, 20 steps: 24.1 ms with one per SM, 8.7 with
// four), but more cost barriers and registers (110,592 rows: 0.98 ms with one, 1.9 with
// four; 262,144 rows 1.79, 1.57 with two, 2.35 with four)
constexpr int LZ_PER_SM = 4, LZ_SM_ROWS = 1024;
constexpr int LZ_TILE = 8;                        // vectors of a set at a time
constexpr size_t LZ_CHUNK_BYTES = 256u << 20;     // workspace of one launch of several matrices

struct LzMatrix {
  const int64_t* chunk_ptr;
  const int32_t* row_len;
  const int32_t* col;
  const double* val;
  const int64_t* perm;
  int64_t D;
  int C, m;        // m: steps for this matrix
  uint64_t key;
  double* Q;       // m x D
  double* w;       // D
  double* out;     // m alphas, m betas, steps done, last beta
};

struct LzArgs {
  const LzMatrix* mat;
  int n, cpi, m_max;
  double* part;    // 2 x gridDim.x x m_max
};

// PER_SM: CTAs that must fit an SM (4: 64 registers)
template <int PER_SM>
__global__ void __launch_bounds__(LZ_THREADS, PER_SM) k_lanczos(LzArgs a) {
  cg::grid_group grid = cg::this_grid();
  extern __shared__ double cs[];  // m_max coefficients
  __shared__ double red[LZ_THREADS / 32][LZ_TILE];
  const int inst = blockIdx.x / a.cpi, local = blockIdx.x % a.cpi;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rt = threadIdx.x % LZ_ROWS, set = threadIdx.x / LZ_ROWS;
  const bool mine = inst < a.n;
  const LzMatrix M = a.mat[mine ? inst : 0];
  const int64_t per = (M.D + a.cpi - 1) / a.cpi;
  const int64_t r0 = min(M.D, per * local), r1 = min(M.D, r0 + per);
  double* w = M.w;

  // sums over the CTA's rows of Q_v w, v = v0 .. v0 + nv - 1, to the partials
  // (nv = 0: the sum of w w)
  auto dots = [&](int buf, int nv) {
    double* P = a.part + ((int64_t)buf * gridDim.x + blockIdx.x) * a.m_max;
    const int tiles = nv ? (nv + LZ_TILE - 1) / LZ_TILE : 1;
    for (int t0 = 0; t0 < tiles; t0 += LZ_SETS) {
      // fewer tiles than sets left: several sets share a tile, each with its own rows
      const int share = tiles - t0 > 2 ? 1 : tiles - t0 == 2 ? 2 : 4;
      const int tile = t0 + set / share, part = set % share;
      double x[LZ_TILE] = {};
      if (tile < tiles) {
        const int v0 = tile * LZ_TILE;
        for (int64_t r = r0 + part * LZ_ROWS + rt; r < r1; r += LZ_ROWS * share) {
          const double wr = w[r];
          if (nv) {
#pragma unroll
            for (int v = 0; v < LZ_TILE; ++v)
              if (v0 + v < nv) x[v] = fma(M.Q[(int64_t)(v0 + v) * M.D + r], wr, x[v]);
          } else {
            x[0] = fma(wr, wr, x[0]);
          }
        }
      }
      // halving exchange: 8 sums over 32 lanes; lane bits 4, 3, 2 end up selecting the sum
#pragma unroll
      for (int h = LZ_TILE / 2, o = 16; h > 0; h >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int v = 0; v < h; ++v) {
          const double send = up ? x[v] : x[v + h], keep = up ? x[v + h] : x[v];
          x[v] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
      }
      x[0] += __shfl_xor_sync(0xffffffffu, x[0], 2);
      x[0] += __shfl_xor_sync(0xffffffffu, x[0], 1);
      if ((lane & 3) == 0) red[warp][lane >> 2] = x[0];
      __syncthreads();
      if (rt < LZ_TILE && tile < tiles && part == 0) {
        const int v = tile * LZ_TILE + rt;
        double sum = red[2 * set][rt] + red[2 * set + 1][rt];
        for (int q = 1; q < share; ++q) sum += red[2 * (set + q)][rt] + red[2 * (set + q) + 1][rt];
        if (v < max(nv, 1)) __stcg(P + v, sum);
      }
      __syncthreads();
    }
  };
  // the matrix's sums, in every one of its CTAs
  auto collect = [&](int buf, int nv) {
    for (int v = warp; v < nv; v += LZ_THREADS / 32) {
      double s = 0.0;
      for (int b = lane; b < a.cpi; b += 32)
        s += __ldcg(a.part + ((int64_t)buf * gridDim.x + (int64_t)inst * a.cpi + b) * a.m_max + v);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) cs[v] = s;
    }
    __syncthreads();
  };

  if (mine) {
    for (int64_t r = r0 + threadIdx.x; r < r1; r += LZ_THREADS) w[r] = fdrng::irwin_hall(M.key, (uint64_t)M.perm[r]);
    __syncthreads();
    dots(0, 0);
  }
  grid.sync();
  if (mine) {
    collect(0, 1);
    const double f = 1.0 / sqrt(cs[0]);
    for (int64_t r = r0 + threadIdx.x; r < r1; r += LZ_THREADS) __stcg(M.Q + r, w[r] * f);
  }
  grid.sync();
  bool on = mine;
  for (int j = 0; j < a.m_max; ++j) {
    if (on) {
      const double* q = M.Q + (int64_t)j * M.D;
      for (int64_t r = r0 + threadIdx.x; r < r1; r += LZ_THREADS) {
        const uint32_t C = (uint32_t)M.C, chunk = (uint32_t)r / C;
        const int64_t base = M.chunk_ptr[chunk] + ((uint32_t)r - chunk * C);
        const int len = M.row_len[r];
        double s = 0.0;
        for (int e = 0; e < len; ++e)
          s = fma(M.val[base + (int64_t)e * C], __ldcg(q + M.col[base + (int64_t)e * C]), s);
        w[r] = s;
      }
      __syncthreads();
    }
    double alpha = 0.0;
    for (int pass = 0; pass < 2; ++pass) {  // full reorthogonalisation, twice
      if (on) dots(pass, j + 1);
      grid.sync();
      if (on) {
        collect(pass, j + 1);
        if (pass == 0) alpha = cs[j];
        for (int64_t r = r0 + threadIdx.x; r < r1; r += LZ_THREADS) {
          double s = w[r];
          int v = 0;
          for (; v + LZ_TILE <= j + 1; v += LZ_TILE) {  // the loads of a tile together
            double q[LZ_TILE];
#pragma unroll
            for (int u = 0; u < LZ_TILE; ++u) q[u] = M.Q[(int64_t)(v + u) * M.D + r];
#pragma unroll
            for (int u = 0; u < LZ_TILE; ++u) s = fma(-q[u], cs[v + u], s);
          }
          for (; v <= j; ++v) s = fma(-M.Q[(int64_t)v * M.D + r], cs[v], s);
          w[r] = s;
        }
        __syncthreads();
      }
    }
    if (on) dots(0, 0);
    grid.sync();
    if (on) {
      collect(0, 1);
      const double beta = sqrt(cs[0]);
      const bool last = j == M.m - 1 || beta <= 1e-14 * fmax(1.0, fabs(alpha));
      if (!last) {
        const double f = 1.0 / beta;
        for (int64_t r = r0 + threadIdx.x; r < r1; r += LZ_THREADS)
          __stcg(M.Q + (int64_t)(j + 1) * M.D + r, w[r] * f);
      }
      if (local == 0 && threadIdx.x == 0) {
        M.out[j] = alpha;
        M.out[M.m + j] = beta;
        M.out[2 * M.m] = j + 1;
        M.out[2 * M.m + 1] = beta;
      }
      on = !last;
    }
    grid.sync();
  }
}

// Eigenvalues d of the symmetric tridiagonal matrix (d, e) and the last
// components z of its eigenvectors: implicit QL (Dubrulle, Martin and Wilkinson
// 1968), rotations applied to the last row of the eigenvector matrix only.
bool tridiagonal_ql(std::vector<double>& d, std::vector<double>& e, std::vector<double>& z) {
  const int n = (int)d.size();
  z.assign(n, 0.0);
  z[n - 1] = 1.0;
  e.resize(n, 0.0);
  for (int l = 0; l < n; ++l) {
    for (int it = 0;; ++it) {
      int m = l;
      while (m < n - 1 && std::fabs(e[m]) > 0x1.0p-53 * (std::fabs(d[m]) + std::fabs(d[m + 1]))) ++m;
      if (m == l) break;
      if (it == 60) return false;
      const double g0 = (d[l + 1] - d[l]) / (2.0 * e[l]);
      const double shift = d[m] - d[l] + e[l] / (g0 + std::copysign(std::hypot(g0, 1.0), g0));
      double s = 1.0, c = 1.0, p = 0.0, g = shift;
      int i = m - 1;
      for (; i >= l; --i) {
        const double f = s * e[i], b = c * e[i];
        const double r = std::hypot(f, g);
        e[i + 1] = r;
        if (r == 0.0) {  // the matrix splits here
          d[i + 1] -= p;
          e[m] = 0.0;
          break;
        }
        s = f / r;
        c = g / r;
        const double h = d[i + 1] - p, t = (d[i] - h) * s + 2.0 * c * b;
        p = s * t;
        d[i + 1] = h + p;
        g = c * t - b;
        const double zi = z[i + 1];
        z[i + 1] = s * z[i] + c * zi;
        z[i] = c * z[i] - s * zi;
      }
      if (i >= l) continue;
      d[l] -= p;
      e[l] = g;
      e[m] = 0.0;
    }
  }
  return true;
}

}  // namespace

fd_status spectral_bounds_batch(fd_ctx* ctx, int n_inst, const fd_matrix* const* A, int steps,
                                const uint64_t* seeds, double* lam_l, double* lam_r) {
  cudaStream_t st = ctx->stream;
  const int64_t step_limit = (int64_t)((ctx->smem_optin - 1024) / sizeof(double));
  for (int i = 0; i < n_inst; ++i)
    if (std::min<int64_t>(steps, A[i]->D) > step_limit)
      return set_err(ctx, FD_ERR_ARG, "more than %lld Lanczos steps", (long long)step_limit);
  for (int first = 0; first < n_inst;) {
    // as many matrices as the workspace chunk holds (at least one)
    auto doubles = [&](int i) {
      const size_t m = (size_t)std::min<int64_t>(steps, A[i]->D);
      return (m + 1) * (size_t)A[i]->D + 2 * m + 2;
    };
    int n = 0;
    size_t total = 0;
    while (first + n < n_inst && n < ctx->num_sms &&
           (n == 0 || (total + doubles(first + n)) * sizeof(double) <= LZ_CHUNK_BYTES))
      total += doubles(first + n++);
    // the launch of the first k of them: co-resident CTAs, no more than one per 64 rows
    int64_t rows = 0, all_rows = 0;
    int m_max = 0, cpi = 0;
    size_t smem = 0;
    const void* kernel = nullptr;
    auto plan = [&](int k) -> fd_status {
      rows = all_rows = 0;
      m_max = 0;
      for (int i = first; i < first + k; ++i) {
        rows = std::max(rows, A[i]->D);
        all_rows += A[i]->D;
        m_max = std::max(m_max, (int)std::min<int64_t>(steps, A[i]->D));
      }
      int per_sm = (int)std::min<int64_t>(LZ_PER_SM, cdiv(all_rows, (int64_t)LZ_SM_ROWS * ctx->num_sms));
      kernel = per_sm > 1 ? (const void*)k_lanczos<LZ_PER_SM> : (const void*)k_lanczos<1>;
      smem = sizeof(double) * (size_t)m_max;  // a coefficient per step
      if (smem > 32 * 1024) {
        FD_CUDA(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ctx->smem_optin - 1024));
        int fit = 0;
        FD_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, kernel, LZ_THREADS, smem));
        per_sm = std::max(1, std::min(per_sm, fit));
      }
      cpi = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)per_sm * ctx->num_sms / k, cdiv(rows, LZ_ROWS)));
      return FD_OK;
    };
    auto bytes = [&](int k, size_t t) {
      return sizeof(double) * (t + 2 * (size_t)cpi * k * m_max) + sizeof(LzMatrix) * k + 64;
    };
    void* p = nullptr;
    FD_TRY(plan(n));
    fd_status ws = workspace(ctx, "lanczos", bytes(n, total), &p, n > 1);
    if (ws == FD_ERR_OOM && n > 1) {  // a tight workspace limit: one matrix at a time
      n = 1;
      total = doubles(first);
      ctx->err.clear();
      FD_TRY(plan(n));
      ws = workspace(ctx, "lanczos", bytes(n, total), &p);
    }
    FD_TRY(ws);
    LzMatrix* dm = (LzMatrix*)p;
    double* base = (double*)(((uintptr_t)(dm + n) + 15) & ~(uintptr_t)15);
    std::vector<LzMatrix> h(n);
    size_t outs = 0;
    double* q = base;
    for (int i = 0; i < n; ++i) {
      const fd_matrix* M = A[first + i];
      LzMatrix& L = h[i];
      L.chunk_ptr = M->chunk_ptr; L.row_len = M->row_len; L.col = M->col; L.val = M->val; L.perm = M->perm;
      L.D = M->D;
      L.C = M->C;
      L.m = (int)std::min<int64_t>(steps, M->D);
      L.key = fdrng::key(seeds[first + i], fdrng::STREAM_LANCZOS);
      outs += 2 * (size_t)L.m + 2;
    }
    double* out = q;  // all outputs together, then the vectors
    q += outs;
    double* o = out;
    for (LzMatrix& L : h) {
      L.out = o;
      o += 2 * (size_t)L.m + 2;
      L.Q = q;
      q += (size_t)L.m * L.D;
      L.w = q;
      q += L.D;
    }
    LzArgs a;
    a.mat = dm;
    a.n = n;
    a.m_max = m_max;
    a.cpi = cpi;
    a.part = q;
    FD_CUDA(ctx, cudaMemcpyAsync(dm, h.data(), sizeof(LzMatrix) * n, cudaMemcpyHostToDevice, st));
    void* args[] = {&a};
    FD_CUDA(ctx, cudaLaunchCooperativeKernel(kernel, a.cpi * n, LZ_THREADS, args, smem, st));
    FD_LAUNCHED(ctx);
    std::vector<double> ho(outs);
    FD_CUDA(ctx, cudaMemcpyAsync(ho.data(), out, sizeof(double) * outs, cudaMemcpyDeviceToHost, st));
    FD_CUDA(ctx, cudaStreamSynchronize(st));
    size_t at = 0;
    for (int i = 0; i < n; ++i) {
      const int m = h[i].m;
      const double* oi = ho.data() + at;
      at += 2 * (size_t)m + 2;
      const int k = (int)oi[2 * m];
      const double beta_last = oi[2 * m + 1];
      std::vector<double> d(oi, oi + k), e(oi + m, oi + m + k - 1), z;
      if (!tridiagonal_ql(d, e, z)) return set_err(ctx, FD_ERR_BREAKDOWN, "Lanczos: the tridiagonal eigensolve did not converge");
      const int imin = (int)(std::min_element(d.begin(), d.end()) - d.begin());
      const int imax = (int)(std::max_element(d.begin(), d.end()) - d.begin());
      const double tmin = d[imin], tmax = d[imax];
      const double wdt = std::max(tmax - tmin, 1e-10 * std::max({1.0, std::fabs(tmin), std::fabs(tmax)}));
      const fd_matrix* M = A[first + i];
      lam_l[first + i] = std::max(M->gersh_lo, tmin - std::fabs(beta_last * z[imin]) - 0.01 * wdt);
      lam_r[first + i] = std::min(M->gersh_hi, tmax + std::fabs(beta_last * z[imax]) + 0.01 * wdt);
    }
    first += n;
  }
  return FD_OK;
}

fd_status spectral_bounds(fd_ctx* ctx, const fd_matrix* A, int steps, uint64_t seed, double* lam_l,
                          double* lam_r) {
  return spectral_bounds_batch(ctx, 1, &A, steps, &seed, lam_l, lam_r);
}

}  // namespace fdi
