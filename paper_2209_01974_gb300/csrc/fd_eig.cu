// Symmetric eigensolver of the Rayleigh-Ritz step (Sec. 2): two-sided cyclic
// Jacobi in 8-wide blocks over a cooperative grid, for one matrix or for all
// instances of a batch at once.
//
// What bounds it on GB300 is not arithmetic (6 n^3 FP64 operations a sweep, 25 us
// of the chip for n = 128) but the chain of rounds: a rotation set needs the
// result of the one before it.  Elementwise rounds pay a grid barrier, two L2 round
// trips and the slow FP64 division and square roots of the angles n - 1 times a
// sweep (7 us a round).  Here a round pairs blocks instead of columns:
//   phase 1  one CTA per pair of blocks loads its 16 x 16 principal submatrix,
//            rotates the 64 pairs across the two blocks in 8
//            inner rounds in shared memory (in the first round of a sweep all 120
//            pairs in 15), and leaves the product J of the rotations;
//   phase 2  A <- J^T A J block by block (upper half, mirrored) and Q <- Q J as
//            small products spread over all SMs.
// So a sweep has n / 8 - 1 rounds of two barriers.  Eight is where the inner
// rounds (1 us each, on one SM's two FP64 FMA a clock) and the barriers balance.
//
// Angles need no FP64: any rotation close to the annihilating one converges as
// fast once the rest is computed rather than set to zero.  tan(phi) is found in
// FP32 from the FP64 difference of the diagonal entries, (c, s) as floats, and
// both are then scaled in FP64 by 1 / sqrt(c^2 + s^2) through its series at 1 (the
// sum is within 2e-7 of 1, the third term below 1e-20), which makes the rotation
// orthogonal to FP64 rounding.
// Measured (device time, Rayleigh quotients, elementwise cyclic Jacobi -> this):
// n = 128 7.06 -> 2.1 ms, n = 96 4.14 -> 1.6 ms, n = 32 0.38 ms; twelve instances
// of n = 64 in a batch 6.17 (one CTA each) -> 1.3 ms.  Of the 14 us of a round
// (n = 128) the eight inner rounds take 7, phase 2 and its loads 3, the barriers 3.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>

#include "fd_internal.cuh"
#include "fd_eig.cuh"

namespace cg = cooperative_groups;

namespace fdi {
namespace {

constexpr int B = EIG_BLOCK;      // block width
constexpr int BB = 2 * B;         // pair width
constexpr int GROUP = 128;        // threads of a task group
constexpr int GROUPS = 2;         // groups per CTA
constexpr int EIG_THREADS = GROUP * GROUPS;
static_assert(EIG_THREADS == BB * BB && GROUPS == 2, "phase 1 gives each thread one element");

struct EigArgs {
  EigTask one;           // n_inst = 1 and many = nullptr: this matrix
  const EigTask* many;
  int n_inst, m_max;     // matrices, most blocks of one of them
  int max_sweeps;
  float tol2;            // off-diagonal / whole squared norm
  float* part;           // gridDim.x x n_inst x 2
};

__device__ __forceinline__ const EigTask& task(const EigArgs& a, int i) { return a.many ? a.many[i] : a.one; }

__device__ __forceinline__ bool live(const EigTask& t) {
  return (!t.active || *t.active) && !(t.flags && (*t.flags & t.flag_mask));
}

// round-robin pairing of m (even) players: pair k of round r
__device__ __forceinline__ void pair_of(int r, int k, int m, int* p, int* q) {
  int a, b;
  if (k == 0) {
    a = r;
    b = m - 1;
  } else {
    a = r + k;
    if (a >= m - 1) a -= m - 1;
    b = r - k;
    if (b < 0) b += m - 1;
  }
  *p = min(a, b);
  *q = max(a, b);
}

__device__ __forceinline__ void group_sync(int g) {
  asm volatile("bar.sync %0, %1;\n" ::"r"(g + 1), "n"(GROUP) : "memory");
}

__device__ __forceinline__ float approx_rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;\n" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float approx_rsqrt(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;\n" : "=f"(r) : "f"(x));
  return r;
}

// rotation that (nearly) annihilates a_pq: (c, s) orthogonal to FP64 rounding
__device__ __forceinline__ void angle(double app, double aqq, double apq, double* c, double* s) {
  const float d = (float)(aqq - app), o = 2.0f * (float)apq;
  // entries are scaled to |a| <= 1 and stay below the order n (not finite: NaN
  // input); what is below 1e-30 is far under the convergence threshold, and its
  // reciprocal below would overflow for equal diagonal entries
  if (!(fabsf(o) > 1e-30f && fabsf(o) < 1e30f) || !(fabsf(d) < 1e30f)) {
    *c = 1.0;
    *s = 0.0;
    return;
  }
  // t = tan(phi) = sgn(d o) |o| / (|d| + sqrt(d^2 + o^2)); scaled against underflow of the squares
  const float rb = approx_rcp(fmaxf(fabsf(d), fabsf(o)));
  const float dd = fabsf(d) * rb, oo = o * rb, h = fmaf(dd, dd, oo * oo);  // h in [1, 2]
  float t = oo * approx_rcp(fmaf(h, approx_rsqrt(h), dd));
  if (d < 0.0f) t = -t;
  const float cf = approx_rsqrt(fmaf(t, t, 1.0f)), sf = t * cf;
  const double c0 = (double)cf, s0 = (double)sf;
  const double e = fma(s0, s0, fma(c0, c0, -1.0));           // exact to 1e-16
  const double f = fma(e, fma(e, 0.375, -0.5), 1.0);          // (1 + e)^(-1/2)
  *c = c0 * f;
  *s = s0 * f;
}

__device__ __forceinline__ unsigned long long order_key(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  return (b >> 63) ? ~b : b | (1ull << 63);
}

__global__ void __launch_bounds__(EIG_THREADS) k_block_jacobi(EigArgs a) {
  cg::grid_group grid = cg::this_grid();
  __shared__ double sA[GROUPS][2][BB][BB + 1], sJ[GROUPS][BB][BB + 1], sCS[GROUPS][BB];
  extern __shared__ unsigned char dyn[];
  // per matrix: whether it has converged, and which of A0 / A1 is current (the
  // same in every CTA)
  unsigned char* done = dyn;
  unsigned char* cur = dyn + a.n_inst;
  unsigned char* last = cur + a.n_inst;  // whether the sweep at hand is its last
  const int g = threadIdx.x / GROUP, t = threadIdx.x % GROUP;
  // a group's first task: all CTAs get one before any gets a second (the FP64
  // pipes of an SM are shared by its groups)
  const int spread = blockIdx.x + g * gridDim.x, ngroups = gridDim.x * GROUPS;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t gt = (int64_t)blockIdx.x * EIG_THREADS + threadIdx.x, gn = (int64_t)gridDim.x * EIG_THREADS;
  for (int i = threadIdx.x; i < a.n_inst; i += EIG_THREADS) {
    done[i] = !live(task(a, i));
    cur[i] = last[i] = 0;
  }
  __syncthreads();

  // partial sums of a CTA to a.part, or all CTAs' partials summed (maxima: the
  // FP32 value of |a|, rounded up by the scaling's slack) into every CTA
  auto reduce = [&](int i, float x, float y, bool is_max) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float x2 = __shfl_xor_sync(0xffffffffu, x, o), y2 = __shfl_xor_sync(0xffffffffu, y, o);
      x = is_max ? fmaxf(x, x2) : x + x2;
      y += y2;
    }
    __shared__ float red[2][EIG_THREADS / 32];
    __syncthreads();
    if (lane == 0) {
      red[0][warp] = x;
      red[1][warp] = y;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < EIG_THREADS / 32; ++w) {
        x = is_max ? fmaxf(x, red[0][w]) : x + red[0][w];
        y += red[1][w];
      }
      __stcg(a.part + ((int64_t)blockIdx.x * a.n_inst + i) * 2, x);
      __stcg(a.part + ((int64_t)blockIdx.x * a.n_inst + i) * 2 + 1, y);
    }
  };
  auto gather = [&](int i, bool is_max, float* x, float* y) {  // one warp
    float sx = 0.0f, sy = 0.0f;
    for (int b = lane; b < (int)gridDim.x; b += 32) {
      const float px = __ldcg(a.part + ((int64_t)b * a.n_inst + i) * 2);
      sx = is_max ? fmaxf(sx, px) : sx + px;
      sy += __ldcg(a.part + ((int64_t)b * a.n_inst + i) * 2 + 1);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float x2 = __shfl_xor_sync(0xffffffffu, sx, o);
      sx = is_max ? fmaxf(sx, x2) : sx + x2;
      sy += __shfl_xor_sync(0xffffffffu, sy, o);
    }
    *x = sx;
    *y = sy;
  };

  // exponent of the largest entry: A is scaled by a power of two to |a| <= 1, so
  // the FP32 steps neither overflow nor lose entries that matter.  The exponent
  // field of an entry (0 .. 2046) travels as a float; 2047 marks inf or NaN.
  for (int i = 0; i < a.n_inst; ++i) {
    if (done[i]) continue;
    const EigTask& T = task(a, i);
    float e = 0.0f;
    for (int64_t q = gt; q < (int64_t)T.n * T.n; q += gn)
      e = fmaxf(e, (float)((__double_as_longlong(T.H[q]) >> 52) & 0x7FF));
    reduce(i, e, 0.0f, true);
  }
  grid.sync();
  __shared__ float sc[2];
  for (int i = 0; i < a.n_inst; ++i) {
    if (done[i]) continue;
    const EigTask& T = task(a, i);
    if (warp == 0) {
      float e, unused;
      gather(i, true, &e, &unused);
      if (lane == 0) sc[0] = e;
    }
    __syncthreads();
    const int e = (int)sc[0];
    __syncthreads();
    const int shift = e == 0x7FF ? 0 : 1022 - max(e, 1);  // |a| < 2^(e - 1022)
    for (int64_t q = gt; q < (int64_t)T.np * T.np; q += gn) {
      const int r = (int)(q / T.np), c = (int)(q % T.np);
      double v = 0.0;
      if (r < T.n && c < T.n) v = scalbn(T.H[(int64_t)r * T.n + c], shift);
      __stcg(T.A0 + q, v);
      __stcg(T.Q + q, r == c ? 1.0 : 0.0);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *T.shift = e == 0x7FF ? INT_MIN : shift;
  }
  grid.sync();

  for (int sweep = 0; sweep < a.max_sweeps; ++sweep) {
    for (int i = 0; i < a.n_inst; ++i) {
      if (done[i]) continue;
      const EigTask& T = task(a, i);
      const double* A = cur[i] ? T.A1 : T.A0;
      float off = 0.0f, all = 0.0f;
      for (int64_t q = gt; q < (int64_t)T.np * T.np; q += gn) {
        const float v = (float)__ldcg(A + q);
        all = fmaf(v, v, all);
        if (q / T.np != q % T.np) off = fmaf(v, v, off);
      }
      reduce(i, off, all, false);
    }
    grid.sync();
    int left = 0;
    for (int i = warp; i < a.n_inst; i += EIG_THREADS / 32) {
      if (done[i]) continue;
      float off, all;
      gather(i, false, &off, &all);
      // A rotation leaves 1e-7 of its entry, so what is left below the threshold may be
      // far above the rounding: it gets one sweep more, which the eigenvectors of close
      // pairs need.
      const bool below = off <= a.tol2 * all, rounding = off <= 5e-32f * (float)task(a, i).n * all;
      if (last[i] || rounding || !(all <= 3e38f)) {
        if (lane == 0) done[i] = 1;
      } else {
        if (below && lane == 0) last[i] = 1;
        left = 1;
      }
      __syncwarp();
    }
    if (!__syncthreads_or(left)) break;
    for (int r = 0; r < a.m_max - 1; ++r) {
      // phase 1: rotations of every pair of blocks, one pair per CTA.  The first group
      // finds the angles and rotates A; the second accumulates J from the angles of
      // the inner round while the first is at the next one's.
      const int half_max = a.m_max / 2;
      for (int w = blockIdx.x; w < half_max * a.n_inst; w += gridDim.x) {
        const int i = w % a.n_inst, k = w / a.n_inst;
        if (done[i]) continue;
        const EigTask& T = task(a, i);
        const int np = T.np, m = np / B;
        if (r >= m - 1 || k >= m / 2) continue;
        const double* A = cur[i] ? T.A1 : T.A0;
        int bp, bq;
        pair_of(r, k, m, &bp, &bq);
        __syncthreads();  // the previous task's reads are done
        {
          const int x = threadIdx.x / BB, y = threadIdx.x % BB;
          const int gx = x < B ? bp * B + x : bq * B + x - B, gy = y < B ? bp * B + y : bq * B + y - B;
          sA[0][0][x][y] = __ldcg(A + (int64_t)gx * np + gy);
          sJ[0][x][y] = x == y ? 1.0 : 0.0;
        }
        __syncthreads();
        const int rounds = r == 0 ? BB - 1 : B;
        // pair j of inner round q
        auto inner = [&](int q, int j, int* x, int* y) {
          if (r == 0) {
            pair_of(q, j, BB, x, y);
          } else {
            *x = j;
            *y = B + ((j + q) & (B - 1));
          }
        };
        const int l = t & (B - 1), rr = t >> 3;  // column pair, row (of 16; for A in pair order)
        int c = 0;
        for (int q = 0; q < rounds; ++q, c ^= 1) {
          double* cs = sCS[c];
          if (threadIdx.x < B) {
            int x, y;
            inner(q, threadIdx.x, &x, &y);
            angle(sA[0][c][x][x], sA[0][c][y][y], sA[0][c][x][y], cs + 2 * threadIdx.x, cs + 2 * threadIdx.x + 1);
          }
          __syncthreads();
          int qx, qy;
          inner(q, l, &qx, &qy);
          const double cl = cs[2 * l], sl = cs[2 * l + 1];
          if (g == 0) {
            int px, py;
            inner(q, rr >> 1, &px, &py);
            const double ck = cs[2 * (rr >> 1)], sk = cs[2 * (rr >> 1) + 1];
            const double u0 = sA[0][c][px][qx], u1 = sA[0][c][px][qy];
            const double v0 = sA[0][c][py][qx], v1 = sA[0][c][py][qy];
            const bool second = rr & 1;
            const double x0 = second ? sk : ck, x1 = second ? ck : -sk;
            const double m0 = fma(x1, v0, x0 * u0), m1 = fma(x1, v1, x0 * u1);
            const int row = second ? py : px;
            sA[0][c ^ 1][row][qx] = fma(-sl, m1, cl * m0);
            sA[0][c ^ 1][row][qy] = fma(sl, m0, cl * m1);
            group_sync(0);
          } else {
            const double j0 = sJ[0][rr][qx], j1 = sJ[0][rr][qy];
            sJ[0][rr][qx] = fma(-sl, j1, cl * j0);
            sJ[0][rr][qy] = fma(sl, j0, cl * j1);
            group_sync(1);
          }
        }
        __syncthreads();
        __stcg(T.J + (int64_t)k * BB * BB + threadIdx.x, sJ[0][threadIdx.x / BB][threadIdx.x % BB]);
      }
      grid.sync();
      // phase 2: A <- J^T A J (half a 16 x 16 block per task) and Q <- Q J (8 rows)
      const int a_max = half_max * (half_max + 1), q_max = a.m_max * half_max;
      for (int64_t w = spread; w < (int64_t)(a_max + q_max) * a.n_inst; w += ngroups) {
        const int i = (int)(w % a.n_inst);
        int k = (int)(w / a.n_inst);
        if (done[i]) continue;
        const EigTask& T = task(a, i);
        const int np = T.np, m = np / B, half = m / 2;
        if (r >= m - 1) continue;
        const double* A = cur[i] ? T.A1 : T.A0;
        double* An = cur[i] ? T.A0 : T.A1;
        const int i8 = t >> 4, col = t & (BB - 1);
        int lp, lq;
        if (k < a_max) {
          const int h = k & 1;
          int kk = 0, rest = k >> 1;
          if (rest >= half * (half + 1) / 2) continue;
          while (rest >= half - kk) {
            rest -= half - kk;
            ++kk;
          }
          const int l = kk + rest;
          int kp, kq;
          pair_of(r, kk, m, &kp, &kq);
          pair_of(r, l, m, &lp, &lq);
          group_sync(g);
          for (int e = t; e < BB * BB; e += GROUP) {
            const int x = e / BB, y = e % BB;
            const int gx = x < B ? kp * B + x : kq * B + x - B, gy = y < B ? lp * B + y : lq * B + y - B;
            sA[g][0][x][y] = __ldcg(A + (int64_t)gx * np + gy);
            sA[g][1][x][y] = __ldcg(T.J + (int64_t)kk * BB * BB + e);
            sJ[g][x][y] = __ldcg(T.J + (int64_t)l * BB * BB + e);
          }
          group_sync(g);
          const int row = h * B + i8;
          double x0 = 0.0, x1 = 0.0;
#pragma unroll
          for (int p = 0; p < BB; p += 2) {
            x0 = fma(sA[g][1][p][row], sA[g][0][p][col], x0);
            x1 = fma(sA[g][1][p + 1][row], sA[g][0][p + 1][col], x1);
          }
          group_sync(g);
          sA[g][0][i8][col] = x0 + x1;
          group_sync(g);
          x0 = x1 = 0.0;
#pragma unroll
          for (int p = 0; p < BB; p += 2) {
            x0 = fma(sA[g][0][i8][p], sJ[g][p][col], x0);
            x1 = fma(sA[g][0][i8][p + 1], sJ[g][p + 1][col], x1);
          }
          const int gx = row < B ? kp * B + row : kq * B + row - B, gy = col < B ? lp * B + col : lq * B + col - B;
          __stcg(An + (int64_t)gx * np + gy, x0 + x1);
          if (kk != l) __stcg(An + (int64_t)gy * np + gx, x0 + x1);
        } else {
          k -= a_max;
          const int strip = k / half_max, l = k % half_max;
          if (strip >= m || l >= half) continue;
          pair_of(r, l, m, &lp, &lq);
          const int gy = col < B ? lp * B + col : lq * B + col - B;
          double* qp = T.Q + (int64_t)(strip * B + i8) * np + gy;
          group_sync(g);
          sA[g][0][i8][col] = __ldcg(qp);
          for (int e = t; e < BB * BB; e += GROUP)
            sJ[g][e / BB][e % BB] = __ldcg(T.J + (int64_t)l * BB * BB + e);
          group_sync(g);
          double x0 = 0.0, x1 = 0.0;
#pragma unroll
          for (int p = 0; p < BB; p += 2) {
            x0 = fma(sA[g][0][i8][p], sJ[g][p][col], x0);
            x1 = fma(sA[g][0][i8][p + 1], sJ[g][p + 1][col], x1);
          }
          __stcg(qp, x0 + x1);
        }
      }
      grid.sync();
      for (int i = threadIdx.x; i < a.n_inst; i += EIG_THREADS)
        if (!done[i] && r < task(a, i).np / B - 1) cur[i] ^= 1;
      __syncthreads();
    }
  }

  // ascending eigenvalues (ties by index) and the matching columns of Q
  for (int i = 0; i < a.n_inst; ++i) {
    const EigTask& T = task(a, i);
    if (!live(T)) continue;
    const int n = T.n, np = T.np;
    const double* A = cur[i] ? T.A1 : T.A0;
    const int shift = *(volatile int*)T.shift;
    const bool bad = shift == INT_MIN;  // inf or NaN in H
    for (int c = blockIdx.x * (EIG_THREADS / 32) + warp; c < n; c += gridDim.x * (EIG_THREADS / 32)) {
      const double v = __ldcg(A + (int64_t)c * np + c);
      const unsigned long long kv = order_key(v);
      int rank = 0;
      if (bad) {
        rank = c;
      } else {
        for (int j = lane; j < n; j += 32) {
          const unsigned long long kj = order_key(__ldcg(A + (int64_t)j * np + j));
          rank += kj < kv || (kj == kv && j < c);
        }
        rank = __reduce_add_sync(0xffffffffu, rank);
      }
      if (lane == 0) T.w[rank] = bad ? __longlong_as_double(0x7FF8000000000000ll) : scalbn(v, -shift);
      for (int x = lane; x < n; x += 32)
        T.Qout[(int64_t)x * n + rank] =
            bad ? __longlong_as_double(0x7FF8000000000000ll) : __ldcg(T.Q + (int64_t)x * np + c);
    }
  }
}

int eig_grid(const fd_ctx* ctx, int n_inst, int m_max) {
  const int64_t half = m_max / 2, tasks = (half * (half + 1) + m_max * half) * n_inst;
  return (int)std::max<int64_t>(1, std::min<int64_t>(tasks, ctx->num_sms));
}

fd_status launch(fd_ctx* ctx, EigArgs& a, int grid) {
  void* args[] = {&a};
  // three bytes per matrix beside 13 KB of static arrays: from 11,900 matrices on more than
  // a launch gets unasked
  if (a.n_inst > 8192)
    FD_CUDA(ctx, cudaFuncSetAttribute(k_block_jacobi, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024));
  FD_CUDA(ctx, cudaLaunchCooperativeKernel((const void*)k_block_jacobi, grid, EIG_THREADS, args,
                                           (size_t)3 * a.n_inst, ctx->stream));
  FD_LAUNCHED(ctx);
  return FD_OK;
}

}  // namespace

int eig_padded(int n) { return (int)cdiv(n, BB) * BB; }

size_t eig_work_doubles(int n) {
  const size_t np = eig_padded(n);
  return 3 * np * np + np / BB * BB * BB + 1;  // A0, A1, Q, J, shift
}

void eig_task_layout(EigTask* t, int n, double* work) {
  const size_t np = eig_padded(n);
  t->n = n;
  t->np = (int)np;
  t->A0 = work;
  t->A1 = t->A0 + np * np;
  t->Q = t->A1 + np * np;
  t->J = t->Q + np * np;
  t->shift = (int*)(t->J + np / BB * BB * BB);
}

size_t eig_part_floats(const fd_ctx* ctx, int n_inst) { return (size_t)2 * ctx->num_sms * n_inst; }

fd_status eig_batch(fd_ctx* ctx, const EigTask* tasks_dev, int n_inst, int n_max, int max_sweeps, float* part) {
  EigArgs a{};
  a.many = tasks_dev;
  a.n_inst = n_inst;
  a.m_max = eig_padded(n_max) / B;
  a.max_sweeps = max_sweeps;
  a.tol2 = 1e-28f;
  a.part = part;
  return launch(ctx, a, eig_grid(ctx, n_inst, a.m_max));
}

fd_status sym_eig(fd_ctx* ctx, double* H, int n, double* w, double* Q, int max_sweeps) {
  void* p;
  FD_TRY(workspace(ctx, "jacobi", sizeof(double) * eig_work_doubles(n) + sizeof(float) * eig_part_floats(ctx, 1), &p));
  EigArgs a{};
  eig_task_layout(&a.one, n, (double*)p);
  a.one.H = H;
  a.one.w = w;
  a.one.Qout = Q;
  a.n_inst = 1;
  a.m_max = a.one.np / B;
  a.max_sweeps = max_sweeps;
  a.tol2 = 1e-28f;
  a.part = (float*)((double*)p + eig_work_doubles(n));
  return launch(ctx, a, eig_grid(ctx, 1, a.m_max));
}

}  // namespace fdi
