// The Chebyshev filter of small matrices, all degree steps in one launch
// (Sec. 2, Alg. 2).
//
// A launched step cannot take less than about 3.5 us (launch, then a chain of
// dependent loads: row -> chunk -> entries -> gathers -> stores), whatever the
// matrix: 4 us at 1,728 rows, 8 us at 4,900 rows and nb = 16 in FP64, where the
// FP64 pipe itself needs 1.5 us.  The columns of a block are independent, so here
// one CTA, or a thread-block cluster where one SM's arithmetic would set the
// time, takes a panel of the block's columns through all steps.  Each CTA owns a
// run of rows and keeps their matrix entries and accumulator, and a copy of all
// rows of the panel's x_{k-1} and x_{k-2}, in shared memory: gathers are local, and a
// new row goes to the other CTAs as coalesced distributed-shared-memory stores
// before the cluster's hardware barrier.  (Gathering remotely instead, from the
// other CTAs' shared memory or through L2, was 2 to 4 times slower: scattered
// 8-byte reads cost several clocks each.)  Clusters never wait for one another.
// Measured per step (launched steps then -> this): 400 rows 6.6 -> 1.4 us
// (FP64), 0.76 (FP32); 1,728 rows, nb = 16, FP64 6.6 -> 1.8, FP32 5.3 -> 1.6,
// float-float 6.6 -> 1.4; 4,900 rows of 8 entries, nb = 16, FP64 8.5 -> 5.6, FP32
// 8.6 -> 2.1; 4,096 stencil rows, nb = 32, FP64 8.6 -> 4.8.
//
// A panel is PW units of 8 bytes wide (one double, one float-float pair, two
// floats), a thread holds one unit of a row at a time.  The matrix is scaled while
// it is staged, A' = 2 (alpha A + beta), so a step is
//   x_k = (sum_{j > 0} a'_ij x_j) + (a'_ii x_i - x_{k-2}),
// nnz + 1 operations on GB300's slow FP64 pipe instead of nnz + 4; the split into the
// two sums keeps the rounding error where it was (measured against quadruple
// precision at degrees 20 .. 8000: 0.96 .. 1.02 of the launched step's; taking
// -x_{k-2} first into one chain would cost 1.2 to 1.4 times).  The first step is half of
// A' x_0 (exact).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "fd_ff.cuh"
#include "fd_internal.cuh"
#include "fd_step.cuh"

namespace fdi {
namespace small {

using ffa::ff;

// arithmetic on 8-byte units
template <typename T>
struct Ops;
template <>
struct Ops<double> {
  using U = double;
  using S = double;
  static constexpr int E = 1;  // block columns per unit
  static __device__ __forceinline__ U mul(S a, U x) { return a * x; }
  static __device__ __forceinline__ U fma(S a, U x, U c) { return ::fma(a, x, c); }
  static __device__ __forceinline__ U neg(U x) { return -x; }
  static __device__ __forceinline__ U add(U x, U y) { return x + y; }
  static __device__ __forceinline__ U half(U x) { return 0.5 * x; }
  static __device__ __forceinline__ U madd(U c, S a, U x) { return ::fma(a, x, c); }
  static __device__ __forceinline__ U zero() { return 0.0; }
  static __host__ __device__ __forceinline__ S coef(double v) { return v; }
};
template <>
struct Ops<float> {
  using U = float2;
  using S = float;
  static constexpr int E = 2;
  static __device__ __forceinline__ U mul(S a, U x) { return make_float2(a * x.x, a * x.y); }
  static __device__ __forceinline__ U fma(S a, U x, U c) { return make_float2(fmaf(a, x.x, c.x), fmaf(a, x.y, c.y)); }
  static __device__ __forceinline__ U neg(U x) { return make_float2(-x.x, -x.y); }
  static __device__ __forceinline__ U add(U x, U y) { return make_float2(x.x + y.x, x.y + y.y); }
  static __device__ __forceinline__ U half(U x) { return make_float2(0.5f * x.x, 0.5f * x.y); }
  static __device__ __forceinline__ U madd(U c, S a, U x) { return fma(a, x, c); }
  static __device__ __forceinline__ U zero() { return make_float2(0.0f, 0.0f); }
  static __host__ __device__ __forceinline__ S coef(double v) { return (float)v; }
};
template <>
struct Ops<ff> {
  using U = ff;
  using S = ff;
  static constexpr int E = 1;
  static __device__ __forceinline__ U mul(S a, U x) { return a * x; }
  static __device__ __forceinline__ U fma(S a, U x, U c) { return ffa::fma(a, x, c); }
  static __device__ __forceinline__ U neg(U x) { return -x; }
  static __device__ __forceinline__ U add(U x, U y) { return x + y; }  // normalises
  static __device__ __forceinline__ U half(U x) { return ff(0.5f * x.hi, 0.5f * x.lo); }
  static __device__ __forceinline__ U madd(U c, S a, U x) { return c + a * x; }
  static __device__ __forceinline__ U zero() { return ff(0.0f, 0.0f); }
  static __host__ __device__ __forceinline__ S coef(double v) { return ff(v); }
};

// One block of columns of one matrix.  V: rows in the original order (perm,
// nullptr: SELL order), ldv in elements; X[k & 1] (SELL order, ldw) holds x_k from one
// launch to the next when the steps are split.
template <typename T>
struct Block {
  const int64_t* chunk_ptr;
  const int32_t* row_len;
  const int32_t* col;
  const double* val;
  const int64_t* perm;
  int D, C, max_row;
  T* V;
  int64_t ldv;
  T* X[2];
  int64_t ldw;
  double a2, b2;       // 2 alpha, 2 beta
  int n, k0, k1;       // degree; this launch takes steps k0 .. k1
};

// Steps of one launch are split where the accumulator is complete (step_terms): k1 = 2 mod 3.
constexpr int MAX_STEPS = 999;

constexpr int MAX_ROWS = 65535;  // columns are kept as 16-bit row numbers

// shared memory of a CTA with R of D rows, in bytes
template <typename T>
__host__ __device__ inline size_t cta_smem(int D, int R, int pw, int max_row) {
  return 2 * 8 * (size_t)D * pw + (size_t)R * (8 * (size_t)pw + (size_t)max_row * (2 + sizeof(typename Ops<T>::S)) + 2);
}
__host__ __device__ inline int cta_rows(int D, int cluster) {
  const int r = (D + cluster - 1) / cluster;
  return (r + 3) & ~3;
}

__device__ __forceinline__ uint32_t shared_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// store one unit at the same place in the shared memory of CTA `rank` of the cluster
template <typename U>
__device__ __forceinline__ void store_rank(uint32_t addr, uint32_t rank, const U& u) {
  static_assert(sizeof(U) == 8, "8-byte units");
  uint2 raw;
  memcpy(&raw, &u, 8);
  asm volatile("{\n .reg .u32 a;\n mapa.shared::cluster.u32 a, %0, %1;\n st.shared::cluster.v2.u32 [a], {%2, %3};\n}\n"
               ::"r"(addr), "r"(rank), "r"(raw.x), "r"(raw.y) : "memory");
}
template <bool CLUSTER>
__device__ __forceinline__ void step_barrier() {
  if (CLUSTER)
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
  else
    __syncthreads();
}

// The filter steps b.k0 .. b.k1 of the panel of PW units at unit u0, by the CTA of
// rank `rank` in a cluster of `ranks`; mu: coefficient k at mu[k - mu0].  Every
// thread of the cluster calls it.
template <typename T, int PW, bool CLUSTER, typename Mu>
__device__ __forceinline__ void filter_panel(const Block<T>& b, int u0, uint32_t rank, uint32_t ranks,
                                             unsigned char* smem, Mu&& mu) {
  using O = Ops<T>;
  using U = typename O::U;
  using S = typename O::S;
  const int R = cta_rows(b.D, (int)ranks);
  const int r0 = (int)rank * R, rows = max(0, min(R, b.D - r0));
  const int all = b.D * PW;                          // units of a whole vector
  U* x = reinterpret_cast<U*>(smem);                 // 2 x D x PW: x_k in buffer k & 1
  U* acc = x + 2 * all;                              // R x PW
  S* val = reinterpret_cast<S*>(acc + R * PW);       // max_row x R
  uint16_t* col = reinterpret_cast<uint16_t*>(val + (size_t)b.max_row * R);  // max_row x R
  uint16_t* len = col + (size_t)b.max_row * R;       // R
  const int units = rows * PW, own = r0 * PW;
  constexpr int GATHERS = 4;  // in flight together
  auto global = [&](T* p, int64_t ld, int row, int u) {
    return reinterpret_cast<U*>(p + (int64_t)row * ld + (int64_t)(u0 + u) * O::E);
  };
  for (int i = threadIdx.x; i < rows; i += blockDim.x) {
    const uint32_t row = (uint32_t)(r0 + i), C = (uint32_t)b.C, chunk = row / C;
    const int64_t base = b.chunk_ptr[chunk] + (row - chunk * C);
    const int n = b.row_len[row];
    len[i] = (uint16_t)n;
    for (int e = 0; e < n; ++e) {
      const double v = b.val[base + (int64_t)e * C];
      val[(size_t)e * R + i] = O::coef(e == 0 ? ::fma(b.a2, v, b.b2) : b.a2 * v);
      col[(size_t)e * R + i] = (uint16_t)b.col[base + (int64_t)e * C];
    }
  }
  for (int q = threadIdx.x; q < all; q += blockDim.x) {
    const int row = q / PW, u = q % PW;
    if (b.k0 == 1) {
      x[q] = *global(b.V, b.ldv, b.perm ? (int)b.perm[row] : row, u);
    } else {
      x[q] = *global(b.X[0], b.ldw, row, u);
      x[all + q] = *global(b.X[1], b.ldw, row, u);
      if (q >= own && q < own + units) acc[q - own] = *global(b.V, b.ldv, b.perm ? (int)b.perm[row] : row, u);
    }
  }
  step_barrier<CLUSTER>();
  for (int k = b.k0; k <= b.k1; ++k) {
    const int cur = (k - 1) & 1;  // x_{k-1}; the other buffer holds x_{k-2}
    const U* xc = x + cur * all;
    U* xn = x + (cur ^ 1) * all;
    const int terms = k == 2 ? 3 : k < 2 ? 0 : step::step_terms(k, b.n);
    S m0{}, m1{}, m2{};
    if (terms) {
      m0 = mu(k - 2);
      m1 = mu(k - 1);
      m2 = mu(k);
    }
    for (int q = threadIdx.x; q < units; q += blockDim.x) {
      const int i = q / PW;
      const int u = q % PW;
      const int n = len[i];
      const U xi = xc[own + q];
      U z = O::zero();
      if (k > 1) z = xn[own + q];
      const U d = k > 1 ? O::fma(val[i], xi, O::neg(z)) : O::mul(val[i], xi);
      U s = O::zero();
      for (int e0 = 1; e0 < n; e0 += GATHERS) {
        U g[GATHERS];
#pragma unroll
        for (int p = 0; p < GATHERS; ++p)
          if (e0 + p < n) g[p] = xc[(int)col[(size_t)(e0 + p) * R + i] * PW + u];
#pragma unroll
        for (int p = 0; p < GATHERS; ++p)
          if (e0 + p < n) {
            const S a = val[(size_t)(e0 + p) * R + i];
            s = e0 + p == 1 ? O::mul(a, g[p]) : O::fma(a, g[p], s);
          }
      }
      U y = O::add(s, d);
      if (k == 1) y = O::half(y);
      xn[own + q] = y;
      if (CLUSTER) {
        const uint32_t a = shared_addr(xn + own + q);
        for (uint32_t r = 1; r < ranks; ++r) store_rank(a, rank + r < ranks ? rank + r : rank + r - ranks, y);
      }
      if (terms) {
        U o;
        if (k == 2) {
          o = O::madd(O::madd(O::mul(m0, z), m1, xi), m2, y);
        } else {
          o = acc[q];
          if (terms > 2) o = O::madd(o, m0, z);
          if (terms > 1) o = O::madd(o, m1, xi);
          o = O::madd(o, m2, y);
        }
        acc[q] = o;
      }
    }
    step_barrier<CLUSTER>();
  }
  for (int q = threadIdx.x; q < units; q += blockDim.x) {
    const int i = q / PW, u = q % PW, row = r0 + i;
    const int vrow = b.perm ? (int)b.perm[row] : row;
    *global(b.V, b.ldv, vrow, u) = acc[q];
    if (b.k1 < b.n) {
      *global(b.X[0], b.ldw, row, u) = x[own + q];
      *global(b.X[1], b.ldw, row, u) = x[all + own + q];
    }
  }
}

}  // namespace small
}  // namespace fdi
