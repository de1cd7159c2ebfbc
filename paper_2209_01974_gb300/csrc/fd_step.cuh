// Device building blocks of the fused Chebyshev step (Sec. 2, Alg. 2), shared
// by the single-block filter and the batched persistent filter.
//
// Work mapping: a group of G lanes owns one SELL row; each lane holds CPL
// 16-byte vectors of the row (G * CPL * 16 bytes = nb * sizeof(T)), so every
// gathered row of W1 is one fully coalesced access.  A warp holds 32/G
// consecutive rows of one SELL chunk, so the warp's matrix loads at entry j
// touch adjacent words of the chunk's column-major slab.  Entry 0 of every
// SELL row is its diagonal, so the row's own W1 vector (needed for the beta
// term) is the first gathered vector.  W2 and V are touched once per step and
// use evict-first (.cs) loads and stores, keeping L2 for the W1 gathers.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace fdi {
namespace step {

template <typename T>
struct V16;
template <>
struct V16<double> {
  static constexpr int E = 2;
  double v[2];
  __device__ __forceinline__ void ldg(const double* p) {
    double2 t = __ldg(reinterpret_cast<const double2*>(p));
    v[0] = t.x; v[1] = t.y;
  }
  // coherent loads of vectors written by the previous step (see step_wait): ld keeps
  // its place in the program, ldm may move between other loads
  __device__ __forceinline__ void ldm(const double* p) {
    const double2 t = *reinterpret_cast<const double2*>(p);
    v[0] = t.x; v[1] = t.y;
  }
  __device__ __forceinline__ void ld(const double* p) {
    asm volatile("ld.global.v2.f64 {%0, %1}, [%2];\n" : "=d"(v[0]), "=d"(v[1]) : "l"(p) : "memory");
  }
  __device__ __forceinline__ void ldcs(const double* p) {
    asm volatile("ld.global.cs.v2.f64 {%0, %1}, [%2];\n" : "=d"(v[0]), "=d"(v[1]) : "l"(p) : "memory");
  }
  __device__ __forceinline__ void stcs(double* p) const {
    __stcs(reinterpret_cast<double2*>(p), make_double2(v[0], v[1]));
  }
  __device__ __forceinline__ void st(double* p) const {
    *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
  }
  // loads and stores with an L2 eviction policy (createpolicy); the loads do
  // not allocate in L1
  __device__ __forceinline__ void ld_pol(const double* p, uint64_t pol) {
    asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v2.f64 {%0, %1}, [%2], %3;\n"
                 : "=d"(v[0]), "=d"(v[1]) : "l"(p), "l"(pol) : "memory");
  }
  __device__ __forceinline__ void st_pol(double* p, uint64_t pol) const {
    asm volatile("st.global.L2::cache_hint.v2.f64 [%0], {%1, %2}, %3;\n"
                 :: "l"(p), "d"(v[0]), "d"(v[1]), "l"(pol));
  }
};
template <>
struct V16<float> {
  static constexpr int E = 4;
  float v[4];
  __device__ __forceinline__ void ldg(const float* p) {
    float4 t = __ldg(reinterpret_cast<const float4*>(p));
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
  }
  __device__ __forceinline__ void ldm(const float* p) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
  }
  __device__ __forceinline__ void ld(const float* p) {
    asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];\n"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "l"(p) : "memory");
  }
  __device__ __forceinline__ void ldcs(const float* p) {
    asm volatile("ld.global.cs.v4.f32 {%0, %1, %2, %3}, [%4];\n"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "l"(p) : "memory");
  }
  __device__ __forceinline__ void stcs(float* p) const {
    __stcs(reinterpret_cast<float4*>(p), make_float4(v[0], v[1], v[2], v[3]));
  }
  __device__ __forceinline__ void st(float* p) const {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  }
  __device__ __forceinline__ void ld_pol(const float* p, uint64_t pol) {
    asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;\n"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "l"(p), "l"(pol) : "memory");
  }
  __device__ __forceinline__ void st_pol(float* p, uint64_t pol) const {
    asm volatile("st.global.L2::cache_hint.v4.f32 [%0], {%1, %2, %3, %4}, %5;\n"
                 :: "l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "l"(pol));
  }
};

// L2 eviction policies for cache_hint accesses: the whole access range evicts
// last (data re-read within a short window) or first (streamed once)
__device__ __forceinline__ uint64_t policy_evict_last() {
  uint64_t p;
  asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;\n" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t p;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;\n" : "=l"(p));
  return p;
}

// read-only load of one matrix value (float-float values have their own)
template <typename T>
__device__ __forceinline__ T ldg_val(const T* p) { return __ldg(p); }

template <typename T>
struct SellArgs {
  const int64_t* chunk_ptr;
  const int32_t* row_len;
  const int32_t* col;
  const T* val;
  int64_t D;
  int C;
};

// Step k holds x_{k-2} (z), x_{k-1} (the row's own gathered vector) and x_k, so
// one step in three adds the last three terms to the accumulator (MODE_GENERIC)
// and the two others leave it alone (MODE_PLAIN): 11/3 vectors moved per step on
// average instead of five.  The terms enter the sum in the same order and from
// the same stored values as one by one.  MODE_EITHER decides by nacc at run time.
enum { MODE_SPMMV = 0, MODE_SECOND = 1, MODE_GENERIC = 2, MODE_PLAIN = 3, MODE_EITHER = 4 };

template <typename T>
struct StepArgs {
  const T* X; int64_t ldx;   // gathered operand x_{k-1}
  const T* Z; int64_t ldz;   // x_{k-2}, row-wise (may alias Y or Vout at the same row)
  T* Y; int64_t ldy;         // x_k output, or nullptr
  const T* Vin; int64_t ldvi;
  T* Vout; int64_t ldvo;
  T c_ax, c_x;               // x_k = c_ax * (A x_{k-1}) + c_x * x_{k-1} [- x_{k-2}]
  T mu0, mu1, mu2;           // SECOND: Vout = mu0 z + mu1 x + mu2 y; GENERIC: Vout = Vin + [mu0 z +]
                             // [mu1 x +] mu2 y, the last nacc (1 .. 3) of the terms, or no accumulation (0)
  int nacc;
  int scaled;                // the matrix is A' = c_ax A + c_x I: c_ax, c_x are not applied again
};

template <int MODE, typename S>
__device__ __forceinline__ bool accumulates(const S& s) {
  return MODE == MODE_SECOND || MODE == MODE_GENERIC || (MODE == MODE_EITHER && s.nacc);
}

// Which of the generic steps 3 .. n accumulate, and how many terms: the second
// step has added mu_0 .. mu_2, then every third step adds three, and the last
// step whatever is left.
__host__ __device__ __forceinline__ int step_terms(int k, int n) {
  const int r = (k - 2) % 3;
  return r == 0 ? 3 : k == n ? r : 0;
}

// Programmatic dependent launch: a step kernel lets the next one's CTAs start
// while its own last CTAs run (step_release), and touches the vectors the
// previous step wrote only after that step has completed (step_wait); what it
// loads before the wait (matrix entries, hop lists) is written by no step.
// Every thread passes step_wait, so a step's completion implies its
// predecessors'.  The vectors are read with coherent loads (a step starts
// before its operands are final, which rules out the read-only path).
__device__ __forceinline__ void step_release() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void step_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

constexpr int WARPS = 8;
constexpr int BATCH = 4;   // entries per batch; SELL chunk lengths are multiples of 8
constexpr int MIN_BLOCKS = 12;     // FP32 steps: 4-warp CTAs, 48 resident warps per SM (<= 40 registers)
constexpr int MIN_BLOCKS_F64 = 4;  // matrix-free and batched FP64 steps: 8-warp CTAs with 64 registers
// CTA shape of the fused step (k_cheb_step): warps per CTA and resident CTAs
// per SM (the launch bounds).  FP32: 48 warps per SM (more spill, fewer hide less
// latency: 14 CTAs 28 % slower); FP64, bound by its pipe, 32 warps with 64 registers,
// in 4-warp CTAs because the last wave then ends more evenly (8-warp CTAs 1 to 3 %
// slower); other arithmetic types may specialise it.
template <typename T>
struct StepShape {
  static constexpr int warps = 4;
  static constexpr int min_blocks = sizeof(T) == 4 ? MIN_BLOCKS : 8;
};
template <typename T>
__host__ __device__ constexpr int step_warps() { return StepShape<T>::warps; }
template <typename T>
__host__ __device__ constexpr int step_min_blocks() { return StepShape<T>::min_blocks; }

template <typename T, int NB>
struct Layout {
  static constexpr int E = V16<T>::E;
  static constexpr int Q = NB / E;                 // 16-byte vectors per row
  static constexpr int G = Q >= 32 ? 32 : Q;        // lanes per row
  static constexpr int CPL = Q / G;                 // vectors per lane
  static constexpr int RPW = 32 / G;                // rows per warp
  static_assert(NB % E == 0 && Q % G == 0, "nb must fill whole 16-byte vectors");
};

// The first BATCH entries of a SELL row and where the rest is.
template <typename T>
struct RowHead {
  const int32_t* cp;
  const T* vp;
  uint32_t C;
  int32_t c[BATCH];
  T a[BATCH];
  // Rows at or beyond D inside the last chunk are SELL padding rows: their
  // entries exist (value 0, column 0), but they have no vector row.
  __device__ __forceinline__ void load(const SellArgs<T>& A, int64_t row, bool active) {
    C = (uint32_t)A.C;
    const uint32_t r = (uint32_t)row, chunk = r / C;  // rows < 2^31: a 64-bit division costs tens of instructions
    const int64_t base = __ldg(A.chunk_ptr + chunk) + (r - chunk * C);
    cp = A.col + base;
    vp = A.val + base;
#pragma unroll
    for (int u = 0; u < BATCH; ++u) {
      c[u] = __ldg(cp + u * C);
      a[u] = ldg_val(vp + u * C);
    }
    if (!active) { c[0] = 0; a[0] = T(0); }
  }
};

// FP64 and float-float steps sum a row as (sum_{j > 0} a_ij x_j) + (a_ii x_i - z):
// with the matrix scaled beforehand that is the whole of x_k, in nnz + 1 operations
// instead of nnz + 4 on the pipes that bound these steps, at the same rounding
// error (see fd_small.cuh).
template <typename T, int MODE>
__host__ __device__ constexpr bool split_diagonal() { return sizeof(T) == 8 && MODE != MODE_SPMMV; }

// Gather-accumulate s = sum_j a_ij x_j over the SELL row (SPLIT: without the
// diagonal), returning the row's own vector xi (entry 0 is the diagonal).  Entries are taken BATCH at a time:
// the matrix loads of a batch, then all its gathers, so a row of up to BATCH
// entries costs one round trip of dependent loads.  Chunk lengths are padded to
// a multiple of BATCH with (0, own row) entries, so the matrix loads need no
// bounds; the gathers and FMAs of entries past the row's own length are
// skipped (FP64 arithmetic, not memory, bounds the FP64 step on GB300).
template <typename T, int NB, bool SPLIT = false>
__device__ __forceinline__ void row_product(const RowHead<T>& h, const T* X, int64_t ldx, int len, int wlen,
                                            int gl, V16<T> (&acc)[Layout<T, NB>::CPL],
                                            V16<T> (&xi)[Layout<T, NB>::CPL]) {
  using L = Layout<T, NB>;
  constexpr int E = L::E;
  const uint32_t ld = (uint32_t)ldx;
  const T* xl = X + gl * E;
#pragma unroll
  for (int v = 0; v < L::CPL; ++v) {
    xi[v].ld(xl + (uint64_t)(uint32_t)h.c[0] * ld + v * L::G * E);
#pragma unroll
    for (int e = 0; e < E; ++e) acc[v].v[e] = SPLIT ? T(0) : h.a[0] * xi[v].v[e];
  }
#pragma unroll
  for (int u = 1; u < BATCH; ++u) {
    if (u < len) {  // entries past the row's length are padding: skip their FMAs
#pragma unroll
      for (int v = 0; v < L::CPL; ++v) {
        V16<T> x;
        x.ld(xl + (uint64_t)(uint32_t)h.c[u] * ld + v * L::G * E);
#pragma unroll
        for (int e = 0; e < E; ++e) acc[v].v[e] = fma(h.a[u], x.v[e], acc[v].v[e]);
      }
    }
  }
  for (int j0 = BATCH; j0 < wlen; j0 += BATCH) {
    int32_t c[BATCH];
    T a[BATCH];
#pragma unroll
    for (int u = 0; u < BATCH; ++u) {
      c[u] = __ldg(h.cp + (j0 + u) * h.C);
      a[u] = ldg_val(h.vp + (j0 + u) * h.C);
    }
#pragma unroll
    for (int u = 0; u < BATCH; ++u) {
      if (j0 + u < len) {
#pragma unroll
        for (int v = 0; v < L::CPL; ++v) {
          V16<T> x;
          x.ld(xl + (uint64_t)(uint32_t)c[u] * ld + v * L::G * E);
#pragma unroll
          for (int e = 0; e < E; ++e) acc[v].v[e] = fma(a[u], x.v[e], acc[v].v[e]);
        }
      }
    }
  }
}

__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];\n" ::"l"(p));
}
// bulk L2 prefetch of `bytes` contiguous bytes (16-byte aligned address and
// size), issued by one thread to the copy engine; nothing waits for it
__device__ __forceinline__ void prefetch_l2_bulk(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(p), "r"(bytes) : "memory");
}

// L2 prefetch for the rows [r0, r1) of a later CTA: the 128-byte lines of
// their row-wise operands (the own row of X, Z, Vin) and the SELL slabs of the
// chunks that start inside the range.  A prefetch holds no register and no
// scoreboard entry, so the later CTA finds its first, dependent loads in L2.
template <typename T, int NB, int MODE>
__device__ __forceinline__ void prefetch_rows(const SellArgs<T>& A, const StepArgs<T>& s,
                                              int64_t r0, int64_t r1) {
  constexpr int LPR = (NB * (int)sizeof(T) + 127) / 128;  // lines per vector row
  constexpr int NS = MODE == MODE_GENERIC ? 3 : MODE == MODE_SPMMV ? 1 : 2;
  const int n = (int)(r1 - r0) * LPR;
  for (int q = threadIdx.x; q < NS * n; q += blockDim.x) {
    const int st = q / n, rq = q % n;
    const int64_t row = r0 + rq / LPR;
    const int64_t off = (int64_t)(rq % LPR) * (128 / (int)sizeof(T));
    const T* p = st == 0 ? s.X + row * s.ldx : st == 1 ? s.Z + row * s.ldz : s.Vin + row * s.ldvi;
    prefetch_l2(p + off);
  }
  if (threadIdx.x >= blockDim.x - 32) {
    const uint32_t C = (uint32_t)A.C, c0 = ((uint32_t)r0 + C - 1) / C, c1 = ((uint32_t)r1 + C - 1) / C;
    if (c0 >= c1) return;
    const int64_t e0 = A.chunk_ptr[c0], e1 = A.chunk_ptr[c1];
    const int64_t l0c = (e0 * 4) >> 7, l1c = (e1 * 4 + 127) >> 7;
    const int64_t l0v = (e0 * (int64_t)sizeof(T)) >> 7, l1v = (e1 * (int64_t)sizeof(T) + 127) >> 7;
    const int64_t nc = l1c - l0c, nv = l1v - l0v;
    const char* cb = reinterpret_cast<const char*>(A.col);
    const char* vb = reinterpret_cast<const char*>(A.val);
    for (int64_t q = threadIdx.x & 31; q < nc + nv; q += 32)
      prefetch_l2(q < nc ? cb + ((l0c + q) << 7) : vb + ((l0v + q - nc) << 7));
  }
}

// x_k of one row from its product (and its diagonal entry a0), and the accumulator
template <typename T, int NB, int MODE>
__device__ __forceinline__ void step_epilogue(const StepArgs<T>& s, int64_t row, int gl, T a0,
                                              const V16<T> (&acc)[Layout<T, NB>::CPL],
                                              const V16<T> (&xi)[Layout<T, NB>::CPL],
                                              const V16<T> (&z)[Layout<T, NB>::CPL],
                                              const V16<T> (&vin)[Layout<T, NB>::CPL]) {
  using L = Layout<T, NB>;
  constexpr int E = L::E;
#pragma unroll
  for (int v = 0; v < L::CPL; ++v) {
    const int64_t off = gl * E + v * L::G * E;
    V16<T> y;
    if (MODE == MODE_SPMMV) {
#pragma unroll
      for (int e = 0; e < E; ++e) y.v[e] = s.c_ax * acc[v].v[e] + s.c_x * xi[v].v[e];
      y.st(s.Y + row * s.ldy + off);
    } else {
#pragma unroll
      for (int e = 0; e < E; ++e) {
        if constexpr (split_diagonal<T, MODE>()) {
          if (s.scaled) {
            y.v[e] = acc[v].v[e] + fma(a0, xi[v].v[e], -z[v].v[e]);
          } else {
            const T ax = acc[v].v[e] + a0 * xi[v].v[e];
            y.v[e] = s.c_ax * ax + s.c_x * xi[v].v[e] - z[v].v[e];
          }
        } else {
          y.v[e] = s.c_ax * acc[v].v[e] + s.c_x * xi[v].v[e] - z[v].v[e];
        }
      }
      if (accumulates<MODE>(s)) {
        V16<T> o;
        if (MODE == MODE_SECOND) {
#pragma unroll
          for (int e = 0; e < E; ++e)
            o.v[e] = s.mu0 * z[v].v[e] + s.mu1 * xi[v].v[e] + s.mu2 * y.v[e];
        } else {
#pragma unroll
          for (int e = 0; e < E; ++e) {
            T a = vin[v].v[e];
            if (s.nacc > 2) a = a + s.mu0 * z[v].v[e];
            if (s.nacc > 1) a = a + s.mu1 * xi[v].v[e];
            o.v[e] = a + s.mu2 * y.v[e];
          }
        }
        o.stcs(s.Vout + row * s.ldvo + off);
      }
      if (s.Y) y.st(s.Y + row * s.ldy + off);
    }
  }
}

// One fused Chebyshev step (or a plain SpMMV) for the warp's rows row0 ..
// row0 + RPW - 1 (row0 < D, a multiple of RPW); all 32 lanes must call it.
// WAIT: the step runs under programmatic dependent launch; the row's first
// entries are loaded before the wait.
template <typename T, int NB, int MODE, bool WAIT = false>
__device__ __forceinline__ void cheb_rows(const SellArgs<T>& A, const StepArgs<T>& s,
                                          int64_t row0) {
  using L = Layout<T, NB>;
  constexpr int E = L::E;
  const int lane = threadIdx.x & 31;
  const int g = lane / L::G, gl = lane % L::G;
  const int64_t row = row0 + g;
  const bool active = row < A.D;
  const int len = active ? __ldg(A.row_len + row) : 0;
  RowHead<T> h;
  h.load(A, row, active);
  const int wlen = __reduce_max_sync(0xffffffffu, len);
  if (WAIT) step_wait();

  // the row-wise operands do not depend on the gathers: issue them first
  V16<T> z[L::CPL], vin[L::CPL];
  if (MODE != MODE_SPMMV && active) {
#pragma unroll
    for (int v = 0; v < L::CPL; ++v) {
      const int64_t off = gl * E + v * L::G * E;
      z[v].ldcs(s.Z + row * s.ldz + off);
      if (MODE != MODE_SECOND && accumulates<MODE>(s)) vin[v].ldcs(s.Vin + row * s.ldvi + off);
    }
  }
  V16<T> acc[L::CPL], xi[L::CPL];
  row_product<T, NB, split_diagonal<T, MODE>()>(h, s.X, s.ldx, len, wlen, gl, acc, xi);
  if (!active) return;

  step_epilogue<T, NB, MODE>(s, row, gl, h.a[0], acc, xi, z, vin);
}

// ---------------------------------------------------------------------------
// Matrix-free Hubbard operator (Sec. 4 runs FD on Hubbard matrices; the
// paper's production runs apply them without storing them):
//   (H x)_(u,d) = U n(u,d) x_(u,d) + sum_u' h_up(u,u') x_(u',d)
//                                  + sum_d' h_dn(d,d') x_(u,d')
// with row (u, d) = u * dim_dn + d.  The up-spin hops of consecutive rows
// (u, d), (u, d + 1) read consecutive rows (u', d), (u', d + 1): whole
// coalesced row blocks; the down-spin hops stay inside the u slab.
// ---------------------------------------------------------------------------
template <typename T>
struct KronArgs {
  int64_t D, dim_dn;
  const uint32_t* bits_up;
  const uint32_t* bits_dn;
  const int64_t* ptr_up;
  const int32_t* col_up;
  const T* val_up;
  const int64_t* ptr_dn;
  const int32_t* col_dn;
  const T* val_dn;
  const T* diag;  // 25 entries: U * n for n doubly occupied sites
};

// s = sum_j h_ij x_j for row (u, d), the entries in the order of the stored
// row (diagonal first, then ascending columns: the up hops to u' < u, the
// down hops, the up hops to u' > u), so the sums round as in the SELL kernel
// (SPLIT: without the diagonal).  Bound by the latency of a hop's table entry and of
// the row that it names: one plain loop per table, so that the compiler unrolls it and
// moves the loads of several hops ahead of their sums, and 32-bit row numbers
// (D < 2^31).  Ring of 10 sites, nb = 16, FP64 and float-float, 2 x 90 steps:
// 5.64 and 3.30 ms; in batches of four hops whose loads keep their place, with 64-bit
// numbers, 7.85 and 4.24 ms.
template <typename T, int NB, bool SPLIT>
__device__ __forceinline__ void kron_row_product(const KronArgs<T>& K, const T* X, int64_t ldx,
                                                 int64_t row, int gl, V16<T> (&acc)[Layout<T, NB>::CPL],
                                                 V16<T> (&xi)[Layout<T, NB>::CPL], T* diag) {
  using L = Layout<T, NB>;
  constexpr int E = L::E;
  const T* xl = X + gl * E;
  const uint32_t dim = (uint32_t)K.dim_dn;
  const uint32_t u = (uint32_t)row / dim, slab = u * dim, d = (uint32_t)row - slab;
  const T dg = K.diag[__popc(__ldg(K.bits_up + u) & __ldg(K.bits_dn + d))];
#pragma unroll
  for (int v = 0; v < L::CPL; ++v) {
    xi[v].ldm(xl + row * ldx + v * L::G * E);
#pragma unroll
    for (int e = 0; e < E; ++e) acc[v].v[e] = SPLIT ? T(0) : dg * xi[v].v[e];
  }
  *diag = dg;
  auto add = [&](T a, uint32_t r) {
#pragma unroll
    for (int v = 0; v < L::CPL; ++v) {
      V16<T> x;
      x.ldm(xl + (uint64_t)r * (uint64_t)ldx + v * L::G * E);
#pragma unroll
      for (int e = 0; e < E; ++e) acc[v].v[e] = fma(a, x.v[e], acc[v].v[e]);
    }
  };
  const int64_t ku = __ldg(K.ptr_up + u), kd = __ldg(K.ptr_dn + d);
  const int nu = (int)(__ldg(K.ptr_up + u + 1) - ku), nd = (int)(__ldg(K.ptr_dn + d + 1) - kd);
  const int32_t *cu = K.col_up + ku, *cd = K.col_dn + kd;
  const T *vu = K.val_up + ku, *vd = K.val_dn + kd;
  int k = 0;
  for (; k < nu && (uint32_t)__ldg(cu + k) < u; ++k) add(ldg_val(vu + k), (uint32_t)__ldg(cu + k) * dim + d);
  for (int j = 0; j < nd; ++j) add(ldg_val(vd + j), slab + (uint32_t)__ldg(cd + j));
  for (; k < nu; ++k) add(ldg_val(vu + k), (uint32_t)__ldg(cu + k) * dim + d);
}

// One fused Chebyshev step with the matrix-free Hubbard operator; the same
// operand loads and epilogue as cheb_rows
template <typename T, int NB, int MODE>
__device__ __forceinline__ void kron_rows(const KronArgs<T>& K, const StepArgs<T>& s, int64_t row0) {
  using L = Layout<T, NB>;
  constexpr int E = L::E;
  const int lane = threadIdx.x & 31;
  const int g = lane / L::G, gl = lane % L::G;
  const int64_t row = row0 + g;
  step_wait();
  if (row >= K.D) return;  // no warp-wide operations follow
  V16<T> z[L::CPL], vin[L::CPL];
  if (MODE != MODE_SPMMV) {
#pragma unroll
    for (int v = 0; v < L::CPL; ++v) {
      const int64_t off = gl * E + v * L::G * E;
      z[v].ldcs(s.Z + row * s.ldz + off);
      if (MODE != MODE_SECOND && accumulates<MODE>(s)) vin[v].ldcs(s.Vin + row * s.ldvi + off);
    }
  }
  V16<T> acc[L::CPL], xi[L::CPL];
  T dg;
  kron_row_product<T, NB, split_diagonal<T, MODE>()>(K, s.X, s.ldx, row, gl, acc, xi, &dg);
  step_epilogue<T, NB, MODE>(s, row, gl, dg, acc, xi, z, vin);
}

}  // namespace step
}  // namespace fdi
