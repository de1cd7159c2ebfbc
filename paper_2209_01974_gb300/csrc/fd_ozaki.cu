// FP64-accurate Gram and rotation products on the tcgen05 tensor cores
// (Ozaki scheme).
//
// GB300 executes FP64 at about 1.2 TFLOP/s but dense bf16 tcgen05.mma at about
// 2 PFLOP/s.  The tall-skinny products of Cholesky-QR and Rayleigh-Ritz
// (Sec. 2) are therefore split into exact integer pieces (Ozaki, Ogita, Oishi,
// Rump, "Error-free transformations of matrix multiplication", Numer.
// Algorithms 2012; Mukunoki et al. 2020 on tensor cores):
//
//   a_ik = 2^{e_i} sum_{s<8} d^a_{s,ik} 2^{-(6+7s)},  -64 <= d <= 64 (7-bit digits)
//   b_kj = 2^{f_j} sum_{t<8} d^b_{t,kj} 2^{-(6+7t)}
//   (AB)_ij = 2^{e_i + f_j} sum_{l<8} 2^{-(12+7l)} sum_{s+t=l} sum_k d^a_s d^b_t
//
// with e_i (f_j) the exponent of the largest |a_ik| over k (|b_kj| over k), so
// each operand is rounded to 55 bits below its row (column) maximum, error at most
// 2^-56, and the pairs s + t >= 8 are dropped.  The digits are balanced (in
// [-64, 63], the first up to 64): every one is exact in bf16, and a product is at
// most 2^12.  A level l sums at most 8 digit pairs; over a K chunk of 512 every
// partial sum stays within 8 * 512 * 2^12 = 2^24, so the FP32 accumulation of the
// tensor core is exact.  (Digits of magnitude and sign up to 127 allow chunks of
// 128 only, and the levels' read-back after each chunk, which the tensor core
// waits for, took a third of the time.)
//
// Two kernels per product.  A streaming kernel cuts each FP64 operand once
// into its 8 bf16 digit slices and writes them to HBM already in the tensor
// core's shared-memory layout (canonical no-swizzle K-major core matrices,
// one contiguous 2 or 4 KB block per 16-deep K step, slice and 64- or
// 128-wide operand block).  The product kernel (one CTA per SM, 512 threads,
// a 128 x 64 output tile, the 8 level accumulators in TMEM: 8 x 64 FP32
// columns = all 512) is a pure Blackwell pipeline: one thread streams the
// digit blocks of each K step into a four-stage shared-memory ring with
// cp.async.bulk (mbarrier complete_tx), one thread issues the step's 12
// tcgen05.mma (36 digit pairs; M 128, N up to 256, K 16) and commits them to the
// stage's "empty" mbarrier, and every 32nd step (K = 512) all threads read
// the levels back with tcgen05.ld, convert them to 32-bit integers, combine
// adjacent levels exactly in 32 bits and add them, scaled by 2^(7 (7 - l)),
// into two 64-bit integer accumulators per output (levels 0-3 and 4-7; value
// = hi 2^28 + lo), exact for up to 2^16 chunks per CTA; one conversion to FP64
// at the end.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <climits>
#include <cmath>

#include "fd_internal.cuh"

namespace fdi {
namespace {

constexpr int OZ_S = 8;             // digits per operand
constexpr int OZ_B = 7;             // bits per digit
constexpr int OZ_F = OZ_S * OZ_B - 1;  // 55 fraction bits
constexpr int OZ_UNIT = OZ_B * (OZ_S - 1) + 2 * (OZ_B - 1);  // accumulator unit 2^-61
constexpr int TM = 128;             // output tile rows (tcgen05 M)
constexpr int TN = 64;              // output tile columns (tcgen05 N)
constexpr int KS = 16;              // K step (one tcgen05.mma)
constexpr int SUBS = 32;            // K steps per exact FP32 chunk (K = 512)
constexpr int NST = 4;              // shared-memory ring stages
constexpr int OZ_THREADS = 512;
constexpr int A_SLICE = TM * KS * 2;                  // 4096 bytes per digit block
constexpr int B_SLICE = TN * KS * 2;                  // 2048 bytes
constexpr int A_ELEMS = A_SLICE / 2, B_ELEMS = B_SLICE / 2;
constexpr int STAGE = OZ_S * (A_SLICE + B_SLICE);     // 49,152 bytes
constexpr int CM_K = 128;                             // K-adjacent core matrices (LBO)
constexpr int CM_MN = (KS / 8) * 128;                 // MN-adjacent 8-row groups (SBO) = 256
constexpr size_t OZ_SMEM = (size_t)NST * STAGE + 2 * NST * 8 + 16;  // + barriers, TMEM address
constexpr size_t LEAVE_BAR = OZ_SMEM - 8;             // barrier of the exit after a timeout
constexpr int64_t OZ_MAX_CHUNKS = 1 << 16;            // per CTA, keeps the accumulators exact
constexpr unsigned TMEM_COLS = 512;                   // 8 levels x 64 columns
constexpr int P_THREAD = 0;                           // bulk-copy producer (warp 0, lanes 0-15)
constexpr int M_THREAD = 32;                          // MMA issuer (warp 1)

// instruction descriptor of tcgen05.mma kind::f16: D FP32 (bits 4-5 = 1),
// A and B bf16 (bits 7-9, 10-12 = 1), both K-major, N >> 3 at bit 17, M >> 4
// at bit 24
__host__ __device__ constexpr uint32_t idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// shared-memory matrix descriptor: start address, leading (K) and stride
// (M/N) byte offsets, descriptor version 1, no swizzle
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((CM_K >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((CM_MN >> 4) & 0x3FFF) << 32) | (1ull << 46);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(bar)));
}

constexpr long long WAIT_CYCLES = 4000000000ll;  // about 2 s at 2 GHz
constexpr long long DRAIN_CYCLES = 200000000ll;  // 0.1 s

// bounded wait for the completion of the barrier phase with the given parity;
// gives up after `limit` SM clock cycles
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, long long limit = WAIT_CYCLES) {
  const long long t0 = clock64();
  for (;;) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    if (done) return true;
    if (clock64() - t0 > limit) return false;
  }
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
// bulk (TMA engine) copy of `bytes` contiguous bytes, completing on `bar`
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

template <int N>
__device__ __forceinline__ void umma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc(N)), "r"(accumulate));
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                   smem_u32(bar))
               : "memory");
}

// 16 columns each of two levels, and the wait for both in the same statement (no
// use of the registers can be scheduled before it)
__device__ __forceinline__ void tmem_ld16x2(uint32_t t0, uint32_t t1, uint32_t (&r0)[16], uint32_t (&r1)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%32];\n"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%33];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(r0[0]), "=r"(r0[1]), "=r"(r0[2]), "=r"(r0[3]), "=r"(r0[4]), "=r"(r0[5]), "=r"(r0[6]), "=r"(r0[7]), "=r"(r0[8]), "=r"(r0[9]), "=r"(r0[10]), "=r"(r0[11]), "=r"(r0[12]), "=r"(r0[13]), "=r"(r0[14]), "=r"(r0[15]),
        "=r"(r1[0]), "=r"(r1[1]), "=r"(r1[2]), "=r"(r1[3]), "=r"(r1[4]), "=r"(r1[5]), "=r"(r1[6]), "=r"(r1[7]), "=r"(r1[8]), "=r"(r1[9]), "=r"(r1[10]), "=r"(r1[11]), "=r"(r1[12]), "=r"(r1[13]), "=r"(r1[14]), "=r"(r1[15])
      : "r"(t0), "r"(t1)
      : "memory");
}

// x 2^(55 - e) rounded to an integer (|x| < 2^e: magnitude at most 2^55), with 64
// added to each of its 8 base-128 digits, so that every field holds its balanced
// digit plus 64
__device__ __forceinline__ unsigned long long biased_fixed(double x, int e) {
  constexpr unsigned long long BIAS = 64ull * (((1ull << 56) - 1) / 127);
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)((bits >> 52) & 0x7FF);
  unsigned long long m = bits & 0xFFFFFFFFFFFFFull;
  if (ex) m |= 1ull << 52;
  const int sh = (ex ? ex : 1) - 1075 - e + OZ_F;  // |x| 2^(F - e) = m 2^sh
  unsigned long long y = 0;
  if (sh >= 0) y = m << sh;
  else if (sh > -64) y = (m + (1ull << (-sh - 1))) >> (-sh);
  return BIAS + ((bits >> 63) ? 0ull - y : y);
}

// bf16 bit pattern of the digit v - 64, v in [0, 128]: the float is built exactly by
// the 2^23 bias trick and its upper half is the bf16 value (8 significant bits)
__device__ __forceinline__ uint32_t bf16_of_digit(uint32_t v) {
  return __float_as_uint(__uint_as_float(0x4B000000u | v) - 8388672.0f) >> 16;
}

// the 8 digit slices of 8 consecutive K values of one operand row (or
// column): slice s of the 8 values is one 16-byte core-matrix row, handed to
// put(s, v)
template <typename Put>
__device__ __forceinline__ void cut8(const double (&x)[8], int e, Put&& put) {
  unsigned long long y[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) y[q] = biased_fixed(x[q], e);
#pragma unroll
  for (int s = 0; s < OZ_S; ++s) {
    const int sh = OZ_B * (OZ_S - 1 - s);
    const uint32_t mask = s == 0 ? 0xFFu : 0x7Fu;  // the first digit may be 64
    uint32_t w[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const uint32_t lo = bf16_of_digit((uint32_t)(y[2 * p] >> sh) & mask);
      const uint32_t hi = bf16_of_digit((uint32_t)(y[2 * p + 1] >> sh) & mask);
      w[p] = lo | (hi << 16);
    }
    put(s, make_uint4(w[0], w[1], w[2], w[3]));
  }
}

// byte offset of (row, k) inside one digit block: 8-row x 16-byte core
// matrices, K-adjacent ones 128 bytes apart, row groups 256 bytes apart
__device__ __forceinline__ int core_offset(int row, int k) {
  return (row >> 3) * CM_MN + (k >> 3) * CM_K + (row & 7) * 16 + (k & 7) * 2;
}

// Exact accumulator of one output: value = hi 2^28 + lo in units of
// 2^-61 2^(e_i + f_j); level l carries the weight 2^(7 (7 - l)).
struct Acc {
  long long hi, lo;
};

// One K step's tensor-core work (issued by one thread).  Level l = s + t collects
// the pairs (s, t) in its TMEM columns l * 64 .., so the products of one slice s of
// A with consecutive slices t of B belong in consecutive columns, and consecutive
// slices of B are consecutive rows of its shared-memory tile: one MMA takes up to
// four of them as one operand of N = 256 (12 MMAs a step instead of 36 of N = 64,
// which are bound by re-reading A from shared memory: 6 KB per 32 clocks of tensor
// work).  Slice 0 of A starts every level of a K chunk, the others accumulate.
template <int S, int T, int CNT>
__device__ __forceinline__ void issue_run(uint32_t tmem, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
  umma<CNT * TN>(tmem + (uint32_t)((S + T) * TN), adesc + (uint64_t)((S * A_SLICE) >> 4),
                 bdesc + (uint64_t)((T * B_SLICE) >> 4), accumulate);
}
template <bool FIRST, int S = 0>
__device__ __forceinline__ void issue_step(uint32_t tmem, uint64_t adesc, uint64_t bdesc) {
  if constexpr (S < OZ_S) {
    constexpr int CNT = OZ_S - S;  // slices of B that meet slice S of A
    constexpr uint32_t ACC = FIRST && S == 0 ? 0u : 1u;
    if constexpr (CNT > 4) {
      issue_run<S, 0, 4>(tmem, adesc, bdesc, ACC);
      issue_run<S, 4, CNT - 4>(tmem, adesc, bdesc, ACC);
    } else {
      issue_run<S, 0, CNT>(tmem, adesc, bdesc, ACC);
    }
    issue_step<FIRST, S + 1>(tmem, adesc, bdesc);
  }
}

// Read the 8 levels of this thread's 16 outputs (TMEM lane = tile row
// 32 (warp & 3) + lane, columns 16 (warp >> 2) ..) into the accumulators.
// Level sums are integers of at most (l + 1) 2^21 (l + 1 pairs x 512 x 2^12), so
// two adjacent levels combine exactly in 32 bits (c_l 2^7 + c_{l+1} <= 7 2^28 + 2^24
// < 2^31 for even l <= 6) and only 32-bit conversions are needed (64-bit ones run
// on GB300's slow FP64 units).
__device__ __forceinline__ void flush(uint32_t tmem, Acc (&acc)[16]) {
  const int w = threadIdx.x >> 5;
  const uint32_t base = tmem + ((uint32_t)(32 * (w & 3)) << 16) + (uint32_t)(16 * (w >> 2));
#pragma unroll 1
  for (int pr = 0; pr < OZ_S / 2; ++pr) {  // level pairs (0,1) (2,3) (4,5) (6,7)
    uint32_t r0[16], r1[16];
    tmem_ld16x2(base + (uint32_t)(2 * pr * TN), base + (uint32_t)((2 * pr + 1) * TN), r0, r1);
    const int sh = (pr & 1) ? 0 : 14;  // pairs (0,1), (4,5) carry 2^14 within hi / lo
#pragma unroll
    for (int c = 0; c < 16; ++c) {
      const int v = __float2int_rz(__uint_as_float(r0[c])) * 128 + __float2int_rz(__uint_as_float(r1[c]));
      const long long t = (long long)v * (1LL << sh);
      if (pr < 2) acc[c].hi += t;
      else acc[c].lo += t;
    }
  }
}

// Before a CTA leaves after a wait that gave up: wait (again with a limit) for the bulk
// copies that it has posted (`loaded` K steps since the ring began), which would otherwise
// arrive in the shared memory of the next CTA, and for the MMAs that it has issued,
// which write TMEM.
__device__ __forceinline__ void drain(unsigned char* smem, uint64_t* full, uint32_t loaded) {
  if (threadIdx.x == P_THREAD)
    for (uint32_t i = loaded > NST ? loaded - NST : 0; i < loaded; ++i)
      mbar_wait(&full[i % NST], (i / NST) & 1u, DRAIN_CYCLES);
  if (threadIdx.x == M_THREAD) {
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + LEAVE_BAR);
    mbar_init(bar);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    umma_commit(bar);  // all MMAs before it
    mbar_wait(bar, 0, DRAIN_CYCLES);
  }
  __syncthreads();
}

// The product pipeline of one CTA.  K step sc reads digit block (sc, s) of A
// at A + sc a_kc + s a_s and of B likewise (bf16 elements).  Returns false if
// a bounded wait gave up (the same answer in every thread).
__device__ __forceinline__ bool run_tile(unsigned char* smem, uint64_t* full, uint64_t* empty, uint32_t tmem,
                                         const __nv_bfloat16* A, int64_t a_kc, int64_t a_s,
                                         const __nv_bfloat16* B, int64_t b_kc, int64_t b_s, int nsub,
                                         bool give_up, Acc (&acc)[16]) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // producer warp: lane 0 posts the stage's byte count, lanes 0-15 issue one
  // bulk copy each (slice lane / 2 of A or B)
  auto load = [&](int sc) {
    const int st = sc % NST;
    unsigned char* dst = smem + (size_t)st * STAGE;
    if (lane == 0) mbar_expect_tx(&full[st], STAGE);
    __syncwarp();
    if (lane < 2 * OZ_S) {
      const int s = lane >> 1;
      if (lane & 1)
        bulk_g2s(dst + OZ_S * A_SLICE + s * B_SLICE, B + sc * b_kc + s * b_s, B_SLICE, &full[st]);
      else
        bulk_g2s(dst + s * A_SLICE, A + sc * a_kc + s * a_s, A_SLICE, &full[st]);
    }
  };
  bool ok = !give_up;
  uint32_t loaded = 0;  // K steps posted by the producer warp
  if (warp == P_THREAD / 32)
    for (; loaded < (uint32_t)nsub && loaded < NST; ++loaded) load((int)loaded);
  for (int sc = 0; sc < nsub; ++sc) {
    const int st = sc % NST;
    const uint32_t par = (uint32_t)(sc / NST) & 1u;
    if (threadIdx.x == M_THREAD && ok) {
      ok = mbar_wait(&full[st], par);
      if (ok) {
        tc_fence_after();
        const uint32_t a0 = smem_u32(smem + (size_t)st * STAGE);
        const uint64_t ad = sdesc(a0), bd = sdesc(a0 + OZ_S * A_SLICE);
        if ((sc % SUBS) == 0) issue_step<true>(tmem, ad, bd);
        else issue_step<false>(tmem, ad, bd);
        umma_commit(&empty[st]);
      }
    }
    if (warp == P_THREAD / 32 && ok && sc + NST < nsub) {
      // the stage is free again once the MMAs of K step sc have completed
      ok = mbar_wait(&empty[st], par);
      if (ok) {
        load(sc + NST);
        ++loaded;
      }
    }
    if ((sc % SUBS) == SUBS - 1 || sc == nsub - 1) {
      // the issuer observes the completion; the others sleep in the barrier
      if (threadIdx.x == M_THREAD && ok) ok = mbar_wait(&empty[st], par);
      if (__syncthreads_or(!ok)) {
        drain(smem, full, loaded);
        return false;
      }
      tc_fence_after();
      flush(tmem, acc);
      tc_fence_before();
      __syncthreads();
    }
  }
  return true;
}

// hi 2^28 + lo scaled by 2^sc, rounded once to nearest (ties to even) by
// integer arithmetic: int64 -> FP64 conversions and FP64 arithmetic run on
// GB300's slow FP64 units
__device__ __forceinline__ double acc_value(const Acc& a, int sc) {
  // 128-bit two's complement N = hi 2^28 + lo as (H, L)
  unsigned long long L = (unsigned long long)a.hi << 28;
  long long H = a.hi >> 36;
  const unsigned long long lo = (unsigned long long)a.lo;
  const unsigned long long L2 = L + lo;
  H += (a.lo >> 63) + (L2 < L ? 1 : 0);  // sign extension of lo, carry
  L = L2;
  const bool neg = H < 0;
  unsigned long long mh = (unsigned long long)H, ml = L;
  if (neg) {  // magnitude
    ml = ~ml + 1;
    mh = ~mh + (ml == 0 ? 1 : 0);
  }
  if (mh == 0 && ml == 0) return 0.0;
  const int p = mh ? 127 - __clzll((long long)mh) : 63 - __clzll((long long)ml);  // leading bit
  unsigned long long m;  // 53-bit significand
  if (p <= 52) {
    m = ml << (52 - p);
  } else {
    const int sh = p - 52;  // 1 .. 75
    unsigned long long q, rem_hi, rem_lo;  // q = N >> sh; remainder bits below
    if (sh < 64) {
      q = (ml >> sh) | (mh << (64 - sh));
      rem_hi = (ml >> (sh - 1)) & 1u;
      rem_lo = sh > 1 ? (ml & ((1ull << (sh - 1)) - 1)) : 0;
    } else {
      q = mh >> (sh - 64);
      rem_hi = sh == 64 ? (ml >> 63) : ((mh >> (sh - 65)) & 1u);
      rem_lo = sh == 64 ? (ml & ~(1ull << 63)) : ((mh & ((1ull << (sh - 65)) - 1)) | ml);
    }
    m = q;
    if (rem_hi && (rem_lo || (m & 1u))) ++m;
  }
  int e = p + sc;  // value = m 2^(e - 52)
  if (m >> 53) {
    m >>= 1;
    ++e;
  }
  if (e < -1022 || e > 1023) return ldexp(neg ? -(double)m : (double)m, e - 52);
  const unsigned long long bits = ((unsigned long long)(neg ? 1 : 0) << 63) |
                                  ((unsigned long long)(e + 1023) << 52) | (m & ((1ull << 52) - 1));
  return __longlong_as_double((long long)bits);
}

// The same for |hi|, |lo| < 2^51 (at most 32 exact chunks): both integers become
// doubles by placing them in the significand of 3 2^79 and 3 2^51; taking both
// offsets off the first leaves hi 2^28 - 3 2^51, a multiple of 2^28 below 2^80 (exact),
// and adding the second rounds hi 2^28 + lo once.  Two FP64 additions and a dozen
// integer instructions instead of 190 (the rotation's tiles end every 4 to 64 K
// steps, and rounding their outputs took as long as the products).
__device__ __forceinline__ double acc_value_small(const Acc& a, int sc) {
  const double x = __longlong_as_double(0x44F8000000000000ll + a.hi);  // (3 2^51 + hi) 2^28
  const double y = __longlong_as_double(0x4338000000000000ll + a.lo);  // 3 2^51 + lo
  const double v = __dadd_rn(__dsub_rn(x, 0x3.0000003p79 /* 3 2^79 + 3 2^51 */), y);
  const long long bits = __double_as_longlong(v);
  const int e = (int)((bits >> 52) & 0x7FF);
  if (e == 0) return 0.0;  // v is an integer: zero
  if (e + sc < 1 || e + sc > 2046) return ldexp(v, sc);
  return __longlong_as_double(bits + ((long long)sc << 52));
}

// CTA prologue: TMEM (warp 0) and the full / empty mbarriers of the ring
__device__ __forceinline__ uint32_t tile_setup(unsigned char* smem, uint64_t** full, uint64_t** empty) {
  unsigned char* tail = smem + (size_t)NST * STAGE;
  *full = reinterpret_cast<uint64_t*>(tail);
  *empty = *full + NST;
  uint32_t* holder = reinterpret_cast<uint32_t*>(tail + 2 * NST * 8);
  if ((threadIdx.x >> 5) == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(holder)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  if (threadIdx.x == 32) {
    for (int i = 0; i < NST; ++i) {
      mbar_init(&(*full)[i]);
      mbar_init(&(*empty)[i]);
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  return *holder;
}

__device__ __forceinline__ void tile_teardown(uint32_t tmem) {
  tc_fence_before();
  __syncthreads();
  if ((threadIdx.x >> 5) == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(TMEM_COLS));
  }
}

// Hand every output of the tile to put(i, j, v): the thread owning it
// converts (scale(i, j) gives the power of two), then the values are staged
// through shared memory (free once the last flush is done) so that the
// stores run with consecutive threads on consecutive columns.
template <typename Scale, typename Put>
__device__ __forceinline__ void write_tile(unsigned char* smem, const Acc (&acc)[16], Scale&& scale,
                                           Put&& put) {
  double* st = reinterpret_cast<double*>(smem);  // [TM][TN + 1]
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = 32 * (w & 3) + lane, col0 = 16 * (w >> 2);
#pragma unroll
  for (int c = 0; c < 16; ++c) st[row * (TN + 1) + col0 + c] = acc_value(acc[c], scale(row, col0 + c));
  __syncthreads();
  for (int e = threadIdx.x; e < TM * TN; e += OZ_THREADS) {
    const int i = e / TN, j = e % TN;
    put(i, j, st[i * (TN + 1) + j]);
  }
}

__device__ __forceinline__ unsigned long long abs_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}

// ---------------------------------------------------------------------------
// scales: exponent e with max |x| < 2^e (frexp); flag non-finite input
// ---------------------------------------------------------------------------
// One CTA takes 128 columns (blockIdx.y) over a slice of the rows: 64 threads
// along the columns, two columns each, times four along the rows, eight rows in
// flight per thread.  Maxima of |x| as 64-bit integers (the bit patterns of
// non-negative doubles order like their values, NaN above inf): integer
// instructions instead of GB300's slow FP64 ones.
// UPPER: X is upper triangular, and what is stored below its diagonal does not enter.
constexpr int CM_COLS = 128, CM_ROWS = 4, CM_UNROLL = 8;
template <bool VEC, bool UPPER>
__global__ void __launch_bounds__(256) k_col_maxabs(const double* __restrict__ X, int64_t ld, int64_t D, int n,
                                                    double* part, int* bad) {
  __shared__ unsigned long long red[CM_ROWS][CM_COLS];
  const int cx = threadIdx.x & 63, ry = threadIdx.x >> 6;
  const int c = blockIdx.y * CM_COLS + 2 * cx;
  const int64_t per = (D + gridDim.x - 1) / gridDim.x;
  const int64_t r0 = per * blockIdx.x, r1 = min(D, r0 + per);
  const bool two = c + 1 < n;
  unsigned long long m0 = 0, m1 = 0;
  if (c < n) {
    for (int64_t r = r0 + ry; r < r1; r += CM_ROWS * CM_UNROLL) {
      double2 v[CM_UNROLL];
#pragma unroll
      for (int u = 0; u < CM_UNROLL; ++u) {
        const int64_t ru = r + u * CM_ROWS;
        v[u] = make_double2(0.0, 0.0);
        if (ru < r1) {
          const double* p = X + ru * ld + c;
          if (VEC && two) {
            v[u] = __ldg(reinterpret_cast<const double2*>(p));
          } else {
            v[u].x = __ldg(p);
            if (two) v[u].y = __ldg(p + 1);
          }
          if (UPPER && ru > c) v[u].x = 0.0;
          if (UPPER && ru > c + 1) v[u].y = 0.0;
        }
      }
#pragma unroll
      for (int u = 0; u < CM_UNROLL; ++u) {
        m0 = max(m0, abs_bits(v[u].x));
        m1 = max(m1, abs_bits(v[u].y));
      }
    }
  }
  red[ry][2 * cx] = m0;
  red[ry][2 * cx + 1] = m1;
  __syncthreads();
  if (threadIdx.x < CM_COLS) {
    const int cc = blockIdx.y * CM_COLS + threadIdx.x;
    const unsigned long long m = max(max(red[0][threadIdx.x], red[1][threadIdx.x]),
                                     max(red[2][threadIdx.x], red[3][threadIdx.x]));
    if (cc < n) {
      if (m >= 0x7FF0000000000000ull) *bad = 1;  // NaN or inf
      part[(int64_t)blockIdx.x * n + cc] = __longlong_as_double((long long)m);
    }
  }
}
// one warp per column
__global__ void k_col_exp(const double* part, int nb, int n, int* ex) {
  const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (c >= n) return;
  unsigned long long m = 0;
  for (int b = lane; b < nb; b += 32) m = max(m, abs_bits(part[(int64_t)b * n + c]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) {
    int e = 0;
    if (m > 0) frexp(__longlong_as_double((long long)m), &e);
    ex[c] = e;
  }
}

// ---------------------------------------------------------------------------
// digit blocks in HBM
//   column-scaled operand (Gram X or Y, rotation M), w columns over K rows:
//     block (kc, s, cb) of 64 columns x 16 k at ((kc * 8 + s) * ncb + cb) * 1024,
//     so a 128-column A tile is two adjacent blocks (4 KB)
//   row-scaled operand (rotation V), D rows over K = n columns:
//     block (rb, kc, s) of 128 rows x 16 k at ((rb * nkc + kc) * 8 + s) * 2048
// ---------------------------------------------------------------------------
template <bool UPPER>
__global__ void k_digits_cols(const double* __restrict__ X, int64_t ld, int64_t D, int w, int wpad,
                              const int* ex, int64_t nkc, __nv_bfloat16* __restrict__ Xd) {
  const int64_t item = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (item >= nkc * 2 * wpad) return;
  const int c = (int)(item % wpad);
  const int64_t g = item / wpad;  // group of 8 consecutive k
  const int64_t k0 = 8 * g, kc = g >> 1;
  double x[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) x[q] = (c < w && k0 + q < D && !(UPPER && k0 + q > c)) ? X[(k0 + q) * ld + c] : 0.0;
  const int ncb = wpad / 64;
  unsigned char* blk = reinterpret_cast<unsigned char*>(Xd + (kc * 8 * ncb + (c >> 6)) * B_ELEMS);
  const int off = core_offset(c & 63, (int)(k0 & 15));
  cut8(x, c < w ? ex[c] : 0, [&](int s, uint4 v) {
    *reinterpret_cast<uint4*>(blk + (size_t)s * ncb * B_SLICE + off) = v;
  });
}

// Eight rows per CTA: each warp brings one row into shared memory and finds its
// exponent (max |v|, written to er[r]; a non-finite value raises *bad), then eight
// threads side by side cut the same eight columns of the eight rows, so a slice's
// stores are whole core matrices (128 consecutive bytes, 256 with the K-adjacent
// one).  One warp per row storing 16 bytes here and there ran at 40 % of the copy
// bandwidth (2,097,152 x 384: 7.3 ms).  The rows go to `keep` as well (D x ldk, ldk
// even): the product overwrites V, and a wait that gives up must leave V as it was.
constexpr int DR_ROWS = 8;
template <bool VEC>
__global__ void __launch_bounds__(256) k_digits_rows(const double* __restrict__ V, int64_t ldv, int64_t D, int n,
                                                     int64_t Dpad, int npad, int* er, int* bad,
                                                     __nv_bfloat16* __restrict__ Vd, double* __restrict__ keep,
                                                     int64_t ldk) {
  extern __shared__ __align__(16) double rows_sm[];  // 8 x (npad + 2)
  __shared__ int exps[DR_ROWS];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t rb = (int64_t)blockIdx.x * DR_ROWS, r = rb + w;
  const int stride = npad + 2;  // 16 bytes apart in the banks
  double* row = rows_sm + w * stride;
  unsigned long long mb = 0;  // max |v| as integer bits (see k_col_maxabs)
  for (int c = 2 * lane; c < npad; c += 64) {
    double2 v = make_double2(0.0, 0.0);
    if (r < D) {
      const double* p = V + r * ldv + c;
      if (VEC && c + 1 < n) {
        v = __ldg(reinterpret_cast<const double2*>(p));
      } else {
        if (c < n) v.x = __ldg(p);
        if (c + 1 < n) v.y = __ldg(p + 1);
      }
      if (c < n) __stcs(reinterpret_cast<double2*>(keep + r * ldk + c), v);
    }
    mb = max(mb, max(abs_bits(v.x), abs_bits(v.y)));
    *reinterpret_cast<double2*>(row + c) = v;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, o));
  if (lane == 0) {
    if (mb >= 0x7FF0000000000000ull) {  // NaN or inf
      *bad = 1;
      mb = 0;
    }
    int e = 0;
    if (mb > 0) frexp(__longlong_as_double((long long)mb), &e);
    if (r < D) er[r] = e;
    exps[w] = e;
  }
  __syncthreads();
  const int64_t nkc = npad / KS;
  for (int item = threadIdx.x; item < npad; item += 256) {  // npad / 8 column groups x 8 rows
    const int q = item & 7, k0 = (item >> 3) * 8;
    const double* src = rows_sm + q * stride + k0;
    double x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = src[u];
    const int64_t rr = rb + q;
    unsigned char* blk = reinterpret_cast<unsigned char*>(Vd + ((rr >> 7) * nkc + (k0 >> 4)) * 8 * A_ELEMS);
    const int off = core_offset((int)(rr & 127), k0 & 15);
    cut8(x, exps[q], [&](int s, uint4 v) { *reinterpret_cast<uint4*>(blk + (size_t)s * A_SLICE + off) = v; });
  }
}

// ---------------------------------------------------------------------------
// Gram: P[slice][i][j] = sum over the slice's K steps of X[k][i] Y[k][j];
// tile (ti, tj) covers i in [128 ti, +128), j in [64 tj, +64); for a symmetric
// product only the tiles that reach the upper triangle (tj >= 2 ti) run
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(OZ_THREADS, 1)
    k_oz_gram(const __nv_bfloat16* __restrict__ Xd, int ncbx, const __nv_bfloat16* __restrict__ Yd, int ncby,
              int64_t nkc, int m, int n, int ntj, int sym, int64_t kc_per_slice, const int* ex,
              const int* ey, double* __restrict__ P, bool give_up, int* err) {
  extern __shared__ __align__(128) unsigned char smem[];
  int t = blockIdx.x, ti = 0, tj;
  if (sym) {
    for (;;) {
      const int cnt = ntj - 2 * ti;
      if (t < cnt) break;
      t -= cnt;
      ++ti;
    }
    tj = 2 * ti + t;
  } else {
    ti = t / ntj;
    tj = t % ntj;
  }
  const int i0 = ti * TM, j0 = tj * TN;
  const int64_t kc0 = (int64_t)blockIdx.y * kc_per_slice;
  const int nsub = (int)min(kc_per_slice, nkc - kc0);
  uint64_t *full, *empty;
  const uint32_t tmem = tile_setup(smem, &full, &empty);
  Acc acc[16];
#pragma unroll
  for (int c = 0; c < 16; ++c) acc[c] = Acc{0, 0};
  const int64_t a_kc = 8LL * ncbx * B_ELEMS, a_s = (int64_t)ncbx * B_ELEMS;
  const int64_t b_kc = 8LL * ncby * B_ELEMS, b_s = (int64_t)ncby * B_ELEMS;
  const bool ok = run_tile(smem, full, empty, tmem, Xd + kc0 * a_kc + (int64_t)(2 * ti) * B_ELEMS, a_kc, a_s,
                           Yd + kc0 * b_kc + (int64_t)tj * B_ELEMS, b_kc, b_s, nsub, give_up, acc);
  if (!ok) {
    if (threadIdx.x == 0) atomicExch(err, 1);
  } else {
    double* Ps = P + (int64_t)blockIdx.y * m * n;
    write_tile(
        smem, acc,
        [&](int i, int j) {
          const int gi = i0 + i, gj = j0 + j;
          return (gi < m && gj < n) ? ex[gi] + ey[gj] - OZ_UNIT : 0;
        },
        [&](int i, int j, double v) {
          const int gi = i0 + i, gj = j0 + j;
          if (gi < m && gj < n) Ps[(int64_t)gi * n + gj] = v;
        });
  }
  tile_teardown(tmem);
}

__global__ void k_oz_gram_reduce(const double* P, int slices, int m, int n, int sym, double* C,
                                 int ldc) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)m * n) return;
  const int i = (int)(e / n), j = (int)(e % n);
  if (sym && i > j) return;
  double s = 0.0;
  for (int q = 0; q < slices; ++q) s += P[(int64_t)q * m * n + e];
  C[(int64_t)i * ldc + j] = s;
  if (sym && i < j) C[(int64_t)j * ldc + i] = s;
}

// ---------------------------------------------------------------------------
// rotation: Out[r][j] = sum_k V[r][k] M[k][j] from the row-scaled digits of V
// and the column-scaled digits of M; tile (rb, jt) covers rows [128 rb, +128)
// and columns [64 jt, +64).
//
// A tile is short (n / 16 K steps, fewer for a triangular M), so its end weighs as
// much as its products: reading the levels back, rounding to FP64 and storing.  The
// CTAs are persistent (one per SM) and take their tiles' K steps as one stream: the
// bulk copies run on into the next tile, and its first NST K steps are issued as
// soon as the levels have been read, so the tensor core works while the threads
// round and store the previous tile from registers.  The grid is a multiple of the
// tiles of a row block, which therefore run at the same time and share its digits
// in L2, and a CTA moves on by one column tile per row block, so that the lengths
// of a triangular M even out.  2,097,152 x 384, triangular M: 14.2 -> 13.0 ms (one
// CTA per tile, 128-bit integer rounding, stores staged in the ring -> this); the
// tensor pipe is active 42 % of the time.
// ---------------------------------------------------------------------------
enum { STORE_8 = 0, STORE_16 = 1, STORE_32 = 2 };  // bytes per store (alignment of Out and its rows)
template <int STORE>
__global__ void __launch_bounds__(OZ_THREADS, 1)
    k_oz_rotate(const __nv_bfloat16* __restrict__ Vd, const __nv_bfloat16* __restrict__ Md, int ncbm,
                int64_t D, int n, int npad, int nrb, int upper, const int* er, const int* em,
                double* __restrict__ Out, int64_t ldo, int give_up_from, int* err) {
  extern __shared__ __align__(128) unsigned char smem[];
  const int njt = npad / TN, per = gridDim.x / njt;  // row blocks in flight
  const int slot = blockIdx.x / njt, col0 = blockIdx.x % njt;
  const int nkc = npad / KS;
  const int64_t a_kc = 8LL * A_ELEMS, a_s = A_ELEMS;
  const int64_t b_kc = 8LL * ncbm * B_ELEMS, b_s = (int64_t)ncbm * B_ELEMS;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto steps = [&](int jt) { return upper ? (jt + 1) * (TN / KS) : nkc; };  // M upper triangular: rows k <= j
  auto next = [&](int jt) { return jt + 1 == njt ? 0 : jt + 1; };
  uint64_t *full, *empty;
  const uint32_t tmem = tile_setup(smem, &full, &empty);
  // producer warp: K step sc of tile (rb, jt) into the stage of stream position g
  auto load = [&](int rb, int jt, int sc, uint32_t g) {
    const int st = (int)(g % NST);
    unsigned char* dst = smem + (size_t)st * STAGE;
    if (lane == 0) mbar_expect_tx(&full[st], STAGE);
    __syncwarp();
    if (lane < 2 * OZ_S) {
      const int s = lane >> 1;
      if (lane & 1)
        bulk_g2s(dst + OZ_S * A_SLICE + s * B_SLICE, Md + (int64_t)jt * B_ELEMS + sc * b_kc + s * b_s, B_SLICE,
                 &full[st]);
      else
        bulk_g2s(dst + s * A_SLICE, Vd + (int64_t)rb * nkc * 8 * A_ELEMS + sc * a_kc + s * a_s, A_SLICE, &full[st]);
    }
  };
  // MMA issuer: the K step at stream position g
  auto issue = [&](int sc, uint32_t g) {
    const int st = (int)(g % NST);
    if (!mbar_wait(&full[st], (g / NST) & 1u)) return false;
    tc_fence_after();
    const uint32_t a0 = smem_u32(smem + (size_t)st * STAGE);
    const uint64_t ad = sdesc(a0), bd = sdesc(a0 + OZ_S * A_SLICE);
    if ((sc % SUBS) == 0) issue_step<true>(tmem, ad, bd);
    else issue_step<false>(tmem, ad, bd);
    umma_commit(&empty[st]);
    return true;
  };
  bool ok = slot < give_up_from;
  // the next K step to load: tile (lrb, ljt), step ls, stream position lg
  int lrb = slot, ljt = col0, ls = 0;
  uint32_t lg = 0;
  auto load_next = [&]() {
    load(lrb, ljt, ls, lg);
    ++lg;
    if (++ls == steps(ljt)) {
      ls = 0;
      lrb += per;
      ljt = next(ljt);
    }
  };
  if (warp == P_THREAD / 32)
    for (int i = 0; i < NST && lrb < nrb; ++i) load_next();
  uint32_t g = 0;  // stream position of the current tile's first K step
  int ahead = 0;   // K steps of the current tile issued already
  int jt = col0;
  for (int rb = slot; rb < nrb; rb += per, jt = next(jt)) {
    const int nsub = steps(jt);
    Acc acc[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) acc[c] = Acc{0, 0};
    for (int sc = 0; sc < nsub; ++sc) {
      const int st = (int)((g + sc) % NST);
      const uint32_t par = ((g + sc) / NST) & 1u;
      if (threadIdx.x == M_THREAD && ok && sc >= ahead) ok = issue(sc, g + sc);
      if (warp == P_THREAD / 32 && ok && lrb < nrb) {
        // the stage is free again once the MMAs of K step sc have completed
        ok = mbar_wait(&empty[st], par);
        if (ok) load_next();
      }
      const bool last = sc == nsub - 1;
      if ((sc % SUBS) == SUBS - 1 || last) {
        // the issuer observes the completion; the others sleep in the barrier
        if (threadIdx.x == M_THREAD && ok) ok = mbar_wait(&empty[st], par);
        if (__syncthreads_or(!ok)) {
          if (threadIdx.x == 0) atomicExch(err, 1);
          drain(smem, full, lg);
          tile_teardown(tmem);
          return;
        }
        tc_fence_after();
        flush(tmem, acc);
        tc_fence_before();
        __syncthreads();
      }
    }
    g += (uint32_t)nsub;
    if (rb + per >= give_up_from) ok = false;  // fd_debug_give_up; in the waits themselves it costs 1.5 %
    // the next tile's first K steps, before this one's results are rounded
    ahead = rb + per < nrb ? min(NST, min(steps(next(jt)), SUBS)) : 0;
    if (threadIdx.x == M_THREAD) {
      tc_fence_after();
      for (int sc = 0; sc < ahead && ok; ++sc) ok = issue(sc, g + sc);
    }
    __syncwarp();
    const int64_t row = (int64_t)rb * TM + 32 * (warp & 3) + lane;
    const int c0 = jt * TN + 16 * (warp >> 2);
    if (row < D && c0 < n) {
      const int e = er[row] - OZ_UNIT;
      double* o = Out + row * ldo + c0;
#pragma unroll
      for (int c = 0; c < 16; c += 4) {
        double v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = acc_value_small(acc[c + u], c0 + c + u < n ? e + __ldg(em + c0 + c + u) : 0);
        if (STORE == STORE_32 && c0 + c + 4 <= n) {
          asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};\n" ::"l"(o + c), "d"(v[0]), "d"(v[1]), "d"(v[2]),
                       "d"(v[3]) : "memory");
        } else if (STORE >= STORE_16 && c0 + c + 4 <= n) {
          *reinterpret_cast<double2*>(o + c) = make_double2(v[0], v[1]);
          *reinterpret_cast<double2*>(o + c + 2) = make_double2(v[2], v[3]);
        } else {
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (c0 + c + u < n) o[c + u] = v[u];
        }
      }
    }
  }
  tile_teardown(tmem);
}

// the failure path in isolation: a barrier nobody arrives on
__global__ void k_wait_unsatisfied(long long limit, int* err) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  __syncthreads();
  const bool ok = mbar_wait(&bar, 0, limit);
  if (__syncthreads_or(!ok) && threadIdx.x == 0) atomicExch(err, 1);
}

// bit d: the shared-memory attribute is set on device d (a function attribute
// is per device; setting it twice is harmless, so racing threads only repeat it)
std::atomic<unsigned long long> attrs_set{0};

fd_status set_attrs(fd_ctx* ctx) {
  const unsigned long long bit = ctx->device < 64 ? 1ull << ctx->device : 0ull;
  if (bit && (attrs_set.load() & bit)) return FD_OK;
  FD_CUDA(ctx, cudaFuncSetAttribute(k_oz_gram, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OZ_SMEM));
  for (auto rot : {k_oz_rotate<STORE_8>, k_oz_rotate<STORE_16>, k_oz_rotate<STORE_32>})
    FD_CUDA(ctx, cudaFuncSetAttribute(rot, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OZ_SMEM));
  const int rows_smem = (int)(sizeof(double) * DR_ROWS * (1024 + 2));
  FD_CUDA(ctx, cudaFuncSetAttribute(k_digits_rows<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, rows_smem));
  FD_CUDA(ctx, cudaFuncSetAttribute(k_digits_rows<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, rows_smem));
  attrs_set.fetch_or(bit);
  return FD_OK;
}

// device error word of the bounded waits: cleared before a launch, read after
fd_status check_wait_flag(fd_ctx* ctx, const int* flag) {
  int h = 0;
  FD_CUDA(ctx, cudaMemcpyAsync(&h, flag, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
  FD_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  if (h) return set_err(ctx, FD_ERR_TIMEOUT, "tensor-core product: a bounded mbarrier wait gave up");
  return FD_OK;
}

// digit workspace; false (no error) if it cannot be allocated: the caller
// then takes the FP64 path
bool digit_workspace(fd_ctx* ctx, const char* name, size_t bytes, __nv_bfloat16** out) {
  void* p = nullptr;
  if (workspace(ctx, name, bytes, &p) != FD_OK) {
    ctx->err.clear();
    return false;
  }
  *out = (__nv_bfloat16*)p;
  return true;
}

// column-scaled digits of a D x w operand (K = D rows, padded to 16; upper: of its
// upper triangle)
fd_status cut_cols(fd_ctx* ctx, const double* X, int64_t ld, int64_t D, int w, const int* ex,
                   __nv_bfloat16* Xd, int64_t nkc, bool upper = false) {
  const int wpad = (int)cdiv(w, TM) * TM;
  const int64_t items = nkc * 2 * wpad;
  auto kernel = upper ? k_digits_cols<true> : k_digits_cols<false>;
  kernel<<<(unsigned)cdiv(items, 256), 256, 0, ctx->stream>>>(X, ld, D, w, wpad, ex, nkc, Xd);
  FD_LAUNCHED(ctx);
  return FD_OK;
}

}  // namespace

// Column exponents of X (n columns over D rows; upper: of its upper triangle);
// non-finite values raise *bad.
static fd_status col_exponents(fd_ctx* ctx, const double* X, int64_t ld, int64_t D, int n, int* ex,
                               int* bad, bool upper = false) {
  // about eight CTAs per SM, at least one unrolled run of rows each
  const int ct = (int)cdiv(n, CM_COLS);
  int nb = (int)std::max<int64_t>(1, std::min<int64_t>(cdiv(8LL * ctx->num_sms, ct), D / (CM_ROWS * CM_UNROLL)));
  void* p;
  if (workspace(ctx, "oz_colmax", sizeof(double) * (size_t)nb * n, &p, true) != FD_OK) {
    ctx->err.clear();
    nb = std::min(nb, 4 * ctx->num_sms);
    FD_TRY(workspace(ctx, "oz_colmax", sizeof(double) * (size_t)nb * n, &p));
  }
  const bool vec = ((uintptr_t)X & 15) == 0 && ld % 2 == 0;
  auto kernel = upper ? vec ? k_col_maxabs<true, true> : k_col_maxabs<false, true>
                      : vec ? k_col_maxabs<true, false> : k_col_maxabs<false, false>;
  kernel<<<dim3(nb, ct), 256, 0, ctx->stream>>>(X, ld, D, n, (double*)p, bad);
  FD_LAUNCHED(ctx);
  k_col_exp<<<(unsigned)cdiv(n, 8), 256, 0, ctx->stream>>>((double*)p, nb, n, ex);
  FD_LAUNCHED(ctx);
  return FD_OK;
}

fd_status oz_gram(fd_ctx* ctx, const double* X, int64_t ldx, const double* Y, int64_t ldy, int64_t D,
                  int m, int n, double* C, int ldc, bool sym, bool* used) {
  *used = false;
  FD_TRY(set_attrs(ctx));
  const bool same = Y == X && ldy == ldx;
  const int64_t nkc = cdiv(D, KS);
  const int ncbx = (int)cdiv(m, TM) * 2, ncby = (int)cdiv(n, TM) * 2;
  __nv_bfloat16 *Xd, *Yd;
  if (!digit_workspace(ctx, "oz_digits_a", sizeof(__nv_bfloat16) * (size_t)nkc * KS * ncbx * 64 * OZ_S, &Xd))
    return FD_OK;
  Yd = Xd;
  if (!same &&
      !digit_workspace(ctx, "oz_digits_b", sizeof(__nv_bfloat16) * (size_t)nkc * KS * ncby * 64 * OZ_S, &Yd))
    return FD_OK;
  void* p;
  FD_TRY(workspace(ctx, "oz_exp", sizeof(int) * ((size_t)m + n + 8), &p));
  int* ex = (int*)p;
  int* ey = ex + m;
  int* bad = ey + n;
  int* err = bad + 1;
  FD_CUDA(ctx, cudaMemsetAsync(bad, 0, 2 * sizeof(int), ctx->stream));
  FD_TRY(col_exponents(ctx, X, ldx, D, m, ex, bad));
  if (!same) FD_TRY(col_exponents(ctx, Y, ldy, D, n, ey, bad));
  else FD_CUDA(ctx, cudaMemcpyAsync(ey, ex, sizeof(int) * n, cudaMemcpyDeviceToDevice, ctx->stream));
  int hbad = 0;
  FD_CUDA(ctx, cudaMemcpyAsync(&hbad, bad, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
  FD_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  if (hbad) return FD_OK;  // non-finite input: the FP64 path propagates it
  FD_TRY(cut_cols(ctx, X, ldx, D, m, ex, Xd, nkc));
  if (!same) FD_TRY(cut_cols(ctx, Y, ldy, D, n, ey, Yd, nkc));
  const int nti = (int)cdiv(m, TM), ntj = (int)cdiv(n, TN);
  int tiles = 0;
  if (sym) {
    for (int ti = 0; ti < nti; ++ti) tiles += std::max(0, ntj - 2 * ti);
  } else {
    tiles = nti * ntj;
  }
  // about four waves of one CTA per SM; at most 2^16 exact chunks per CTA
  int64_t slices = std::max<int64_t>(1, (4LL * ctx->num_sms) / tiles);
  slices = std::min<int64_t>(slices, std::max<int64_t>(1, cdiv(nkc, 4 * SUBS)));
  slices = std::max<int64_t>(slices, cdiv(nkc, OZ_MAX_CHUNKS * SUBS));
  const int64_t kps = cdiv(nkc, slices);
  slices = cdiv(nkc, kps);
  FD_TRY(workspace(ctx, "oz_gram_partial", sizeof(double) * slices * m * n, &p));
  double* P = (double*)p;
  k_oz_gram<<<dim3(tiles, (unsigned)slices), OZ_THREADS, OZ_SMEM, ctx->stream>>>(
      Xd, ncbx, Yd, ncby, nkc, m, n, ntj, sym ? 1 : 0, kps, ex, ey, P,
      ctx->give_up_from >= 0, err);
  FD_LAUNCHED(ctx);
  FD_TRY(check_wait_flag(ctx, err));
  k_oz_gram_reduce<<<(unsigned)cdiv((int64_t)m * n, 256), 256, 0, ctx->stream>>>(P, (int)slices, m, n,
                                                                                sym ? 1 : 0, C, ldc);
  FD_LAUNCHED(ctx);
  *used = true;
  return FD_OK;
}

fd_status oz_rotate(fd_ctx* ctx, double* V, int64_t ldv, int64_t D, int n, const double* M, bool upper,
                    bool* used) {
  *used = false;
  FD_TRY(set_attrs(ctx));
  const int npad = (int)cdiv(n, TN) * TN;  // K of the product, in whole 64-column blocks of M
  const int64_t Dpad = cdiv(D, TM) * TM;
  const int ncbm = (int)cdiv(n, TM) * 2;
  __nv_bfloat16 *Vd, *Md;
  if (!digit_workspace(ctx, "oz_digits_a", sizeof(__nv_bfloat16) * (size_t)Dpad * npad * OZ_S, &Vd))
    return FD_OK;
  if (!digit_workspace(ctx, "oz_digits_m", sizeof(__nv_bfloat16) * (size_t)npad * ncbm * 64 * OZ_S, &Md))
    return FD_OK;
  void* p;
  const int64_t ldk = n + (n & 1);
  if (workspace(ctx, "oz_rot_keep", sizeof(double) * (size_t)D * ldk, &p) != FD_OK) {
    ctx->err.clear();
    return FD_OK;
  }
  double* keep = (double*)p;
  FD_TRY(workspace(ctx, "oz_rot_small", sizeof(int) * ((size_t)n + D + 8), &p));
  int* em = (int*)p;
  int* er = em + n;
  int* bad = er + D;
  int* err = bad + 1;
  FD_CUDA(ctx, cudaMemsetAsync(bad, 0, 2 * sizeof(int), ctx->stream));
  FD_TRY(col_exponents(ctx, M, n, n, n, em, bad, upper));
  FD_TRY(cut_cols(ctx, M, n, n, n, em, Md, npad / KS, upper));
  const size_t rows_smem = sizeof(double) * DR_ROWS * (npad + 2);  // 65.7 KB at the widest, n = 1024
  const bool vec = ((uintptr_t)V & 15) == 0 && (ldv & 1) == 0;
  auto cut_rows = vec ? k_digits_rows<true> : k_digits_rows<false>;
  cut_rows<<<(unsigned)(Dpad / DR_ROWS), 256, rows_smem, ctx->stream>>>(V, ldv, D, n, Dpad, npad, er, bad, Vd, keep, ldk);
  FD_LAUNCHED(ctx);
  int hbad = 0;
  FD_CUDA(ctx, cudaMemcpyAsync(&hbad, bad, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
  FD_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  if (hbad) return FD_OK;  // non-finite input: the FP64 path propagates it
  // V is no longer read (its digits are): the product goes straight into it.  On a
  // timeout V gets its rows back from `keep`.
  static_assert(1024 / KS <= 32 * SUBS, "acc_value_small holds 32 exact chunks");
  const int njt = npad / TN, nrb = (int)(Dpad / TM);
  const unsigned grid = (unsigned)(njt * std::max(1, std::min(nrb, ctx->num_sms / njt)));
  auto rot = ((uintptr_t)V & 31) == 0 && ldv % 4 == 0 ? k_oz_rotate<STORE_32> : vec ? k_oz_rotate<STORE_16> : k_oz_rotate<STORE_8>;
  rot<<<grid, OZ_THREADS, OZ_SMEM, ctx->stream>>>(Vd, Md, ncbm, D, n, npad, nrb, upper ? 1 : 0, er, em, V, ldv,
                                              ctx->give_up_from >= 0 ? ctx->give_up_from : INT_MAX, err);
  FD_LAUNCHED(ctx);
  const fd_status done = check_wait_flag(ctx, err);
  if (done == FD_ERR_TIMEOUT)
    FD_CUDA(ctx, cudaMemcpy2DAsync(V, sizeof(double) * ldv, keep, sizeof(double) * ldk, sizeof(double) * n, D,
                                   cudaMemcpyDeviceToDevice, ctx->stream));
  FD_TRY(done);
  *used = true;
  return FD_OK;
}

}  // namespace fdi

using namespace fdi;

extern "C" fd_status fd_debug_give_up(fd_ctx* ctx, int from_row_block) {
  if (!ctx) return FD_ERR_ARG;
  ctx->err.clear();
  ctx->give_up_from = std::max(from_row_block, -1);
  return FD_OK;
}

extern "C" fd_status fd_check_bounded_wait(fd_ctx* ctx, int limit_us) {
  if (!ctx) return FD_ERR_ARG;
  ctx->err.clear();
  if (limit_us < 1 || limit_us > 10000000) return set_err(ctx, FD_ERR_ARG, "limit_us must be 1 .. 10^7");
  FD_CUDA(ctx, cudaSetDevice(ctx->device));
  int khz = 0;
  FD_CUDA(ctx, cudaDeviceGetAttribute(&khz, cudaDevAttrClockRate, ctx->device));
  void* p;
  FD_TRY(workspace(ctx, "wait_check", sizeof(int), &p));
  int* err = (int*)p;
  FD_CUDA(ctx, cudaMemsetAsync(err, 0, sizeof(int), ctx->stream));
  const long long limit = (long long)limit_us * (khz > 0 ? khz : 2000000) / 1000;
  k_wait_unsatisfied<<<1, 32, 0, ctx->stream>>>(limit, err);
  FD_LAUNCHED(ctx);
  return check_wait_flag(ctx, err);
}
