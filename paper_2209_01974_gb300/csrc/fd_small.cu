// Launches of the one-kernel filter of small matrices (fd_small.cuh).
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>

#include "fd_internal.cuh"
#include "fd_small.cuh"

namespace fdi {
namespace {

using namespace small;

constexpr int MAX_THREADS = 1024;

template <typename T>
struct Params {
  Block<T> b;
  int mu0;                                  // first coefficient held
  typename Ops<T>::S mu[MAX_STEPS + 3];
};

template <typename T, int PW, bool CLUSTER>
__global__ void __launch_bounds__(MAX_THREADS, 1) k_filter_small(const __grid_constant__ Params<T> p) {
  extern __shared__ __align__(16) unsigned char sm_smem[];
  uint32_t rank = 0, ranks = 1;
  if (CLUSTER) {
    asm("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(rank));
    asm("mov.u32 %0, %%cluster_nctarank;\n" : "=r"(ranks));
  }
  filter_panel<T, PW, CLUSTER>(p.b, (int)(blockIdx.x / ranks) * PW, rank, ranks, sm_smem,
                               [&](int k) { return p.mu[k - p.mu0]; });
}

template <typename T, int PW, bool CLUSTER>
fd_status launch(fd_ctx* ctx, const Params<T>& p, int units, int cluster, size_t smem, int threads) {
  auto kernel = k_filter_small<T, PW, CLUSTER>;
  // always the same value: threads on other contexts may launch the kernel meanwhile
  FD_CUDA(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ctx->smem_optin));
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)cluster;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(units / PW * cluster));
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = ctx->stream;
  cfg.attrs = attr;
  cfg.numAttrs = CLUSTER ? 1 : 0;
  FD_CUDA(ctx, cudaLaunchKernelEx(&cfg, kernel, p));
  FD_LAUNCHED(ctx);
  return FD_OK;
}

template <typename T, int PW>
fd_status launch_pw(fd_ctx* ctx, const Params<T>& p, int units, int cluster, size_t smem, int threads) {
  if (cluster > 1) return launch<T, PW, true>(ctx, p, units, cluster, smem, threads);
  return launch<T, PW, false>(ctx, p, units, cluster, smem, threads);
}

}  // namespace

// Clusters of a launch that are resident at once (cached per device and size:
// they depend on the chip's groups of SMs, and every CTA here fills most of one)
int resident_clusters(const fd_ctx* ctx, int cluster) {
  static std::atomic<int> cache[64][9];
  if (cluster == 1) return ctx->num_sms;
  std::atomic<int>* slot = ctx->device < 64 ? &cache[ctx->device][cluster] : nullptr;
  if (slot && slot->load()) return slot->load();
  auto kernel = k_filter_small<double, 1, true>;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ctx->smem_optin) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)cluster;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(ctx->num_sms / cluster * cluster));
  cfg.blockDim = dim3(MAX_THREADS);
  cfg.dynamicSmemBytes = ctx->smem_optin / 2 + 4096;  // one CTA per SM
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  if (slot) slot->store(n);
  return n;
}

// Split of a block of `units` 8-byte columns over panels and clusters, and the
// estimated SM clocks of a step.  A CTA's work: its units times the FP64 pipe's
// clocks (2 FMA a clock, at about 60 % with the few warps a CTA has) or, for FP32 and
// float-float, the issue clocks of an entry; in a cluster the stores of its rows to
// the other CTAs (about 16 clocks per warp); plus the barrier and the latency of a
// step (about 1,500 clocks for a cluster, 800 for a single CTA, and 20 to 60 for every
// further entry of a long row, which one thread takes one after the other).
SmallPlan small_plan(const fd_ctx* ctx, const fd_matrix* M, fd_prec prec, int units) {
  SmallPlan best;
  if (M->kron || M->D > MAX_ROWS || M->max_row > MAX_ROWS) return best;
  const double nnz = (double)M->nnz / (double)M->D;
  const double per_unit = prec == FD_F64 ? (nnz + 1.4) / 1.2 : prec == FD_F32 ? (6 * nnz + 30) / 80 : (20 * nnz + 70) / 80;
  const double chain = prec == FD_F32 ? 0.0 : (prec == FD_FF ? 60.0 : 20.0) * std::max(0, M->max_row - 8);
  for (int pw : {1, 2, 4, 8}) {
    if (units % pw) continue;
    for (int cl = 1; cl <= 8; ++cl) {  // 8: the largest portable cluster
      const int R = cta_rows((int)M->D, cl);
      const size_t smem = prec == FD_F32 ? cta_smem<float>((int)M->D, R, pw, M->max_row)
                                         : cta_smem<double>((int)M->D, R, pw, M->max_row);
      if (smem > ctx->smem_optin - 1024) continue;
      const int threads = std::min(MAX_THREADS, (R * pw + 31) & ~31);
      const int per_sm = std::max(1, std::min<int>((int)(ctx->smem_optin / (smem + 1024)), 2048 / threads));
      const int resident = resident_clusters(ctx, cl);
      if (resident < 1) continue;
      const int64_t panels = units / pw;
      const int64_t layers = cdiv(panels, resident);  // CTAs on the fullest SM
      const int64_t waves = cdiv(layers, per_sm);
      double clocks = (double)layers * R * pw * (per_unit + (cl - 1) * 0.5) + (double)waves * ((cl > 1 ? 1500 : 800) + chain);
      if (cl > 1) clocks *= 1.15;  // near ties go to the smaller cluster
      if (best.cluster == 0 || clocks < best.clocks) {
        best.cluster = cl;
        best.pw = pw;
        best.threads = threads;
        best.smem = smem;
        best.clocks = clocks;
      }
    }
  }
  return best;
}

// SM clocks of a launched step over the same columns: the launch and the chain of
// loads (per batch of entries), and the FP64 pipe (nnz + 4 operations) or the issue
// of the entries.  The launch costs less where steps overlap: dependent launches,
// which FP64 grids below a wave do without, and in float-float a grid whose CTAs
// have the registers of one wave.  Fitted to D = 4,096 .. 17,576, 375 filters of stencil,
// Hubbard, road and random matrices with 3 to 100 entries a row: of launched steps and
// panels the faster one is taken, or one within 10 % of it (21 % in FP32 from 2,744 rows
// on one SM, 41 % in FP64 for 4,900 rows of 4 entries with nb = 64).
static double launched_clocks(const fd_ctx* ctx, const fd_matrix* M, fd_prec prec, int units) {
  const double nnz = (double)M->nnz / (double)M->D, elems = (double)M->D * units / ctx->num_sms;
  const double batches = std::ceil(std::min<double>(M->max_row, 2 * nnz) / step::BATCH);
  const int64_t rows = 4 * (32 / std::max(1, std::min(32, units / 2)));  // of a CTA, 8-byte elements
  const int64_t grid = cdiv(M->D, rows);
  if (prec == FD_F64) return (grid >= 8LL * ctx->num_sms ? 6600 : 10600) + 700 * batches + elems * (nnz + 4) / 2;
  if (prec == FD_F32) return 1800 + 1600 * batches + elems * (8 * nnz + 60) / 128;
  return (grid <= 10LL * ctx->num_sms ? 5000 : 9000) + 1400 * batches + elems * (25 * nnz + 130) / 128;
}

bool filter_small_pays(const fd_ctx* ctx, const fd_matrix* M, fd_prec prec, int nb, SmallPlan* chosen) {
  const int units = prec == FD_F32 ? nb / 2 : nb;
  const SmallPlan plan = small_plan(ctx, M, prec, units);
  if (chosen) *chosen = plan;
  return plan.cluster > 0 && plan.clocks < launched_clocks(ctx, M, prec, units);
}

template <typename T>
static fd_status filter_small_t(fd_ctx* ctx, const fd_matrix* M, const SmallPlan& plan, T* V, int64_t ldv, int units, int n,
                         const double* mu, double alpha, double beta, T* W1, T* W2, int64_t ldw) {
  Params<T> p;
  Block<T>& b = p.b;
  b.chunk_ptr = M->chunk_ptr; b.row_len = M->row_len; b.col = M->col; b.val = M->val;
  b.perm = M->identity ? nullptr : M->perm;
  b.D = (int)M->D; b.C = M->C; b.max_row = M->max_row;
  b.V = V; b.ldv = ldv; b.X[0] = W1; b.X[1] = W2; b.ldw = ldw;
  b.a2 = 2 * alpha; b.b2 = 2 * beta;
  b.n = n;
  for (int k0 = 1; k0 <= n; k0 = b.k1 + 1) {
    b.k0 = k0;
    b.k1 = n;
    if (n - k0 >= MAX_STEPS) {  // end where the accumulator is complete: k1 = 2 mod 3
      b.k1 = k0 + MAX_STEPS - 1;
      b.k1 -= (b.k1 - 2) % 3;
    }
    p.mu0 = std::max(0, k0 - 2);
    for (int k = p.mu0; k <= b.k1; ++k) p.mu[k - p.mu0] = Ops<T>::coef(mu[k]);
    switch (plan.pw) {
      case 1: FD_TRY((launch_pw<T, 1>(ctx, p, units, plan.cluster, plan.smem, plan.threads))); break;
      case 2: FD_TRY((launch_pw<T, 2>(ctx, p, units, plan.cluster, plan.smem, plan.threads))); break;
      case 4: FD_TRY((launch_pw<T, 4>(ctx, p, units, plan.cluster, plan.smem, plan.threads))); break;
      default: FD_TRY((launch_pw<T, 8>(ctx, p, units, plan.cluster, plan.smem, plan.threads))); break;
    }
  }
  return FD_OK;
}

fd_status filter_small(fd_ctx* ctx, const fd_matrix* M, fd_prec prec, void* V, int64_t ldv, int nb, int degree,
                       const double* mu, double alpha, double beta, void* W1, void* W2, int64_t ldw,
                       double* bytes_out, bool* used) {
  *used = false;
  SmallPlan plan;
  if (!filter_small_pays(ctx, M, prec, nb, &plan)) return FD_OK;
  const int units = prec == FD_F32 ? nb / 2 : nb;
  if (prec == FD_F64)
    FD_TRY(filter_small_t<double>(ctx, M, plan, (double*)V, ldv, units, degree, mu, alpha, beta, (double*)W1, (double*)W2, ldw));
  else if (prec == FD_FF)
    FD_TRY(filter_small_t<ff>(ctx, M, plan, (ff*)V, ldv, units, degree, mu, alpha, beta, (ff*)W1, (ff*)W2, ldw));
  else
    FD_TRY(filter_small_t<float>(ctx, M, plan, (float*)V, ldv, units, degree, mu, alpha, beta, (float*)W1, (float*)W2, ldw));
  if (bytes_out) *bytes_out += filter_bytes(M, nb, degree, prec == FD_F32 ? 4.0 : 8.0);
  *used = true;
  return FD_OK;
}

}  // namespace fdi
