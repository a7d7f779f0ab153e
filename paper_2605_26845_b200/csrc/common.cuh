// Device-side building blocks shared by the kernels, and what the launchers share.
//
// In the decomposition kernels one warp owns one demand matrix; sets of rows or columns are bit masks of W 32-bit
// words (W = 1 .. 8), one bit per row or column; masks that every lane holds identically are "uniform".
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/moesched.h"

namespace moesched {

constexpr unsigned FULL = 0xffffffffu;
constexpr int INF32 = 0x7fffffff;

// Index checks of the debug build (-DMOESCHED_CHECKED; the stand-in for a memory checker on machines
// where none can be run): every shared- or global-memory index that comes out of the matching state
// (a matched row or column, a path predecessor, a search level) goes through MS_AT(index, limit).
// In the checked build an index outside [0, limit) is counted in a per-file device counter and
// replaced by 0, so that the access stays in bounds and the kernel ends normally; the host reads the sum
// of the counters through moesched_debug_index_faults(). In the normal build MS_AT(i, n) is just (i).
#ifdef MOESCHED_CHECKED
static __device__ unsigned g_index_faults;
__device__ __forceinline__ int checked_index(int i, int n) {
  if ((unsigned)i >= (unsigned)n) {
    atomicAdd(&g_index_faults, 1u);
    return 0;
  }
  return i;
}
#define MS_AT(i, n) ::moesched::checked_index((i), (n))
using FaultReader = unsigned (*)();
void register_fault_reader(FaultReader reader);   // api.cu
static unsigned read_faults_of_this_file() {
  unsigned v = 0;
  if (cudaMemcpyFromSymbol(&v, g_index_faults, sizeof v) != cudaSuccess) return 0xffffffffu;
  return v;
}
static const bool g_fault_reader_registered = (register_fault_reader(&read_faults_of_this_file), true);
#else
#define MS_AT(i, n) (i)
#endif

enum WorkField { WK_SCAN = 0, WK_AUG = 1, WK_TIGHT = 2, WK_SWEEP = 3, WK_LEVEL = 4, WK_ROT = 5, WK_MATCH = 6, WK_SKIP = 7, WK_POP = 8, WK_BATCH = 9 };

// ---- small helpers on register arrays -------------------------------------------------

// Bit access with a run-time index is written as arithmetic over ALL words (never as
// "touch word k if idx/32 == k"), so that the compiler cannot turn it into an indexed
// access that would push the register array into local memory.
// (Two-word masks take a 64-bit path: one wide shift instead of per-word selects.)
__device__ __forceinline__ unsigned long long as64(const unsigned (&m)[2]) {
  return ((unsigned long long)m[1] << 32) | m[0];
}
template <int W>
__device__ __forceinline__ void clear_bit(unsigned (&m)[W], int idx) {
  if constexpr (W == 2) {
    const unsigned long long b = 1ull << idx;
    m[0] &= ~(unsigned)b;
    m[1] &= ~(unsigned)(b >> 32);
    return;
  }
  const unsigned bit = 1u << (idx & 31);
  const int wi = idx >> 5;
#pragma unroll
  for (int k = 0; k < W; ++k) m[k] &= ~(wi == k ? bit : 0u);
}
template <int W>
__device__ __forceinline__ bool any_bit(const unsigned (&m)[W]) {
  unsigned o = 0;
#pragma unroll
  for (int k = 0; k < W; ++k) o |= m[k];
  return o != 0;
}
template <int W>
__device__ __forceinline__ bool intersects(const unsigned (&a)[W], const unsigned (&b)[W]) {
  unsigned o = 0u;
#pragma unroll
  for (int k = 0; k < W; ++k) o |= a[k] & b[k];
  return o != 0u;
}

// Level of the search history (levels 1..level, W words each) that contains row r, 0 if none does. Every row
// belongs to one level only, so lane d can look at level d and a vote finds it.
template <int W>
__device__ __forceinline__ int level_of_row(const unsigned* hist, int level, int r, int lane) {
  int lvl = 0;
  for (int base = 1; base <= level && lvl == 0; base += 32) {
    const int d = base + lane;
    const bool at = d <= level && ((hist[d * W + (r >> 5)] >> (r & 31)) & 1u);
    const unsigned found = __ballot_sync(FULL, at);
    if (found != 0u) lvl = base + __ffs(found) - 1;
  }
  return lvl;
}

// ---- cluster helpers ---------------------------------------------------------------------

__device__ __forceinline__ unsigned cluster_ctarank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// generic address of the same shared-memory offset in CTA `rank` of the cluster
__device__ __forceinline__ int* map_to_cta(int* local_smem_ptr, unsigned rank) {
  unsigned long long out;
  asm volatile("mapa.u64 %0, %1, %2;" : "=l"(out) : "l"((unsigned long long)local_smem_ptr), "r"(rank));
  return reinterpret_cast<int*>(out);
}

__host__ __device__ inline size_t align16(size_t v) { return (v + 15) & ~(size_t)15; }
__device__ __forceinline__ unsigned smem_addr(const void* p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}

// Every warp of a cluster launch passes here exactly once before it returns.
template <bool CLUSTER>
__device__ __forceinline__ void cluster_epilogue() {
  if constexpr (CLUSTER) cluster_sync_all();
}

// One row set of the search history (W words at hist + level * W). The set is uniform and EVERY lane stores
// it (same address, same value: one shared-memory transaction), so that a lane which reads the history later
// reads what it wrote itself, in program order: no warp barrier is needed between the store and the loads (one is before
// the next store there, see peel.cuh). The matching x[] is kept the same way (every lane makes every update). Four
// or eight words go in 16-byte stores, two or six in 8-byte stores (hist is 16-byte aligned).
template <int W>
__device__ __forceinline__ void hist_store(unsigned* hist, int level, const unsigned (&F)[W]) {
  if constexpr (W % 4 == 0) {
#pragma unroll
    for (int q = 0; q < W; q += 4)
      *reinterpret_cast<uint4*>(hist + level * W + q) = make_uint4(F[q], F[q + 1], F[q + 2], F[q + 3]);
  } else if constexpr (W % 2 == 0) {
#pragma unroll
    for (int q = 0; q < W; q += 2) *reinterpret_cast<uint2*>(hist + level * W + q) = make_uint2(F[q], F[q + 1]);
  } else {
#pragma unroll
    for (int w = 0; w < W; ++w) hist[level * W + w] = F[w];
  }
}
template <int W>
__device__ __forceinline__ void hist_load(const unsigned* hist, int level, unsigned (&H)[W]) {
  if constexpr (W % 4 == 0) {
#pragma unroll
    for (int q = 0; q < W; q += 4) {
      const uint4 v = *reinterpret_cast<const uint4*>(hist + level * W + q);
      H[q] = v.x;
      H[q + 1] = v.y;
      H[q + 2] = v.z;
      H[q + 3] = v.w;
    }
  } else if constexpr (W % 2 == 0) {
#pragma unroll
    for (int q = 0; q < W; q += 2) {
      const uint2 v = *reinterpret_cast<const uint2*>(hist + level * W + q);
      H[q] = v.x;
      H[q + 1] = v.y;
    }
  } else {
#pragma unroll
    for (int w = 0; w < W; ++w) H[w] = hist[level * W + w];
  }
}

// Time of one expert batch of g tokens (see moesched_model_t).
__device__ __forceinline__ long long batch_time_ns(const moesched_model_t& m, long long g) {
  if (g <= 0) return 0;
  const long long beyond = g > m.expert_knee_tokens ? g - m.expert_knee_tokens : 0;
  return m.expert_fixed_ns + (beyond * m.expert_ps_per_token + 999) / 1000;
}

// Division by a divisor fixed for the whole launch (the link speed): floor(x / d) for
// 0 <= x < 2^55 as a multiply-high and a shift (Granlund-Montgomery: with l = ceil(log2 d) and
// m = ceil(2^(55+l) / d), m*d lies in [2^(55+l), 2^(55+l) + 2^l], which makes the quotient exact
// for every 55-bit x).
struct FastDiv {
  unsigned long long m;
  int sh;
};
inline FastDiv make_fastdiv(long long d) {
  int l = 0;
  while ((1LL << l) < d) ++l;
  const unsigned __int128 num = (unsigned __int128)1 << (55 + l);
  FastDiv f;
  f.m = (unsigned long long)((num + (unsigned __int128)(d - 1)) / (unsigned __int128)d);
  f.sh = 55 + l;
  return f;
}
__device__ __forceinline__ long long fast_div(long long x, const FastDiv& f) {
  const unsigned long long hi = __umul64hi(f.m, (unsigned long long)x);
  const unsigned long long lo = f.m * (unsigned long long)x;
  return (long long)(f.sh >= 64 ? hi >> (f.sh - 64) : (hi << (64 - f.sh)) | (lo >> f.sh));
}

// ---- host-side launch geometry ---------------------------------------------------------------
struct Geometry {
  int cpl;       // columns per lane, 1 .. 8
  int S;         // shared-memory row stride in ints
  bool cluster;  // matrix split over a 2-CTA cluster
  int wpb;       // matrices per CTA
  size_t smem;   // dynamic shared memory per CTA
  int threads_per_cta = 0;   // 0: one warp per matrix
  bool max_shared = false;   // shared memory rather than L1, for kernels that run beside this one
};
Geometry plan_geometry(int N);
constexpr size_t SMEM_LIMIT = 227 * 1024;   // shared memory one CTA may request on sm_100a
int sm_count();   // SMs of the current device (148 on B200), cached per device

cudaError_t run_mw(int B, int N, const int32_t* demand, int k_max, uint8_t* perm, int32_t* dur, int32_t* count,
                   int32_t* residual, int32_t* status, long long* work, cudaStream_t stream);
cudaError_t run_bvn(int B, int N, const int32_t* demand, int k_max, uint8_t* perm, int32_t* coef, int32_t* count,
                    int32_t* aug, int32_t* scratch, int32_t* status, long long* work, cudaStream_t stream);
cudaError_t run_bvn_small(int B, int N, const int32_t* demand, int k_max, uint8_t* perm, int32_t* coef, int32_t* count,
                          int32_t* aug, int32_t* status, cudaStream_t stream);
// row stride (ints) of the global working copy used by the Birkhoff kernel
inline int bvn_scratch_stride(int N) { return (N + 7) / 8 * 8; }
cudaError_t run_eval(int B, int N, const int32_t* demand, int k_stride, const uint8_t* perm, const int32_t* dur,
                     const int32_t* count, const moesched_model_t& model, long long* overlap, long long* serial,
                     long long* idle_ns, long long* idle_tok, long long* unserved, int32_t* status,
                     long long* prefix_overlap, long long* prefix_unserved, cudaStream_t stream, bool jobs = false);
// matching order and budget choice (order_kernel.cu)
cudaError_t run_order(int B, int k_stride, const long long* leg, const long long* comp, const int32_t* count,
                      const int32_t* eval_status, int32_t* order, long long* best_ns, long long* emission_ns,
                      int32_t* rule, int32_t* status, cudaStream_t stream);
cudaError_t run_permute(int B, int N, int k_stride, const uint8_t* perm, const int32_t* dur, const int32_t* order,
                        uint8_t* perm_out, int32_t* dur_out, cudaStream_t stream);
cudaError_t run_best_budget(int B, int k_stride, const int32_t* count, const long long* prefix_overlap,
                            const long long* prefix_unserved, long long price, int32_t* best_k, long long* best_cost,
                            cudaStream_t stream);

// left in status[b] by a kernel that holds 16-bit entries for a matrix that has others (never equal to a final status)
constexpr int CLASS_I32 = 65;

bool model_in_range(const moesched_model_t& m);
cudaError_t run_ideal_a2a(int B, int N, const int32_t* demand, const moesched_model_t& model, long long* comm_ns,
                          long long* makespan_ns, int32_t* status, cudaStream_t stream);

cudaError_t run_sinkhorn(int B, int N, const int32_t* demand, int iters, double smooth, int scale_bits,
                         double* scaled, int32_t* fixed, double* stretch, double* row_err, int32_t* status,
                         cudaStream_t stream);
cudaError_t run_sinkhorn_durations(int B, int k_stride, const int32_t* coef, const int32_t* count,
                                   const double* stretch, int scale_bits, int32_t* dur, cudaStream_t stream);

cudaError_t run_bvn_real(int B, int N, const double* matrix, double tol, int k_max, uint8_t* perm, double* lambda,
                         int32_t* count, double* sum_lambda, double* max_left, double* scratch, int32_t* status,
                         cudaStream_t stream);

// All of an SM's memory that can be shared memory is, while the kernel runs there. (A preference: failing is harmless.)
template <typename Kernel>
void prefer_shared_memory(Kernel kern) {
  if (cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) != cudaSuccess)
    (void)cudaGetLastError();
}

// Dynamic shared memory beyond 48 KB has to be permitted, kernel by kernel and for the whole process. What is permitted is always the
// most there is, whatever this launch needs: a smaller figure would take it away from a launch of the same kernel on another
// thread, between that thread's permission and its launch.
template <typename Kernel>
cudaError_t permit_shared_memory(Kernel kern, size_t smem) {
  return smem > 48 * 1024 ? cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_LIMIT) : cudaSuccess;
}

// Launch helper shared by the three kernels.
template <typename Kernel, typename... Args>
cudaError_t launch_warp_kernel(Kernel kern, const Geometry& ge, int B, cudaStream_t stream, Args... args) {
  if (cudaError_t e = permit_shared_memory(kern, ge.smem); e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(ge.threads_per_cta != 0 ? ge.threads_per_cta : 32 * ge.wpb);
  cfg.dynamicSmemBytes = ge.smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  if (ge.cluster) {
    cfg.gridDim = dim3(2 * B);
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
  } else {
    cfg.gridDim = dim3((B + ge.wpb - 1) / ge.wpb);
  }
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

}  // namespace moesched
