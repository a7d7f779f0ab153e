// Device-side building blocks shared by the kernels in which one warp owns one
// demand matrix: the matrix is held in shared memory (as int32 above 232 ranks it
// is spread over the two CTAs of a thread-block cluster) or in a global working
// copy, and the matching state lives in registers.
//
// Ownership: lane l owns columns (and rows, where a per-row value is kept in
// registers) l*CPL .. l*CPL+CPL-1, CPL = 1, 2, 4 or 8, so that a row scan is one
// vector load per lane. Sets of rows or columns are bit masks of W = CPL 32-bit
// words; masks that every lane holds identically are "uniform".
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
__device__ __forceinline__ void set_bit(unsigned (&m)[W], int idx) {
  if constexpr (W == 2) {
    const unsigned long long b = 1ull << idx;
    m[0] |= (unsigned)b;
    m[1] |= (unsigned)(b >> 32);
    return;
  }
  const unsigned bit = 1u << (idx & 31);
  const int wi = idx >> 5;
#pragma unroll
  for (int k = 0; k < W; ++k) m[k] |= (wi == k ? bit : 0u);
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
// word k of the set {t, t+1, ...}
__device__ __forceinline__ unsigned ge_word(int t, int k) {
  const int lo = k * 32;
  return t <= lo ? 0xffffffffu : (t >= lo + 32 ? 0u : (0xffffffffu << (t - lo)));
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

// ---- the matrix in shared memory --------------------------------------------------------
// Rows [0, split) live in this CTA's shared memory, rows [split, N) in the
// partner CTA of the cluster (far == generic pointer into its shared memory).
// Without a cluster split >= N and far is unused.
struct MatView {
  int* near_;
  int* far_;
  int S;      // row stride in ints, a multiple of CPL
  int split;  // first row held by the partner CTA
  __device__ __forceinline__ int* row(int r) const {
    return r < split ? near_ + r * S : far_ + (r - split) * S;
  }
};

template <int CPL>
struct RowVec {
  int v[CPL];
};

// Vector load of the lane's CPL consecutive columns of one row. The caller
// guarantees lane*CPL < S.
template <int CPL>
__device__ __forceinline__ RowVec<CPL> load_cols(const int* rowp, int lane) {
  RowVec<CPL> r;
  if constexpr (CPL == 1) {
    r.v[0] = rowp[lane];
  } else if constexpr (CPL == 2) {
    int2 t = *reinterpret_cast<const int2*>(rowp + lane * 2);
    r.v[0] = t.x; r.v[1] = t.y;
  } else if constexpr (CPL == 4) {
    int4 t = *reinterpret_cast<const int4*>(rowp + lane * 4);
    r.v[0] = t.x; r.v[1] = t.y; r.v[2] = t.z; r.v[3] = t.w;
  } else {
    int4 t = *reinterpret_cast<const int4*>(rowp + lane * 8);
    int4 q = *reinterpret_cast<const int4*>(rowp + lane * 8 + 4);
    r.v[0] = t.x; r.v[1] = t.y; r.v[2] = t.z; r.v[3] = t.w;
    r.v[4] = q.x; r.v[5] = q.y; r.v[6] = q.z; r.v[7] = q.w;
  }
  return r;
}

// The same matrix held as 16-bit entries (all values <= 65535): half the shared memory per
// matrix, hence twice the matrices per SM for the kernels that shared memory limits.
struct MatView16 {
  unsigned short* base;
  int S;   // row stride in entries, a multiple of CPL
  __device__ __forceinline__ unsigned short* row(int r) const { return base + r * S; }
};

template <int CPL>
__device__ __forceinline__ RowVec<CPL> load_cols(const unsigned short* rowp, int lane) {
  RowVec<CPL> r;
  if constexpr (CPL == 1) {
    r.v[0] = rowp[lane];
  } else if constexpr (CPL == 2) {
    const unsigned t = *reinterpret_cast<const unsigned*>(rowp + lane * 2);
    r.v[0] = t & 0xffffu; r.v[1] = t >> 16;
  } else if constexpr (CPL == 4) {
    const uint2 t = *reinterpret_cast<const uint2*>(rowp + lane * 4);
    r.v[0] = t.x & 0xffffu; r.v[1] = t.x >> 16; r.v[2] = t.y & 0xffffu; r.v[3] = t.y >> 16;
  } else {
    const uint4 t = *reinterpret_cast<const uint4*>(rowp + lane * 8);
    r.v[0] = t.x & 0xffffu; r.v[1] = t.x >> 16; r.v[2] = t.y & 0xffffu; r.v[3] = t.y >> 16;
    r.v[4] = t.z & 0xffffu; r.v[5] = t.z >> 16; r.v[6] = t.w & 0xffffu; r.v[7] = t.w >> 16;
  }
  return r;
}

// ---- bulk asynchronous copy global -> shared with an mbarrier ---------------------------

__device__ __forceinline__ unsigned smem_addr(const void* p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}

// Issued by one lane. bytes is a multiple of 16, both addresses 16-byte aligned,
// bytes < 2^20 (transaction-count range of an mbarrier phase).
__device__ __forceinline__ void bulk_load_issue(void* smem_dst, const void* gmem_src, unsigned bytes,
                                                unsigned long long* mbar) {
  unsigned bar = smem_addr(mbar);
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar));
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_addr(smem_dst)),
      "l"(gmem_src), "r"(bytes), "r"(bar)
      : "memory");
}

// All lanes wait for phase 0 of the barrier. The wait is bounded: false means
// the copy did not land within the limit (never observed; reported, not spun on).
__device__ __forceinline__ bool bulk_load_wait(unsigned long long* mbar) {
  unsigned bar = smem_addr(mbar);
  for (int it = 0; it < (1 << 22); ++it) {
    unsigned done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar)
        : "memory");
    if (done) return true;
  }
  return false;
}

// The same barrier used for a SERIES of bulk copies into one staging buffer: initialised once, armed and
// waited for once per copy (the phase parity alternates), invalidated before its memory is used for
// anything else.
__device__ __forceinline__ void mbar_init(unsigned long long* mbar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(mbar)));
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_inval(unsigned long long* mbar) {
  asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_addr(mbar)) : "memory");
}
// Issued by one thread. bytes is a multiple of 16, both addresses 16-byte aligned, bytes < 2^20.
__device__ __forceinline__ void mbar_bulk_copy(void* smem_dst, const void* gmem_src, unsigned bytes,
                                               unsigned long long* mbar) {
  const unsigned bar = smem_addr(mbar);
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_addr(smem_dst)),
      "l"(gmem_src), "r"(bytes), "r"(bar)
      : "memory");
}
// Bounded wait for the phase with the given parity; false if the copy did not land within the limit.
__device__ __forceinline__ bool mbar_wait(unsigned long long* mbar, unsigned parity) {
  const unsigned bar = smem_addr(mbar);
  for (int it = 0; it < (1 << 22); ++it) {
    unsigned done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}
// Rows per staged copy: as many whole rows of N int32 as fit `stage_bytes`, such that every copy is a
// multiple of 16 bytes; 0 when the matrix cannot be staged (odd N, misaligned source, no room for a row).
__device__ __forceinline__ int staged_rows(const int32_t* src, int N, size_t stage_bytes) {
  if ((N & 1) || (reinterpret_cast<uintptr_t>(src) & 15)) return 0;
  int rows = (int)(stage_bytes / ((size_t)N * 4));
  if (N & 3) rows &= ~1;   // N = 2 mod 4: an even number of rows makes a multiple of 16 bytes
  return rows;
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

// ---- load one matrix into shared memory (one warp) ----------------------------------------
// Copies rows [r0, r1) of the N x N matrix at g into dst with row stride S.
// Returns false if the bounded wait of the bulk copy ran out.
__device__ __forceinline__ bool load_rows(int* dst, const int32_t* g, int N, int S, int r0, int r1, int lane,
                                          unsigned long long* mbar) {
  const int rows = r1 - r0;
  if (rows <= 0) return true;
  const size_t bytes = (size_t)rows * N * 4;
  const int32_t* src = g + (size_t)r0 * N;
  const bool bulk = (S == N) && (bytes % 16 == 0) && ((reinterpret_cast<uintptr_t>(src) & 15) == 0) &&
                    bytes < (1u << 20);
  if (bulk) {
    if (lane == 0) bulk_load_issue(dst, src, (unsigned)bytes, mbar);
    __syncwarp();
    return bulk_load_wait(mbar);
  }
  for (int r = 0; r < rows; ++r)
    for (int c = lane; c < S; c += 32) dst[r * S + c] = c < N ? src[(size_t)r * N + c] : 0;
  __syncwarp();
  return true;
}

// ---- per-warp set-up shared by the kernels ----------------------------------------------------
// Shared memory of one warp: [matrix rows held here][hist: (N+1)*W words of search levels][x: N shorts][mbarrier][flag].
// In cluster mode the grid has two CTAs (one warp each) per matrix: CTA 0 of the pair
// works, CTA 1 loads rows [split, N) into its own shared memory and then only keeps
// them available to CTA 0 (distributed shared memory) until the final cluster barrier.
struct WarpCtx {
  int b;          // matrix index
  int lane;
  MatView M;
  unsigned* hist;
  short* x;
  bool loaded;    // the matrix arrived in shared memory
  bool worker;    // false: this warp has nothing more to do (return after cluster_epilogue)
};

__host__ __device__ inline size_t align16(size_t v) { return (v + 15) & ~(size_t)15; }
__host__ __device__ inline size_t hist_bytes_for(int N, int W) { return align16((size_t)(N + 1) * W * 4); }
__host__ __device__ inline size_t warp_smem_bytes(int N, int S, int W, bool cluster) {
  const int rows_here = cluster ? (N + 1) / 2 : N;
  return align16((size_t)rows_here * S * 4) + hist_bytes_for(N, W) + align16((size_t)N * 2) + 16;
}

template <int CPL, bool CLUSTER>
__device__ __forceinline__ WarpCtx warp_prologue(int B, int N, int S, const int32_t* demand,
                                                 unsigned char* smem_raw) {
  WarpCtx cx;
  cx.lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int wpb = blockDim.x >> 5;
  const int split = CLUSTER ? (N + 1) / 2 : N;
  const int rows_here = CLUSTER ? split : N;
  const size_t mat_bytes = align16((size_t)rows_here * S * 4);
  const size_t hist_bytes = hist_bytes_for(N, CPL);
  const size_t x_bytes = align16((size_t)N * 2);
  unsigned char* base = smem_raw + (size_t)warp * warp_smem_bytes(N, S, CPL, CLUSTER);
  int* mat = reinterpret_cast<int*>(base);
  cx.hist = reinterpret_cast<unsigned*>(base + mat_bytes);
  cx.x = reinterpret_cast<short*>(base + mat_bytes + hist_bytes);
  unsigned long long* mbar = reinterpret_cast<unsigned long long*>(base + mat_bytes + hist_bytes + x_bytes);
  int* peer_flag = reinterpret_cast<int*>(mbar + 1);
  cx.M.near_ = mat;
  cx.M.far_ = mat;
  cx.M.S = S;
  cx.M.split = split;
  cx.worker = true;
  cx.loaded = true;
  if constexpr (CLUSTER) {
    const unsigned crank = cluster_ctarank();
    cx.b = blockIdx.x >> 1;   // grid = 2 B, so always < B
    const int32_t* g = demand + (size_t)cx.b * N * N;
    if (crank == 0) cx.loaded = load_rows(mat, g, N, S, 0, split, cx.lane, mbar);
    else cx.loaded = load_rows(mat, g, N, S, split, N, cx.lane, mbar);
    if (cx.lane == 0) *peer_flag = cx.loaded ? 1 : 0;
    cx.M.far_ = map_to_cta(mat, 1);
    cluster_sync_all();
    if (crank != 0) cx.worker = false;
    else cx.loaded = cx.loaded && (*map_to_cta(peer_flag, 1) != 0);
  } else {
    cx.b = blockIdx.x * wpb + warp;
    if (cx.b >= B) { cx.worker = false; return cx; }
    cx.loaded = load_rows(mat, demand + (size_t)cx.b * N * N, N, S, 0, N, cx.lane, mbar);
  }
  return cx;
}

// One warp: rows of N int32 arrive in `stage` by bulk copies of rows_per_copy rows each and are narrowed to
// 16 bits into dst (row stride S, padding columns zeroed). Kept out of line so that its registers do not
// count against the kernel that calls it once. Returns false if a copy did not land within its bounded wait.
static __device__ __noinline__ bool stage_and_narrow(const int32_t* src, int N, int S, int rows_per_copy, int lane,
                                              unsigned short* dst, int* stage, unsigned long long* mbar) {
  if (lane == 0) mbar_init(mbar);
  __syncwarp();
  unsigned parity = 0;
  bool ok = true;
  for (int r0 = 0; r0 < N; r0 += rows_per_copy) {
    const int rows = min(rows_per_copy, N - r0);
    if (lane == 0) mbar_bulk_copy(stage, src + (size_t)r0 * N, (unsigned)(rows * N * 4), mbar);
    __syncwarp();
    if (!mbar_wait(mbar, parity)) {
      mbar_wait(mbar, parity);   // one more bounded wait for the copy in flight before giving up
      ok = false;
      break;
    }
    parity ^= 1u;
    for (int r = 0; r < rows; ++r)
      for (int c = lane; c < S; c += 32)
        dst[(r0 + r) * S + c] = c < N ? (unsigned short)stage[r * N + c] : (unsigned short)0;
    __syncwarp();   // the staging rows are free again
  }
  if (ok && lane == 0) mbar_inval(mbar);
  __syncwarp();
  return ok;
}

// Variant for matrices whose entries all fit 16 bits: the warp's shared memory is
// [N x S entries of 16 bits][hist][x]; the entries are narrowed while they are loaded.
__host__ __device__ inline size_t warp_smem_bytes16(int N, int S, int W) {
  return align16((size_t)N * S * 2) + hist_bytes_for(N, W) + align16((size_t)N * 2);
}

struct WarpCtx16 {
  int b;
  int lane;
  MatView16 M;
  unsigned* hist;
  short* x;
  bool worker;
  bool loaded;    // false: a bulk copy did not land within its bounded wait
};

// STAGED: the rows come in by bulk asynchronous copies and are narrowed from a staging area (scoring, whose
// short launches are dominated by the load); otherwise plain coalesced loads narrow on the fly (greedy: with
// the staged loop in its prologue the compiler gives the whole kernel 128 registers instead of 64, 16
// instead of 22 warps per SM, measured 12.4 ms against 12.1 ms on 4096 matrices of 64 ranks).
template <int CPL, bool STAGED>
__device__ __forceinline__ WarpCtx16 warp_prologue16(int B, int N, int S, const int32_t* demand,
                                                     unsigned char* smem_raw) {
  WarpCtx16 cx;
  cx.lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int wpb = blockDim.x >> 5;
  unsigned char* base = smem_raw + (size_t)warp * warp_smem_bytes16(N, S, CPL);
  const size_t mat_bytes = align16((size_t)N * S * 2);
  cx.M.base = reinterpret_cast<unsigned short*>(base);
  cx.M.S = S;
  cx.hist = reinterpret_cast<unsigned*>(base + mat_bytes);
  cx.x = reinterpret_cast<short*>(base + mat_bytes + hist_bytes_for(N, CPL));
  cx.b = blockIdx.x * wpb + warp;
  cx.worker = cx.b < B;
  cx.loaded = true;
  if (!cx.worker) return cx;
  const int32_t* src = demand + (size_t)cx.b * N * N;
  // The int32 rows come in by bulk asynchronous copies, a few rows at a time, into the memory that will
  // hold the search history later (nothing lives there yet), and are narrowed from there; the barrier of
  // the copies borrows the first bytes of x. Matrices that cannot be staged take plain loads.
  const int rows_per_copy = STAGED ? staged_rows(src, N, hist_bytes_for(N, CPL)) : 0;
  if (STAGED && rows_per_copy > 0) {
    cx.loaded = stage_and_narrow(src, N, S, rows_per_copy, cx.lane, cx.M.base, reinterpret_cast<int*>(cx.hist),
                                 reinterpret_cast<unsigned long long*>(cx.x));
    return cx;
  }
  for (int r = 0; r < N; ++r)
    for (int c = cx.lane; c < S; c += 32)
      cx.M.base[r * S + c] = c < N ? (unsigned short)src[(size_t)r * N + c] : (unsigned short)0;
  __syncwarp();
  return cx;
}

// Every warp of a cluster launch passes here exactly once before it returns.
template <bool CLUSTER>
__device__ __forceinline__ void cluster_epilogue() {
  if constexpr (CLUSTER) cluster_sync_all();
}

// One row set of the search history (W words at hist + level * W). The set is uniform and EVERY lane stores
// it (same address, same value: one shared-memory transaction), so that a lane which reads the history later
// reads what it wrote itself, in program order: no warp barrier is needed between the store and the loads. The
// matching x[] is kept the same way (every lane makes every update). Two words go in one 8-byte store, four
// or eight in 16-byte stores (hist is 16-byte aligned and W * 4 divides 16 or is a multiple of it).
template <int W>
__device__ __forceinline__ void hist_store(unsigned* hist, int level, const unsigned (&F)[W], int /*lane*/) {
  if constexpr (W == 2) {
    *reinterpret_cast<uint2*>(hist + level * 2) = make_uint2(F[0], F[1]);
  } else if constexpr (W % 4 == 0) {
#pragma unroll
    for (int q = 0; q < W; q += 4)
      *reinterpret_cast<uint4*>(hist + level * W + q) = make_uint4(F[q], F[q + 1], F[q + 2], F[q + 3]);
  } else {
#pragma unroll
    for (int w = 0; w < W; ++w) hist[level * W + w] = F[w];
  }
}
template <int W>
__device__ __forceinline__ void hist_load(const unsigned* hist, int level, unsigned (&H)[W]) {
  if constexpr (W == 2) {
    const uint2 v = *reinterpret_cast<const uint2*>(hist + level * 2);
    H[0] = v.x;
    H[1] = v.y;
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
  int cpl;       // columns per lane: 1, 2, 4 or 8
  int S;         // shared-memory row stride in ints
  bool cluster;  // matrix split over a 2-CTA cluster
  int wpb;       // warps (matrices) per CTA
  size_t smem;   // dynamic shared memory per CTA
};
Geometry plan_geometry(int N);
constexpr size_t SMEM_LIMIT = 227 * 1024;   // shared memory one CTA may request on sm_100a
int sm_count();   // SMs of the current device (148 on B200), cached per device

cudaError_t run_mw(int B, int N, const int32_t* demand, int k_max, uint8_t* perm, int32_t* dur, int32_t* count,
                   int32_t* residual, int32_t* status, long long* work, cudaStream_t stream);
cudaError_t run_bvn(int B, int N, const int32_t* demand, int k_max, uint8_t* perm, int32_t* coef, int32_t* count,
                    int32_t* aug, int32_t* scratch, int32_t* status, long long* work, cudaStream_t stream);
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

// scoring with one CTA per matrix, for the matrices whose status holds CLASS_U16 (64 < N <= 256)
cudaError_t run_eval_team(int B, int N, const int32_t* demand, int k_stride, const uint8_t* perm, const int32_t* dur,
                          const int32_t* count, const moesched_model_t& model, long long* overlap, long long* serial,
                          long long* idle_ns, long long* idle_tok, long long* unserved, int32_t* status,
                          cudaStream_t stream);

// class codes the pre-pass leaves in status[b] (never equal to a final status)
constexpr int CLASS_U16 = 64;
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

// Launch helper shared by the three kernels.
template <typename Kernel, typename... Args>
cudaError_t launch_warp_kernel(Kernel kern, const Geometry& ge, int B, cudaStream_t stream, Args... args) {
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ge.smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(32 * ge.wpb);
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
