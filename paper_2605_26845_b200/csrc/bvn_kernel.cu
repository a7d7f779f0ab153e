// Birkhoff-von Neumann decomposition (paper Sec. 3.1), one warp per demand matrix.
//
// The matrix is balanced by north-west-corner padding, then peeled: after each subtraction the rows whose
// matched entry reached zero are re-matched and the lexicographically smallest perfect matching is restored
// (Peeler in peel.cuh).
//
// What bounds it: a dependent chain of searches, about 1100 instructions per matching at N = 64. A full GPU (4096
// matrices of 64 ranks) issues 2.4 instructions per cycle and SM, 70 % of the integer pipe; with one warp per scheduler
// or less the time is the chain's latency (3.3 cycles per instruction). Against one row set per column with an
// OR-reduction per word of every search level, B200: 4096 x N = 64 37.7 -> 25.5 ms, 1024 x N = 128 244 -> 122 ms,
// 256 x N = 256 1152 -> 493 ms (that was with a CTA of eight warps per matrix), one N = 64 12.9 -> 7.2 ms.
// (Warps that slept while they were ahead of the others on their scheduler gained 4 % when a matching took 1700
// instructions; now a full GPU takes the same time with and without it. A team of two, four or eight warps per matrix that
// exchanges its votes through shared memory is slower at every size, however few the matrices: 148 of 256 ranks, 1200
// matchings, 20.7 -> 28.1, 25.2, 29.3 ms; three of 100 ranks 39.9 -> 57 ms with two. Every warp has to repeat the arithmetic
// on whole sets, and a barrier per vote costs more than the divided tests save.)
#include "peel.cuh"
#include "small.cuh"

namespace moesched {

// MODE 0: matrix in this CTA's shared memory; 1: split over a 2-CTA cluster; 2: working copy
// in global memory (scratch), which leaves room for many more warps per SM.
// COUNT: the per-matrix work counters are wanted (they are plain register increments that the
// compiler drops, registers included, when nothing reads them).
//
// The north-west-corner fill needs no walk: with the deficits of the rows and of the columns laid end to end along one
// line, cell (i, j) gets the overlap of row i's stretch and column j's, so a row's cells are found by its own lanes
// from two prefix sums while the row is copied (the walk, one cell after the other through memory, was most of the
// set-up).
template <int W, int MODE, bool COUNT>
__global__ void __launch_bounds__(128, W <= 2 ? 7 : 0) bvn_kernel(int B, int N, int S, const int32_t* __restrict__ demand, int k_max,
                                                  uint8_t* __restrict__ perm, int32_t* __restrict__ coef,
                                                  int32_t* __restrict__ count, int32_t* __restrict__ aug,
                                                  int32_t* scratch, int32_t* __restrict__ status,
                                                  long long* __restrict__ work_out) {
  constexpr bool CLUSTER = MODE == 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b = CLUSTER ? (int)(blockIdx.x >> 1) : (int)(blockIdx.x * (blockDim.x >> 5) + warp);
  if (b >= B) return;   // (a cluster grid has exactly two CTAs per matrix)
  PeelMatrix<int, CLUSTER> mem;
  mem.S = S;
  mem.split = CLUSTER ? (N + 1) / 2 : N;
  unsigned char* base = smem_raw;
  if constexpr (MODE == 2) {
    base += (size_t)warp * peel_smem_bytes(N, W);
    mem.near_ = mem.far_ = scratch + (size_t)b * N * S;
  } else {
    base += (size_t)warp * (peel_smem_bytes(N, W) + align16((size_t)mem.split * S * 4));
    mem.near_ = mem.far_ = reinterpret_cast<int*>(base + peel_smem_bytes(N, W));
  }
  if constexpr (CLUSTER) {
    mem.far_ = map_to_cta(mem.near_, 1);
    cluster_sync_all();
    if (cluster_ctarank() != 0) { cluster_epilogue<true>(); return; }   // lends its shared memory until the end
  }

  unsigned work[MOESCHED_WORK_FIELDS];
#pragma unroll
  for (int q = 0; q < MOESCHED_WORK_FIELDS; ++q) work[q] = 0u;

  // ---- row and column sums, validation: lane c of slot s owns row and column s * 32 + c ----
  const int32_t* D = demand + (size_t)b * N * N;
  long long csum[W], rsum[W];
#pragma unroll
  for (int s = 0; s < W; ++s) csum[s] = rsum[s] = 0;
  int neg = 0;
#pragma unroll
  for (int w = 0; w < W; ++w) {
#pragma unroll 4
    for (int q = 0; q < 32; ++q) {
      const int r = w * 32 + q;
      if (r >= N) break;
      unsigned lo = 0u, hi = 0u;   // exact row sum from two 32-bit sums: low and high halves of the entries
#pragma unroll
      for (int s = 0; s < W; ++s) {
        const int v = s * 32 + lane < N ? D[(size_t)r * N + s * 32 + lane] : 0;
        neg |= v < 0;
        csum[s] += v;
        lo += (unsigned)v & 0xffffu;
        hi += (unsigned)v >> 16;
      }
      lo = __reduce_add_sync(FULL, lo);
      hi = __reduce_add_sync(FULL, hi);
      if (lane == q) rsum[w] = ((long long)hi << 16) + lo;
    }
  }
  neg = __any_sync(FULL, neg);
  long long T = 0;
#pragma unroll
  for (int s = 0; s < W; ++s) T = max(T, max(csum[s], rsum[s]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) T = max(T, __shfl_xor_sync(FULL, T, o));
  int st_code = neg || T > 2147483647LL ? MOESCHED_ST_BAD_INPUT : MOESCHED_ST_OK;
  int k = 0;

  if (st_code == MOESCHED_ST_OK) {
    // ---- deficits as stretches of a line: row r covers [rend - its deficit, rend), and the columns likewise ----
    long long rend[W], cend[W];
    {
      long long rcarry = 0, ccarry = 0;
#pragma unroll
      for (int s = 0; s < W; ++s) {
        const bool in = s * 32 + lane < N;
        long long r = in ? T - rsum[s] : 0, c = in ? T - csum[s] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const long long ur = __shfl_up_sync(FULL, r, o), uc = __shfl_up_sync(FULL, c, o);
          if (lane >= o) { r += ur; c += uc; }
        }
        rend[s] = r + rcarry;
        cend[s] = c + ccarry;
        rcarry = __shfl_sync(FULL, rend[s], 31);
        ccarry = __shfl_sync(FULL, cend[s], 31);
      }
    }

    // ---- working copy, support graph: row r starts out, nominally, at position r ----
    Peeler<W, int, CLUSTER> pl;
    pl.mem = mem;
    pl.reset(base, N, lane);
    int nnz = 0;
    {
      int32_t* ao = aug != nullptr ? aug + (size_t)b * N * N : nullptr;
      long long r_from = 0;
#pragma unroll
      for (int w = 0; w < W; ++w) {
        for (int q = 0; q < 32; ++q) {
          const int r = w * 32 + q;
          if (r >= N) break;
          const long long r_to = __shfl_sync(FULL, rend[w], q);
          PosEntry<W> e;
          e.row8 = (unsigned)r << 8;
#pragma unroll
          for (int s = 0; s < W; ++s) {
            const int c = s * 32 + lane;
            int v = 0;
            if (c < N) {
              v = D[(size_t)r * N + c];
              const long long more = min(r_to, cend[s]) - max(r_from, cend[s] - (T - csum[s]));
              if (more > 0) v += (int)more;
              *mem.cell(r, c) = v;
              if (ao != nullptr) ao[(size_t)r * N + c] = v;
            }
            e.a[s] = __ballot_sync(FULL, v > 0);
            nnz += __popc(e.a[s]);
          }
          pl.seat(r, e);
          r_from = r_to;
        }
      }
    }
    __syncwarp();

    uint8_t* pout = perm + (size_t)b * k_max * N;
    int32_t* cout_ = coef + (size_t)b * k_max;
    while (nnz > 0 && k < k_max) {
      unsigned lo8 = (unsigned)N << 8;   // rows below lo8 >> 8 have their final column
      if (!pl.repair(lo8, work)) { st_code = MOESCHED_ST_INTERNAL; break; }
      if (k == 0) lo8 = 0u;
      work[WK_SKIP] += lo8 >> 8;
      pl.canonicalise(lo8, work);
      pl.fetch_values();

      // coefficient = smallest matched entry; subtract it along the matching; what reaches zero leaves the graph
      int cmin = INF32;
#pragma unroll
      for (int s = 0; s < W; ++s)
        if (pl.valid(s)) cmin = min(cmin, pl.val[s]);
      cmin = __reduce_min_sync(FULL, cmin);
      unsigned zero = 0u;
#pragma unroll
      for (int s = 0; s < W; ++s) {
        pl.val[s] -= cmin;
        if (pl.valid(s)) {
          if (pl.val[s] == 0) zero |= 1u << s;
          pout[MS_AT((int)(pl.key[s] >> 8), N)] = (uint8_t)(s * 32 + lane);
        }
      }
      nnz -= pl.drop_edges(zero);
      if (lane == 0) cout_[k] = cmin;
      pout += N;
      ++k;
      work[WK_MATCH]++;
    }
    if (st_code == MOESCHED_ST_OK && nnz > 0) st_code = MOESCHED_ST_TRUNCATED;
  }

  if (lane == 0) {
    count[b] = k;
    status[b] = st_code;
  }
  if constexpr (COUNT) {
    if (work_out != nullptr && lane == 0) {
#pragma unroll
      for (int q = 0; q < MOESCHED_WORK_FIELDS; ++q) work_out[(size_t)b * MOESCHED_WORK_FIELDS + q] = work[q];
    }
  }
  cluster_epilogue<CLUSTER>();
}

// ---- host side ---------------------------------------------------------------------------

cudaError_t run_bvn(int B, int N, const int32_t* demand, int k_max, uint8_t* perm, int32_t* coef, int32_t* count,
                    int32_t* aug, int32_t* scratch, int32_t* status, long long* work, cudaStream_t stream) {
  // Up to eight ranks bitmaps are faster than searches whatever the batch (small.cuh has both sides; at eight ranks and beyond 10000
  // matrices they are even, 2 % behind at 40000). Work counters count searches, of which that kernel has none: with them it is this one.
  if (N <= SMALL_MAX_N && work == nullptr) return run_bvn_small(B, N, demand, k_max, perm, coef, count, aug, status, stream);
  Geometry ge = plan_geometry(N);
#define MOESCHED_GO(C, M)                                                                                     \
  do {                                                                                                        \
    if (ge.max_shared) prefer_shared_memory(work != nullptr ? bvn_kernel<C, M, true> : bvn_kernel<C, M, false>); \
    if (work != nullptr)                                                                                      \
      return launch_warp_kernel(bvn_kernel<C, M, true>, ge, B, stream, B, N, ge.S, demand, k_max, perm, coef, \
                                count, aug, scratch, status, work);                                       \
    return launch_warp_kernel(bvn_kernel<C, M, false>, ge, B, stream, B, N, ge.S, demand, k_max, perm, coef,  \
                              count, aug, scratch, status, work);                                         \
  } while (0)
  // Without scratch the matrix is held in shared memory, split over a 2-CTA cluster where one CTA cannot hold it. So it is
  // with scratch when the whole batch fits half of the SMs' shared memory that way (the greedy kernel often runs beside):
  // a value that a moved row needs is 30 instead of 300 cycles away (N = 64, 4 matrices per SM: 3 % of the time; below 33
  // ranks there is nothing to be had).
  const size_t held = peel_smem_bytes(N, ge.cpl) + align16((size_t)N * N * 4);
  const bool resident = N > 32 && (size_t)((B + sm_count() - 1) / sm_count()) * (held + 1024) <= SMEM_LIMIT / 2;
  if (scratch != nullptr && !resident) {
    // working copy in global memory: shared memory only for the position table and the search levels
    ge.cluster = false;
    ge.S = bvn_scratch_stride(N);
    // four matrices per CTA once there are enough of them to give every SM several CTAs;
    // a small batch is spread one matrix per CTA so that no SM sits idle
    ge.wpb = B >= 16 * sm_count() ? 4 : 1;
    ge.smem = peel_smem_bytes(N, ge.cpl) * ge.wpb;
    // Left to itself the driver divides an SM's memory for this kernel alone, and a greedy CTA of the same batch (149 KB at 256
    // ranks) does not fit what is left beside a single one of these (18 KB of 164): the greedy part then waits until SMs
    // are empty (whole path, 256 matrices of 256 ranks, 565 -> 646 ms).
    ge.max_shared = ge.cpl == 8;
    switch (ge.cpl) {
      case 1: MOESCHED_GO(1, 2);
      case 2: MOESCHED_GO(2, 2);
      case 3: MOESCHED_GO(3, 2);
      case 4: MOESCHED_GO(4, 2);
      case 5: MOESCHED_GO(5, 2);
      case 6: MOESCHED_GO(6, 2);
      case 7: MOESCHED_GO(7, 2);
      default: MOESCHED_GO(8, 2);
    }
  }
  ge.S = N;
  ge.smem = held;
  ge.cluster = ge.smem > SMEM_LIMIT;
  if (ge.cluster) ge.smem = peel_smem_bytes(N, ge.cpl) + align16((size_t)((N + 1) / 2) * N * 4);
  ge.wpb = !ge.cluster && N <= 32 ? 4 : 1;
  ge.smem *= ge.wpb;
  if (ge.cluster) MOESCHED_GO(8, 1);
  switch (ge.cpl) {
    case 1: MOESCHED_GO(1, 0);
    case 2: MOESCHED_GO(2, 0);
    case 3: MOESCHED_GO(3, 0);
    case 4: MOESCHED_GO(4, 0);
    case 5: MOESCHED_GO(5, 0);
    case 6: MOESCHED_GO(6, 0);
    case 7: MOESCHED_GO(7, 0);
    default: MOESCHED_GO(8, 0);
  }
#undef MOESCHED_GO
}

}  // namespace moesched
