// Birkhoff-von Neumann decomposition of at most SMALL_MAX_N ranks: bitmaps over all sets of columns (small.cuh) in place of
// the searches of peel.cuh. One warp per matrix, lane c owns column c.
#include "small.cuh"

namespace moesched {

// The matrix lies in shared memory, no more of it than the warps of the CTA need: with a fixed 4 KB a CTA, for one warp or for four, the
// CTAs of a thousand matrices took a division of the SMs' memory beside which no greedy CTA could start, and a step of greedy
// and Birkhoff became as long as one after the other (paths run one after another, 800 matrices of 8 ranks 91 us, now 45; by searches 51).
// Up to three ranks it is in registers (1000 of 3 ranks 22.5 -> 18.6 us; with more, choosing a register costs more than the load:
// decompositions of 592 matrices of 8 ranks 41 -> 50).
template <int N>
constexpr bool IN_REGISTERS = N <= 3;

template <int N>
__global__ void __launch_bounds__(128) bvn_small_kernel(int B, const int32_t* __restrict__ demand, int k_max,
                                                        uint8_t* __restrict__ perm, int32_t* __restrict__ coef,
                                                        int32_t* __restrict__ count, int32_t* __restrict__ aug,
                                                        int32_t* __restrict__ status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b = blockIdx.x * (blockDim.x >> 5) + warp;
  if (b >= B) return;
  const bool in = lane < N;
  int* A = reinterpret_cast<int*>(smem_raw) + warp * (N * 32) + lane;   // column `lane`, 32 apart

  // ---- the matrix, row and column sums, validation: lane i owns row and column i ----
  const int32_t* D = demand + (size_t)b * N * N;
  int v[N];
  bool neg = false;
  long long csum = 0, rsum = 0;
#pragma unroll
  for (int r = 0; r < N; ++r) v[r] = in ? D[r * N + lane] : 0;
#pragma unroll
  for (int r = 0; r < N; ++r) {
    neg |= v[r] < 0;
    csum += v[r];
    // exact row sum from two 32-bit sums: low and high halves of the entries
    const unsigned lo = __reduce_add_sync(FULL, (unsigned)v[r] & 0xffffu), hi = __reduce_add_sync(FULL, (unsigned)v[r] >> 16);
    if (lane == r) rsum = ((long long)hi << 16) + lo;
  }
  const long long most = max(csum, rsum);
  int st_code = MOESCHED_ST_OK, k = 0;
  if (__any_sync(FULL, neg || most > 2147483647LL)) st_code = MOESCHED_ST_BAD_INPUT;
  if (st_code == MOESCHED_ST_OK) {
    const int T = (int)__reduce_max_sync(FULL, (unsigned)most);
    // ---- north-west-corner padding: deficits as stretches of a line, a cell gets the overlap of its row's and its column's ----
    long long rend = in ? T - rsum : 0, cend = in ? T - csum : 0;
#pragma unroll
    for (int o = 1; o < N; o <<= 1) {
      const long long ur = __shfl_up_sync(FULL, rend, o), uc = __shfl_up_sync(FULL, cend, o);
      if (lane >= o) { rend += ur; cend += uc; }
    }
    unsigned rows = 0u;
    long long r_from = 0;
#pragma unroll
    for (int r = 0; r < N; ++r) {
      const long long r_to = __shfl_sync(FULL, rend, r);
      const long long more = min(r_to, cend) - max(r_from, cend - (T - csum));
      r_from = r_to;
      if (in && more > 0) v[r] += (int)more;
      if (v[r] > 0) rows |= 1u << r;
      if constexpr (!IN_REGISTERS<N>) A[r * 32] = v[r];
      if (aug != nullptr && in) aug[(size_t)b * N * N + r * N + lane] = v[r];
    }

    SmallMatcher<N> m;
    m.begin(lane, rows);
    int left = (int)__reduce_add_sync(FULL, (unsigned)__popc(rows));
    unsigned gone = SmallMatcher<N>::ALL;
    uint8_t* pout = perm + (size_t)b * k_max * N;
    int32_t* cout_ = coef + (size_t)b * k_max;
    while (left > 0 && k < k_max) {
      if (!m.update(gone, k == 0)) { st_code = MOESCHED_ST_INTERNAL; break; }
      // coefficient = smallest matched entry; subtract it along the matching; what reaches zero leaves the graph
      int* cell = A + MS_AT(m.row, N) * 32;
      int val = v[0];
      if constexpr (IN_REGISTERS<N>) {
#pragma unroll
        for (int r = 1; r < N; ++r) val = m.row == r ? v[r] : val;
      } else {
        val = *cell;
      }
      const int c = (int)__reduce_min_sync(FULL, in ? (unsigned)val : 0x7fffffffu);
      val -= c;
      if constexpr (IN_REGISTERS<N>) {
#pragma unroll
        for (int r = 0; r < N; ++r) v[r] = m.row == r ? val : v[r];
      } else {
        if (in) *cell = val;
      }
      const unsigned lost = in && val == 0 ? 1u << m.row : 0u;
      m.rows &= ~lost;
      gone = __reduce_or_sync(FULL, lost);
      left -= __popc(gone);
      if (in) pout[MS_AT(m.row, N)] = (uint8_t)lane;
      if (lane == 0) cout_[k] = c;
      pout += N;
      ++k;
    }
    if (st_code == MOESCHED_ST_OK && left > 0) st_code = MOESCHED_ST_TRUNCATED;
  }
  if (lane == 0) {
    count[b] = k;
    status[b] = st_code;
  }
}

cudaError_t run_bvn_small(int B, int N, const int32_t* demand, int k_max, uint8_t* perm, int32_t* coef, int32_t* count,
                          int32_t* aug, int32_t* status, cudaStream_t stream) {
  Geometry ge = {};
  ge.wpb = B >= 16 * sm_count() ? 4 : 1;
  static_assert(SMALL_MAX_N == 8, "a kernel for every size");
  switch (N) {
#define MOESCHED_GO(n) \
  case n:                                                                    \
    if (!IN_REGISTERS<n>) ge.smem = (size_t)ge.wpb * n * 32 * sizeof(int);   \
    return launch_warp_kernel(bvn_small_kernel<n>, ge, B, stream, B, demand, k_max, perm, coef, count, aug, status);
    MOESCHED_GO(1) MOESCHED_GO(2) MOESCHED_GO(3) MOESCHED_GO(4) MOESCHED_GO(5) MOESCHED_GO(6) MOESCHED_GO(7) MOESCHED_GO(8)
#undef MOESCHED_GO
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace moesched
