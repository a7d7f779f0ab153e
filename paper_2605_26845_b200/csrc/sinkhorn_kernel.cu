// Sinkhorn-Knopp scaling (the preprocessing paper Sec. 3.1 names for the Birkhoff-von Neumann
// decomposition), IEEE double throughout.
//
// X = D + smooth; one sweep divides every entry by the sum of its row, then every entry by the sum
// of its column (correctly rounded). The sums are defined left to right (rows) and top to bottom
// (columns) with one rounding per operation, so that the result does not depend on how the work
// is spread over threads.
//
// Up to 160 ranks (resident_kernel) a CTA holds one matrix in shared memory, an odd number of doubles to a row, and thread
// t walks row t from the left and column t from the top in turn: neither walk has bank conflicts, and a sweep is two
// walks. The pending column scaling of one sweep is applied while the next one walks the rows.
// What bounds it: the divisions, 2 N^2 a sweep, all N of a walk's step by the same divisor. A walk's divisors come
// with their reciprocals (one per row or column and sweep), and a quotient is made from the reciprocal by two
// residual corrections (P. Markstein, IBM J. Res. Dev. 34, 1990: with y the correctly rounded reciprocal of b, q a
// faithful quotient and r = a - q b, which a fused multiply-add gives exactly, the rounded value of q + r y is the
// correctly rounded a / b; the first correction makes q faithful). Five operations without a branch, eight of them in flight; the
// ordinary division, one at a time, is left for operands near the ends of the exponent range.
// B200, 20 sweeps: 1024 x N = 64 1.09 -> 0.28 ms, 4096 x N = 64 3.27 -> 0.81 ms, 512 x N = 33 0.36 -> 0.09 ms.
//
// Above that (streamed_kernel) one warp has a matrix, in the caller's `scaled` buffer:
//   * a column sum is accumulated by the lane that owns the column (column c: lane c % 32) while
//     the warp walks the rows from the top -- coalesced loads, sequential order;
//   * a row sum is accumulated by the lane that owns the row of the current block of 32 rows: the
//     warp loads 32 x 32 tiles with coalesced row loads into shared memory (row stride 33, no
//     bank conflicts) and every lane then adds its row's 32 entries in order.
// Every arithmetic step uses the round-to-nearest intrinsics, which also keeps the compiler from fusing multiplies and adds
// that are not meant to be.
#include "common.cuh"

namespace moesched {

namespace {

constexpr int SK_TILE = 32 * 33;          // doubles of the tile
constexpr int SK_WARP = SK_TILE + 256;    // plus one row sum per row

// Applies the pending column scaling (entry (r, c) divided by col_div of its column) if HAVE_MUL, writes
// the scaled entries back, and leaves in rsum[r] (shared memory) the sum of row r, left to right.
template <int CPL, bool HAVE_MUL>
__device__ __forceinline__ void row_sums_pass(int N, int lane, double* S, double* tile, const double (&col_div)[CPL],
                                              double* rsum) {
  for (int rb = 0; rb * 32 < N; ++rb) {
    double acc = 0.0;
#pragma unroll
    for (int cb = 0; cb < CPL; ++cb) {
      if (cb * 32 < N) {
        const int c = cb * 32 + lane;
        for (int rr = 0; rr < 32; ++rr) {
          const int r = rb * 32 + rr;
          double v = 0.0;
          if (r < N && c < N) {
            v = S[(size_t)r * N + c];
            if (HAVE_MUL) {
              v = __ddiv_rn(v, col_div[cb]);
              S[(size_t)r * N + c] = v;
            }
          }
          tile[rr * 33 + lane] = v;
        }
        __syncwarp();
        const int lim = min(32, N - cb * 32);
        for (int cc = 0; cc < lim; ++cc) acc = __dadd_rn(acc, tile[lane * 33 + cc]);
        __syncwarp();
      }
    }
    if (rb * 32 + lane < N) rsum[rb * 32 + lane] = acc;
  }
  __syncwarp();
}

// A divisor and its reciprocal; 0 in place of the reciprocal where the quick division must not be used.
__device__ __forceinline__ double2 divisor(double b) {
  const bool ordinary = b > 0x1p-400 && b < 0x1p400;
  return make_double2(b, ordinary ? __drcp_rn(b) : 0.0);
}

// Divides the N entries at x, x + stride, ... by div[0], div[1], ... and returns their sum, first to last.
__device__ __forceinline__ double scale_line(double* x, int stride, int N, const double2* div) {
  constexpr int AT_ONCE = 8;
  constexpr unsigned LOWEST = (1023u - 400u) << 20;   // upper word of 2^-400
  double sum = 0.0;
  int i = 0;
  for (; i + AT_ONCE <= N; i += AT_ONCE) {
    double a[AT_ONCE], q[AT_ONCE];
    bool odd = false;   // an entry below 2^-400 other than zero, or a divisor without a reciprocal
#pragma unroll
    for (int k = 0; k < AT_ONCE; ++k) {
      const double2 d = div[i + k];
      a[k] = x[(i + k) * stride];
      const unsigned hi = (unsigned)__double2hiint(a[k]) | (__double2loint(a[k]) != 0 ? 1u : 0u);
      odd |= hi - 1u < LOWEST - 1u || d.y == 0.0;
      q[k] = __dmul_rn(a[k], d.y);
      q[k] = __fma_rn(__fma_rn(-q[k], d.x, a[k]), d.y, q[k]);
      q[k] = __fma_rn(__fma_rn(-q[k], d.x, a[k]), d.y, q[k]);
    }
    if (odd) {
#pragma unroll 1
      for (int k = 0; k < AT_ONCE; ++k) x[(i + k) * stride] = __ddiv_rn(x[(i + k) * stride], div[i + k].x);
#pragma unroll
      for (int k = 0; k < AT_ONCE; ++k) q[k] = x[(i + k) * stride];
    }
#pragma unroll
    for (int k = 0; k < AT_ONCE; ++k) {
      x[(i + k) * stride] = q[k];
      sum = __dadd_rn(sum, q[k]);
    }
  }
  for (; i < N; ++i) {
    const double q = __ddiv_rn(x[i * stride], div[i].x);
    x[i * stride] = q;
    sum = __dadd_rn(sum, q);
  }
  return sum;
}

__host__ __device__ inline int resident_stride(int N) { return N | 1; }
__host__ __device__ inline size_t resident_smem(int N) {
  return ((size_t)N * resident_stride(N) * 8 + 15 & ~(size_t)15) + (size_t)2 * N * sizeof(double2) + 64 * sizeof(double);
}

}  // namespace

// T: threads, N rounded up to whole warps.
template <int T>
__global__ void __launch_bounds__(T, 1) resident_kernel(int N, const int32_t* __restrict__ demand, int iters, double smooth,
                                                     double scale, double* __restrict__ scaled,
                                                     int32_t* __restrict__ fixed, double* __restrict__ stretch,
                                                     double* __restrict__ row_err, int32_t* __restrict__ status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int b = blockIdx.x, P = resident_stride(N);
  double* X = reinterpret_cast<double*>(smem_raw);
  double2* by_row = reinterpret_cast<double2*>(smem_raw + ((size_t)N * P * 8 + 15 & ~(size_t)15));
  double2* by_col = by_row + N;
  double* part = reinterpret_cast<double*>(by_col + N);   // per warp: distance, stretch
  const int32_t* D = demand + (size_t)b * N * N;
  double* Sout = scaled + (size_t)b * N * N;
  int32_t* Q = fixed + (size_t)b * N * N;

  bool bad = false;
  for (int r = warp; r < N; r += T / 32)
    for (int c = lane; c < N; c += 32) {
      const int d = D[(size_t)r * N + c];
      bad |= d < 0;
      X[r * P + c] = __dadd_rn((double)d, smooth);
    }
  bad = __syncthreads_or(bad);
  double sum = 1.0;
  for (int it = 0; it < iters && !bad; ++it) {
    if (t < N) {
      if (it == 0) {
        sum = 0.0;
        for (int c = 0; c < N; ++c) sum = __dadd_rn(sum, X[t * P + c]);
      } else {
        sum = scale_line(X + t * P, 1, N, by_col);
      }
      by_row[t] = divisor(sum);
    }
    if ((bad = __syncthreads_or(t < N && !(sum > 0.0)))) break;   // a row without mass cannot be scaled
    if (t < N) {
      sum = scale_line(X + t, P, N, by_row);
      by_col[t] = divisor(sum);
    }
    bad = __syncthreads_or(t < N && !(sum > 0.0));
  }
  if (bad) {
    for (int e = t; e < N * N; e += T) { Sout[e] = 0.0; Q[e] = 0; }
    if (t == 0) { stretch[b] = 0.0; row_err[b] = 0.0; status[b] = MOESCHED_ST_BAD_INPUT; }
    return;
  }

  // the last column scaling, the row sums of the result, the fixed-point matrix and the stretch
  double err = 0.0;
  if (t < N) err = fabs(__dadd_rn(scale_line(X + t * P, 1, N, by_col), -1.0));
  __syncthreads();
  // The largest ratio d / q: found by cross multiplication, exact in 64 bits (d < 2^31, q <= 2^25), and divided once. Rounding
  // is monotone and d * scale is exact, so that is the largest of the rounded quotients.
  long long bd = 0, bq = 1;
  bool dropped = false;
  for (int r = warp; r < N; r += T / 32)
    for (int c = lane; c < N; c += 32) {
      const double v = X[r * P + c];
      const int qi = (int)floor(__dadd_rn(__dmul_rn(v, scale), 0.5));
      const int d = D[(size_t)r * N + c];
      Sout[(size_t)r * N + c] = v;
      Q[(size_t)r * N + c] = qi;
      if (d > 0) {
        if (qi <= 0) dropped = true;
        else if (d * bq > bd * qi) { bd = d; bq = qi; }
      }
    }
  double st = __ddiv_rn(__dmul_rn((double)bd, scale), (double)bq);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    err = fmax(err, __shfl_xor_sync(FULL, err, o));
    st = fmax(st, __shfl_xor_sync(FULL, st, o));
  }
  if (lane == 0) { part[2 * warp] = err; part[2 * warp + 1] = st; }
  dropped = __syncthreads_or(dropped);
  if (t == 0) {
    for (int w = 1; w < T / 32; ++w) {
      err = fmax(err, part[2 * w]);
      st = fmax(st, part[2 * w + 1]);
    }
    stretch[b] = st;
    row_err[b] = err;
    status[b] = dropped ? MOESCHED_ST_TRUNCATED : MOESCHED_ST_OK;
  }
}

template <int CPL>
__global__ void __launch_bounds__(128) streamed_kernel(int B, int N, const int32_t* __restrict__ demand, int iters,
                                                       double smooth, double scale, double* __restrict__ scaled,
                                                       int32_t* __restrict__ fixed, double* __restrict__ stretch,
                                                       double* __restrict__ row_err, int32_t* __restrict__ status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b = blockIdx.x * (blockDim.x >> 5) + warp;
  if (b >= B) return;
  double* tile = reinterpret_cast<double*>(smem_raw) + (size_t)warp * SK_WARP;
  double* rsum = tile + SK_TILE;
  const int32_t* D = demand + (size_t)b * N * N;
  double* Sout = scaled + (size_t)b * N * N;
  double* S = Sout;
  int32_t* Q = fixed + (size_t)b * N * N;

  int bad = 0;
  for (int e = lane; e < N * N; e += 32) {
    const int d = D[e];
    bad |= d < 0;
    S[e] = __dadd_rn((double)d, smooth);
  }
  bad = __any_sync(FULL, bad);
  __syncwarp();

  double col_div[CPL];   // column sums of the last column pass: the division by them is still pending
#pragma unroll
  for (int s = 0; s < CPL; ++s) col_div[s] = 1.0;
  for (int it = 0; it < iters && !bad; ++it) {
    if (it == 0) row_sums_pass<CPL, false>(N, lane, S, tile, col_div, rsum);
    else row_sums_pass<CPL, true>(N, lane, S, tile, col_div, rsum);
    // a row without mass cannot be scaled
    int zero = 0;
    for (int r = lane; r < N; r += 32) zero |= !(rsum[r] > 0.0);
    if (__any_sync(FULL, zero)) { bad = 1; break; }
    // divide the rows by their sums and accumulate the column sums from the top
    double csum[CPL];
#pragma unroll
    for (int s = 0; s < CPL; ++s) csum[s] = 0.0;
    for (int r = 0; r < N; ++r) {
      const double rv = rsum[r];
#pragma unroll
      for (int s = 0; s < CPL; ++s) {
        const int c = s * 32 + lane;
        if (c < N) {
          const double v = __ddiv_rn(S[(size_t)r * N + c], rv);
          S[(size_t)r * N + c] = v;
          csum[s] = __dadd_rn(csum[s], v);
        }
      }
    }
    zero = 0;
#pragma unroll
    for (int s = 0; s < CPL; ++s) {
      if (s * 32 + lane < N) zero |= !(csum[s] > 0.0);
      col_div[s] = csum[s];
    }
    if (__any_sync(FULL, zero)) { bad = 1; break; }
    __syncwarp();
  }

  if (bad) {
    __syncwarp();
    for (int e = lane; e < N * N; e += 32) { Sout[e] = 0.0; Q[e] = 0; }
    if (lane == 0) { stretch[b] = 0.0; row_err[b] = 0.0; status[b] = MOESCHED_ST_BAD_INPUT; }
    return;
  }

  // the last column scaling, the row sums of the result, the fixed-point matrix and the stretch
  row_sums_pass<CPL, true>(N, lane, S, tile, col_div, rsum);
  double err = 0.0;
  for (int r = lane; r < N; r += 32) err = fmax(err, fabs(__dadd_rn(rsum[r], -1.0)));
  __syncwarp();
  double st = 0.0;
  int dropped = 0;
  for (int e = lane; e < N * N; e += 32) {
    const double v = S[e];
    const double q = floor(__dadd_rn(__dmul_rn(v, scale), 0.5));
    const int qi = (int)q;
    Q[e] = qi;
    const int d = D[e];
    if (d > 0) {
      if (qi > 0) st = fmax(st, __ddiv_rn(__dmul_rn((double)d, scale), (double)qi));
      else dropped = 1;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    err = fmax(err, __shfl_xor_sync(FULL, err, o));
    st = fmax(st, __shfl_xor_sync(FULL, st, o));
  }
  dropped = __any_sync(FULL, dropped);
  if (lane == 0) {
    stretch[b] = st;
    row_err[b] = err;
    status[b] = dropped ? MOESCHED_ST_TRUNCATED : MOESCHED_ST_OK;
  }
}

__global__ void __launch_bounds__(256) sinkhorn_durations_kernel(int B, int k_stride, const int32_t* __restrict__ coef,
                                                                 const int32_t* __restrict__ count,
                                                                 const double* __restrict__ stretch, double scale,
                                                                 int32_t* __restrict__ dur) {
  const int b = blockIdx.y;
  if (b >= B) return;
  const int K = min(max(count[b], 0), k_stride);
  const double st = stretch[b];
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < K; k += gridDim.x * blockDim.x) {
    const double x = __dmul_rn((double)coef[(size_t)b * k_stride + k], st);
    const double d = ceil(__ddiv_rn(x, scale));
    dur[(size_t)b * k_stride + k] = d >= 2147483647.0 ? 2147483647 : (d > 0.0 ? (int)d : 0);
  }
}

// ---- host side ---------------------------------------------------------------------------

cudaError_t run_sinkhorn(int B, int N, const int32_t* demand, int iters, double smooth, int scale_bits,
                         double* scaled, int32_t* fixed, double* stretch, double* row_err, int32_t* status,
                         cudaStream_t stream) {
  const double scale = (double)(1 << scale_bits);
#define MOESCHED_GO(KERNEL, GRID, THREADS, SMEM, ...)                                                               \
  do {                                                                                                              \
    if (cudaError_t e = permit_shared_memory(KERNEL, SMEM); e != cudaSuccess) return e;                             \
    KERNEL<<<GRID, THREADS, SMEM, stream>>>(__VA_ARGS__ N, demand, iters, smooth, scale, scaled, fixed, stretch,    \
                                            row_err, status);                                                       \
    return cudaGetLastError();                                                                                      \
  } while (0)
  const size_t smem = resident_smem(N);
  if (N <= 160) {   // 207 KB
    if (N <= 32) MOESCHED_GO(resident_kernel<32>, B, 32, smem, );
    if (N <= 64) MOESCHED_GO(resident_kernel<64>, B, 64, smem, );
    if (N <= 96) MOESCHED_GO(resident_kernel<96>, B, 96, smem, );
    if (N <= 128) MOESCHED_GO(resident_kernel<128>, B, 128, smem, );
    MOESCHED_GO(resident_kernel<160>, B, 160, smem, );
  }
  constexpr int WPB = 4;
  constexpr size_t TILES = WPB * SK_WARP * sizeof(double);
  MOESCHED_GO(streamed_kernel<8>, (B + WPB - 1) / WPB, 32 * WPB, TILES, B, );
#undef MOESCHED_GO
}

cudaError_t run_sinkhorn_durations(int B, int k_stride, const int32_t* coef, const int32_t* count,
                                   const double* stretch, int scale_bits, int32_t* dur, cudaStream_t stream) {
  const double scale = (double)(1 << scale_bits);
  // B up to 65535 rows of the grid per launch
  for (int b0 = 0; b0 < B; b0 += 65535) {
    const int nb = min(65535, B - b0);
    dim3 grid((k_stride + 255) / 256 > 64 ? 64 : (k_stride + 255) / 256, nb);
    sinkhorn_durations_kernel<<<grid, 256, 0, stream>>>(nb, k_stride, coef + (size_t)b0 * k_stride, count + b0,
                                                        stretch + b0, scale, dur + (size_t)b0 * k_stride);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace moesched
