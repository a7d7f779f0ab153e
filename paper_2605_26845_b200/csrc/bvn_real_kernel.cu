// Birkhoff-von Neumann decomposition of a REAL-valued matrix (paper Sec. 3.1: A = sum_k lambda_k P_k
// for a doubly stochastic A, as obtained from Sinkhorn-Knopp scaling), one warp per matrix.
//
// The combinatorial part is the one of bvn_kernel.cu (peel.cuh: matching, support graph and searches); only the entries
// are doubles, held in a global working copy. Every arithmetic step is one exact
// IEEE operation (a minimum, a subtraction, a comparison with the tolerance) taken in a fixed
// order, so the result is reproducible bit for bit. A scaled matrix is doubly stochastic only up
// to the error of its last sweep: when the support has no perfect matching left the decomposition
// stops and reports what remains.
#include "peel.cuh"

namespace moesched {

namespace {

__device__ __forceinline__ double warp_min_f64(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(FULL, v, o));
  return v;
}
__device__ __forceinline__ double warp_max_f64(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(FULL, v, o));
  return v;
}

}  // namespace

template <int W>
__global__ void __launch_bounds__(128) bvn_real_kernel(int B, int N, int S, const double* __restrict__ matrix, double tol,
                                                       int k_max, uint8_t* __restrict__ perm,
                                                       double* __restrict__ lambda, int32_t* __restrict__ count,
                                                       double* __restrict__ sum_lambda, double* __restrict__ max_left,
                                                       double* scratch, int32_t* __restrict__ status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b = blockIdx.x * (blockDim.x >> 5) + warp;
  if (b >= B) return;
  const double* src = matrix + (size_t)b * N * N;
  Peeler<W, double, false> pl;
  pl.mem.near_ = pl.mem.far_ = scratch + (size_t)b * N * S;
  pl.mem.S = S;
  pl.mem.split = N;
  pl.reset(smem_raw + (size_t)warp * peel_smem_bytes(N, W), N, lane);

  unsigned work[MOESCHED_WORK_FIELDS];   // not reported
#pragma unroll
  for (int q = 0; q < MOESCHED_WORK_FIELDS; ++q) work[q] = 0u;

  // ---- working copy and support graph: entries at or below the tolerance are dropped; negative or NaN entries reject ----
  int bad = 0, nnz = 0;
#pragma unroll
  for (int w = 0; w < W; ++w) {
    for (int q = 0; q < 32; ++q) {
      const int r = w * 32 + q;
      if (r >= N) break;
      PosEntry<W> e;
      e.row8 = (unsigned)r << 8;
#pragma unroll
      for (int s = 0; s < W; ++s) {
        const int c = s * 32 + lane;
        double v = 0.0;
        if (c < N) {
          v = src[(size_t)r * N + c];
          bad |= !(v >= 0.0);
          if (!(v > tol)) v = 0.0;
          *pl.mem.cell(r, c) = v;
        }
        e.a[s] = __ballot_sync(FULL, v > 0.0);
        nnz += __popc(e.a[s]);
      }
      pl.seat(r, e);
    }
  }
  bad = __any_sync(FULL, bad);

  int st_code = bad ? MOESCHED_ST_BAD_INPUT : MOESCHED_ST_OK;
  int k = 0;
  double total = 0.0;

  if (st_code == MOESCHED_ST_OK) {
    uint8_t* pout = perm + (size_t)b * k_max * N;
    double* lout = lambda + (size_t)b * k_max;
    bool exhausted = false;   // the support has no perfect matching any more
    while (nnz > 0 && k < k_max) {
      unsigned lo8 = (unsigned)N << 8;   // rows below lo8 >> 8 have their final column
      if (!pl.repair(lo8, work)) { exhausted = true; break; }
      if (k == 0) lo8 = 0u;
      pl.canonicalise(lo8, work);
      pl.fetch_values();
      // lambda = smallest matched entry; subtract it along the matching; what falls to the tolerance vanishes
      double cmin = 1e300;
#pragma unroll
      for (int s = 0; s < W; ++s)
        if (pl.valid(s)) cmin = fmin(cmin, pl.val[s]);
      cmin = warp_min_f64(cmin);
      unsigned zero = 0u;
#pragma unroll
      for (int s = 0; s < W; ++s) {
        if (pl.valid(s)) {
          double nv = __dsub_rn(pl.val[s], cmin);
          if (!(nv > tol)) { nv = 0.0; zero |= 1u << s; }
          pl.val[s] = nv;
          pout[MS_AT((int)(pl.key[s] >> 8), N)] = (uint8_t)(s * 32 + lane);
        }
      }
      nnz -= pl.drop_edges(zero);
      if (lane == 0) lout[k] = cmin;
      total = __dadd_rn(total, cmin);
      pout += N;
      ++k;
    }
    if (st_code == MOESCHED_ST_OK && (nnz > 0 || exhausted)) st_code = MOESCHED_ST_TRUNCATED;
  }

  double left = 0.0;
  if (st_code != MOESCHED_ST_BAD_INPUT) {
#pragma unroll
    for (int s = 0; s < W; ++s) {
      const int c = s * 32 + lane;
      if (c < N) {   // the matched entries live in registers
        *pl.mem.cell(pl.vrow[s], c) = pl.val[s];
        for (int r = 0; r < N; ++r) left = fmax(left, *pl.mem.cell(r, c));
      }
    }
    left = warp_max_f64(left);
  }
  if (lane == 0) {
    count[b] = k;
    status[b] = st_code;
    sum_lambda[b] = st_code == MOESCHED_ST_BAD_INPUT ? 0.0 : total;
    max_left[b] = left;
  }
}

cudaError_t run_bvn_real(int B, int N, const double* matrix, double tol, int k_max, uint8_t* perm, double* lambda,
                         int32_t* count, double* sum_lambda, double* max_left, double* scratch, int32_t* status,
                         cudaStream_t stream) {
  Geometry ge = plan_geometry(N);
  ge.cluster = false;
  ge.S = bvn_scratch_stride(N);
  ge.wpb = B >= 16 * sm_count() ? 4 : 1;
  ge.smem = peel_smem_bytes(N, ge.cpl) * ge.wpb;
#define MOESCHED_GO(C)                                                                                              \
  return launch_warp_kernel(bvn_real_kernel<C>, ge, B, stream, B, N, ge.S, matrix, tol, k_max, perm, lambda, count, \
                            sum_lambda, max_left, scratch, status)
  switch (ge.cpl) {
    case 1: MOESCHED_GO(1);
    case 2: MOESCHED_GO(2);
    case 3: MOESCHED_GO(3);
    case 4: MOESCHED_GO(4);
    case 5: MOESCHED_GO(5);
    case 6: MOESCHED_GO(6);
    case 7: MOESCHED_GO(7);
    default: MOESCHED_GO(8);
  }
#undef MOESCHED_GO
}

}  // namespace moesched
