// Schedule scoring (paper Sec. 4.1 "Execution time", Sec. 3.3): one matrix per group of warps, thread t owns one row.
//
// The demand matrix sits in shared memory and is consumed as the matchings are replayed; the schedule streams in from
// global memory, 32 matchings (a chunk) at a time and one chunk ahead (cp.async). Matching k serves
// min(dur_k, remaining demand) tokens on each pair; the busiest pair drives the expert batch time; dispatch, compute and
// combine advance as a three-stage pipeline. Link idleness is obtained from totals: sum_k (N dur_k - s_k) equals
// N * sum_k dur_k minus all served tokens.
//
// What bounds it: shared-memory accesses, four per row and matching (destination, mark, entry read and written), and about
// a dozen instructions around them. So
//   * entry (r, j) lies in bank lane(r) whatever j is (32 words per column, one per lane), so that the gather along a
//     matching never conflicts; 16-bit entries put two rows into a word, one for each of two warps;
//   * that a matching is a permutation is seen from marks: every row marks its destination's byte, and after the chunk
//     every thread compares 32 of the marks, sixteen at a time (the OR-reduction of column masks that they replace cost as
//     much as the replay);
//   * the 64-bit times are left aside until a few hundred matchings have been replayed, then every thread composes the
//     three-stage maps of its share of them and the maps are composed in order over the threads: the recurrence
//     costs two instructions per matching instead of ten in a scan over every chunk. (When every prefix is asked for, the
//     scan over the chunk is what is needed.)
// B200: 4096 complete Birkhoff schedules of 64 ranks (1.08 GB) 0.88 ms (46 instructions per matching).
#include <type_traits>

#include "common.cuh"
#include "schedule_read.h"

namespace moesched {

namespace {

constexpr unsigned FULL_MASK = 0xffffffffu;

__device__ __forceinline__ long long warp_sum64(long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL_MASK, v, o);
  return v;
}

// The stage recurrences x_k = max(a_k, x_{k-1}) + b_k are compositions of maps x -> max(x + p, q) (p = b_k,
// q = a_k + b_k), and such maps compose to a map of the same form: (p2, q2) after (p1, q1) is
// (p1 + p2, max(q1 + p2, q2)). An inclusive scan over the lanes (five steps) therefore gives every matching of a
// chunk its value at once, in exact integer arithmetic, instead of 32 dependent steps.
struct MaxPlus {
  long long p, q;
};
constexpr long long MAXPLUS_NONE = -(1LL << 62);   // q of the identity map (p = 0)
__device__ __forceinline__ MaxPlus maxplus_scan(MaxPlus m, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long up_p = __shfl_up_sync(FULL_MASK, m.p, o);
    const long long up_q = __shfl_up_sync(FULL_MASK, m.q, o);
    if (lane >= o) {   // the maps of the lower lanes act first
      m.q = max(up_q + m.p, m.q);
      m.p += up_p;
    }
  }
  return m;
}
__device__ __forceinline__ long long prefix_sum64(long long v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long up = __shfl_up_sync(FULL_MASK, v, o);
    if (lane >= o) v += up;
  }
  return v;
}

// A run of matchings as a map of the three stage times: dispatch d, compute c, combine e become
//   d + l,  max(c + b, d + x),  max(e + l, c + y, d + z).
struct StageMap {
  long long l, b, x, y, z;
  __device__ __forceinline__ void identity() {
    l = b = 0;
    x = y = z = MAXPLUS_NONE;
  }
  __device__ __forceinline__ void append(long long leg, long long comp) {   // one more matching
    l += leg;
    b += comp;
    x = max(x, l) + comp;
    y = max(y, b) + leg;
    z = max(z, x) + leg;
  }
  __device__ __forceinline__ void then(const StageMap& s) {   // the run s follows
    z = max(max(z + s.l, x + s.y), l + s.z);
    y = max(y + s.l, b + s.y);
    x = max(x + s.b, l + s.x);
    l += s.l;
    b += s.b;
  }
};

constexpr int CHUNK = 32;        // matchings replayed between two barriers
constexpr int BATCH_CHUNKS = 8;  // chunks between two passes over the times
constexpr int BATCH = CHUNK * BATCH_CHUNKS;

// Layout of the shared memory of one matrix. T: threads of the group (all CTAs of a cluster together), t_here: of this CTA.
struct EvalLayout {
  size_t slab,   // entry (r, j) of a 32-bit slab (32 rows) or 16-bit slab (64 rows) lies at j * 128 in it
       stage, marks, gmax, served, durs, maps, flags, total;
  int mark_stride;
};
// A bad destination's mark may go behind the T bytes of a matching that are looked at. There is a gap for it, or it goes into the first
// byte of the next matching (or the 16 behind the last one). The bad matching lacks a mark all the same, unless the one before was
// bad too and marked it for it, and so on up to the first one in the buffers, which nothing else marks.
// One buffer is there to be small. Two do without the gap for 64 ranks, where an SM then holds 12 matrices instead of 11: 4096 complete
// Birkhoff schedules 944 -> 881 us, 1658 schedules of 1024 matchings 132 -> 108. (Elsewhere it is as often slower: 16 of 220 ranks 76 ->
// 80, 300 of 129 106 -> 108.)
__host__ __device__ constexpr int mark_gap(bool narrow, int mark_buffers, bool exact64) {
  return narrow && (mark_buffers == 1 || exact64) ? 0 : 16;
}
__host__ __device__ inline EvalLayout eval_layout(int N, int T, int slabs_here, int warps_here, bool prefix, int mark_buffers,
                                                  int mark_gap) {
  EvalLayout L;
  L.slab = (size_t)(N + 1) * 128;   // one column more than there are: where rows beyond N and bad destinations end up
  L.stage = (size_t)slabs_here * L.slab;
  L.mark_stride = T + mark_gap;
  L.marks = L.stage + 2 * align16((size_t)CHUNK * N + 16);
  L.gmax = L.marks + (size_t)mark_buffers * CHUNK * L.mark_stride + (mark_gap == 0 ? 16 : 0);
  L.served = L.gmax + (prefix ? 2 * CHUNK : BATCH) * sizeof(int);
  L.durs = L.served + (prefix ? 2 * CHUNK : 0) * sizeof(long long);
  L.maps = L.durs + (size_t)warps_here * CHUNK * sizeof(int);
  L.flags = L.maps + (size_t)warps_here * sizeof(StageMap) + 8 * sizeof(long long);
  L.total = align16(L.flags + 4 * sizeof(int));
  return L;
}

__device__ __forceinline__ void async_copy16(void* dst, const void* src, int bytes) {   // bytes beyond are zero-filled
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst)), "l"(src), "r"(bytes) : "memory");
}
// Shared memory by 32-bit address. Marks may lie in the other CTA of a cluster.
__device__ __forceinline__ unsigned load_u8(unsigned at) {
  unsigned v;
  asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(at) : "memory");
  return v;
}
template <bool CLUSTER>
__device__ __forceinline__ void store_u8(unsigned at, unsigned v) {
  if constexpr (CLUSTER) asm volatile("st.shared::cluster.u8 [%0], %1;" ::"r"(at), "r"(v) : "memory");
  else asm volatile("st.shared.u8 [%0], %1;" ::"r"(at), "r"(v) : "memory");
}
template <bool NARROW>
__device__ __forceinline__ int load_entry(unsigned at) {
  int v;
  if constexpr (NARROW) asm volatile("ld.shared.u16 %0, [%1];" : "=r"(v) : "r"(at) : "memory");
  else asm volatile("ld.shared.s32 %0, [%1];" : "=r"(v) : "r"(at) : "memory");
  return v;
}
template <bool NARROW>
__device__ __forceinline__ void store_entry(unsigned at, int v) {
  if constexpr (NARROW) asm volatile("st.shared.u16 [%0], %1;" ::"r"(at), "r"(v) : "memory");
  else asm volatile("st.shared.s32 [%0], %1;" ::"r"(at), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned address_in_cta(unsigned at, unsigned rank) {   // of the cluster
  unsigned out;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(out) : "r"(at), "r"(rank));
  return out;
}
__device__ __forceinline__ void async_copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

}  // namespace

// WARPS: warps of a CTA that share one matrix. NARROW: 16-bit entries (a matrix that does not fit is left, its status marked
// CLASS_I32, to a launch with 32-bit entries and only_class set, which handles nothing else). CLUSTER: the rows are split
// over the two CTAs of a cluster; marks and maxima of both are kept by CTA 0.
// PREFIX: also write, after every matching k, the overlap makespan and the unserved tokens of the
// schedule cut after k+1 matchings (entries beyond count, or all entries of a bad schedule, are -1).
// JOBS (with PREFIX): the two per-matching arrays receive instead the job times of matching k in the
// three-stage flow shop: reconfiguration + transfer time, and the time of its expert batch.
// EXACT: N is the number of threads, so that every address of a chunk is a constant away from the thread's own.
// MARK_BUFFERS: one, at the price of a barrier per chunk, or two (see launch_eval_as).
template <int WARPS, bool NARROW, bool CLUSTER, bool PREFIX, bool JOBS, bool EXACT, int MARK_BUFFERS>
__global__ void __launch_bounds__(WARPS == 1 ? 128 : 32 * WARPS)
    eval_kernel(int B, int n_arg, const int32_t* __restrict__ demand, int k_stride, const uint8_t* __restrict__ perm,
                const int32_t* __restrict__ dur, const int32_t* __restrict__ count, moesched_model_t model,
                FastDiv by_gbps, long long* __restrict__ overlap, long long* __restrict__ serial,
                long long* __restrict__ idle_ns, long long* __restrict__ idle_tok, long long* __restrict__ unserved,
                int32_t* status, long long* __restrict__ prefix_overlap, long long* __restrict__ prefix_unserved,
                int only_class) {
  constexpr int T_HERE = 32 * WARPS, T = CLUSTER ? 2 * T_HERE : T_HERE;
  const int N = EXACT ? T : n_arg;
  using Entry = typename std::conditional<NARROW, unsigned short, int>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31;
  const int warp = WARPS == 1 ? 0 : (int)(threadIdx.x >> 5);   // within the group
  const int t_here = warp * 32 + lane;
  const int rank = CLUSTER ? (int)cluster_ctarank() : 0;
  const int b = CLUSTER ? (int)(blockIdx.x >> 1)
                        : (WARPS == 1 ? (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) : (int)blockIdx.x);
  if (b >= B) return;
  if (only_class != 0 && status[b] != only_class) return;
  const int slabs = NARROW ? (N + 63) / 64 : (N + 31) / 32;
  const int slabs_here = CLUSTER ? WARPS : slabs;   // (the second CTA of a cluster may leave some unused)
  const EvalLayout L = eval_layout(N, T, slabs_here, WARPS, PREFIX, MARK_BUFFERS,
                                   mark_gap(NARROW, MARK_BUFFERS, EXACT && T == 64));
  unsigned char* base = smem_raw + (WARPS == 1 ? (size_t)(threadIdx.x >> 5) * L.total : 0);
  // what both CTAs of a cluster write to is kept by CTA 0
  unsigned char* shared0 = base;
  if constexpr (CLUSTER) shared0 = reinterpret_cast<unsigned char*>(map_to_cta(reinterpret_cast<int*>(base), 0));
  int* gmax = reinterpret_cast<int*>(shared0 + L.gmax);
  unsigned long long* served = reinterpret_cast<unsigned long long*>(shared0 + L.served);
  int* flags = reinterpret_cast<int*>(shared0 + L.flags);   // [parity]: the schedule was found bad since the last barrier
  long long* totals = reinterpret_cast<long long*>(shared0 + L.maps + WARPS * sizeof(StageMap));   // demand, left, then scratch
  StageMap* maps = reinterpret_cast<StageMap*>(base + L.maps);
  int* my_durs = reinterpret_cast<int*>(base + L.durs) + warp * CHUNK;
  auto barrier = [&]() {
    if constexpr (CLUSTER) cluster_sync_all();
    else if constexpr (WARPS == 1) __syncwarp();
    else __syncthreads();
  };

  // thread -> row; threads without a row replay zeros in a spare column and mark a byte of their own
  const int row = NARROW ? (warp >> 1) * 64 + 2 * lane + (warp & 1) : rank * T_HERE + t_here;
  const int t = rank * T_HERE + t_here;
  const bool in = EXACT || row < N;
  unsigned char* cells = base + (NARROW ? (size_t)(warp >> 1) * L.slab + lane * 4 + (warp & 1) * 2
                                        : (size_t)warp * L.slab + lane * 4);
  unsigned mark_at = 0u, mark_step = 1u, cell_step = 128u;
  if (!in) {
    cells = base + (size_t)N * 128 + lane * 4;   // the spare column of slab 0 (always zero)
    cell_step = 0u;
    mark_step = 0u;
    // any byte of N .. T-1, one for each such thread
    mark_at = NARROW ? (unsigned)row : (unsigned)t;
  }

  // ---- shared state, demand (each thread its own row), total, validation ----
  for (int e = t_here; e < MARK_BUFFERS * CHUNK * L.mark_stride / 4; e += T_HERE) reinterpret_cast<int*>(base + L.marks)[e] = 0;
  for (int e = t_here; e < (PREFIX ? 2 * CHUNK : BATCH); e += T_HERE) reinterpret_cast<int*>(base + L.gmax)[e] = 0;
  if constexpr (PREFIX)
    for (int e = t_here; e < 2 * CHUNK; e += T_HERE) reinterpret_cast<unsigned long long*>(base + L.served)[e] = 0ull;
  if (t_here < 8) reinterpret_cast<long long*>(base + L.maps + WARPS * sizeof(StageMap))[t_here] = 0;
  if (t_here < 4) reinterpret_cast<int*>(base + L.flags)[t_here] = 0;
  for (int e = t_here; e < slabs_here * 32; e += T_HERE)   // the spare columns
    *reinterpret_cast<int*>(base + (size_t)(e >> 5) * L.slab + (size_t)N * 128 + (e & 31) * 4) = 0;
  barrier();
  long long mine = 0;
  int neg = 0, big = 0;
  if (in) {
    const int32_t* D = demand + ((size_t)b * N + row) * N;
    if ((N & 3) == 0 && (reinterpret_cast<uintptr_t>(demand) & 15) == 0) {
#pragma unroll 4
      for (int j = 0; j < N; j += 4) {
        const int4 v = *reinterpret_cast<const int4*>(D + j);
        neg |= v.x | v.y | v.z | v.w;   // sign bit
        big |= v.x | v.y | v.z | v.w;
        mine += (long long)v.x + v.y + v.z + v.w;
        *reinterpret_cast<Entry*>(cells + (size_t)j * 128) = (Entry)v.x;
        *reinterpret_cast<Entry*>(cells + (size_t)(j + 1) * 128) = (Entry)v.y;
        *reinterpret_cast<Entry*>(cells + (size_t)(j + 2) * 128) = (Entry)v.z;
        *reinterpret_cast<Entry*>(cells + (size_t)(j + 3) * 128) = (Entry)v.w;
      }
    } else {
#pragma unroll 8
      for (int j = 0; j < N; ++j) {
        const int v = D[j];
        neg |= v;
        big |= v;
        mine += v;
        *reinterpret_cast<Entry*>(cells + (size_t)j * 128) = (Entry)v;
      }
    }
  }
  neg = __any_sync(FULL_MASK, neg < 0);
  big = __any_sync(FULL_MASK, (big & ~0xffff) != 0);
  mine = warp_sum64(mine);
  if (lane == 0) {
    atomicAdd(reinterpret_cast<unsigned long long*>(&totals[0]), (unsigned long long)mine);
    if (neg) flags[2] = 1;
    if (big) flags[3] = 1;
  }
  barrier();
  const long long total = totals[0];
  if (NARROW && flags[3]) {   // uniform (negative entries count as wide too)
    if (t == 0) status[b] = CLASS_I32;
    return;
  }
  const int K = count[b];
  bool bad = flags[2] != 0 || K < 0 || K > k_stride;

  // ---- schedule: where the bytes of a chunk come from ----
  const uint8_t* pb = perm + (size_t)b * k_stride * N;
  const int32_t* db = dur + (size_t)b * k_stride;
  const int skew = (int)(reinterpret_cast<uintptr_t>(pb) & 15);   // a chunk is a multiple of 16 bytes: the same for all
  unsigned char* stage = base + L.stage;
  const size_t stage_bytes = align16((size_t)CHUNK * N + 16);
  // chunk c into its buffer, as aligned groups of 16 bytes; nothing outside the schedules is read
  auto fetch = [&](int c, auto is_first) {
    const int bytes = min(CHUNK, K - c * CHUNK) * N;
    const uint8_t* first = pb + (size_t)c * CHUNK * N;
    unsigned char* dst = stage + (c & 1) * stage_bytes;
    for (int g = t_here; g * 16 < bytes + skew; g += T_HERE) {
      const int from = g * 16 - skew;   // offset of the group from the first byte
      if (decltype(is_first)::value && from < 0 && begins_before_the_array(pb - perm, skew)) {
        for (int q = skew; q < 16 && q - skew < bytes; ++q) dst[q] = first[q - skew];
      } else {
        async_copy16(dst + g * 16, first + from, min(16, bytes - from));
      }
    }
  };
  const int chunks = bad ? 0 : (K + CHUNK - 1) / CHUNK;
  int dk_next = 0;
  if (chunks > 0) {
    fetch(0, std::true_type{});
    dk_next = lane < K ? db[lane] : 0;
  }

  long long dsp = 0, cmp = 0, cmb = 0, comp_sum = 0, dsp1 = 0, dur_sum = 0, served_sum = 0;   // live in warp 0 of CTA 0
  const long long round_up = model.link_gbps - 1;
  // dk < 2^31, bytes_per_token and link_gbps <= 2^20: the dividend stays below 2^55
  auto leg_ns = [&](int dk) {
    return model.reconfig_ns + fast_div((long long)dk * model.bytes_per_token * 8 + round_up, by_gbps);
  };

  // The matchings from k0 on that have been replayed since the last call, all threads: job times, composed in order.
  auto settle_times = [&](int k0, int flag) {
    if (rank == 0) {
      constexpr int PER = BATCH / T_HERE;
      StageMap m;
      m.identity();
      long long d = 0;
#pragma unroll
      for (int i = 0; i < PER; ++i) {
        const int slot = t_here * PER + i, k = k0 + slot;
        if (k < K && slot < BATCH) {
          const int dk = max(db[k], 0);
          m.append(leg_ns(dk), batch_time_ns(model, gmax[slot]));
          d += dk;
          if (k == 0) dsp1 = m.l;
        }
        if (slot < BATCH) gmax[slot] = 0;
      }
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        StageMap s;
        s.l = __shfl_down_sync(FULL_MASK, m.l, o);
        s.b = __shfl_down_sync(FULL_MASK, m.b, o);
        s.x = __shfl_down_sync(FULL_MASK, m.x, o);
        s.y = __shfl_down_sync(FULL_MASK, m.y, o);
        s.z = __shfl_down_sync(FULL_MASK, m.z, o);
        m.then(s);   // lanes whose source lies beyond lane 31 are not looked at any more
        d += __shfl_down_sync(FULL_MASK, d, o);
      }
      if (lane == 0) {
        maps[warp] = m;
        atomicAdd(reinterpret_cast<unsigned long long*>(&totals[2]), (unsigned long long)d);
      }
    }
    barrier();
    if (rank == 0 && warp == 0) {
      StageMap m = maps[0];
      for (int w = 1; w < WARPS; ++w) m.then(maps[w]);
      comp_sum += m.b;
      const long long legs = dsp + m.l;
      // stage sums beyond 2^60 ns are out of range (256 matchings add less than 2^62 + 2^49, so nothing has wrapped yet)
      if (legs > (1LL << 60) || comp_sum > (1LL << 60)) flags[flag] = 1;
      else {
        cmb = max(max(cmb + m.l, cmp + m.y), dsp + m.z);
        cmp = max(cmp + m.b, dsp + m.x);
        dsp = legs;
      }
    }
  };

  // Step c replays chunk c; before that, the marks of chunk c-1 are looked at. One barrier per step, and one more where there is one
  // buffer for marks.
  int k_settled = 0;
  for (int c = 0; c <= chunks; ++c) {
    async_copies_done();
    barrier();
    if (c > 0 && flags[(c - 1) & 1] != 0) { bad = true; break; }   // (written between the last two barriers only: uniform)
    if (c > 0) {
      // every row of the chunk before marked its destination; all T marks of a matching are there iff it is a permutation
      const int p = (c - 1) & 1;
      const unsigned want = 0x01010101u << ((MARK_BUFFERS == 1 ? c - 1 : (c - 1) >> 1) & 1);
      if (rank == 0) {
        unsigned off = 0u;
#pragma unroll
        for (int i = 0; i < T / T_HERE * 2; ++i) {
          const int g = i * T_HERE + t_here;   // group of 16 marks; T / 16 of them to a matching
          const uint4 v = *reinterpret_cast<const uint4*>(base + L.marks + (size_t)(MARK_BUFFERS == 1 ? 0 : p) * CHUNK * L.mark_stride +
                                                          (g / (T / 16)) * L.mark_stride + (g % (T / 16)) * 16);
          off |= (v.x ^ want) | (v.y ^ want) | (v.z ^ want) | (v.w ^ want);
        }
        if (off != 0u) flags[c & 1] = 1;
      }
      if constexpr (MARK_BUFFERS == 1) barrier();   // the marks have been looked at
      if constexpr (PREFIX) {
        if (rank == 0 && warp == 0) {
          // times of the chunk, one matching per lane, then the three-stage recurrence by scans
          const int k0 = (c - 1) * CHUNK, kend = min(CHUNK, K - k0);
          const bool has = lane < kend;
          const int dk = has ? max(db[k0 + lane], 0) : 0;
          const int g = gmax[p * CHUNK + lane];
          const long long served_mine = (long long)served[p * CHUNK + lane];
          gmax[p * CHUNK + lane] = 0;
          served[p * CHUNK + lane] = 0ull;
          const long long comp = has ? batch_time_ns(model, g) : 0;
          const long long leg = has ? leg_ns(dk) : 0;
          comp_sum += warp_sum64(comp);
          dur_sum += warp_sum64((long long)dk);
          const long long dsp_mine = dsp + prefix_sum64(leg, lane);
          // stage sums beyond 2^60 ns are out of range (a chunk adds less than 2^60, so nothing has wrapped yet)
          if (__shfl_sync(FULL_MASK, dsp_mine, 31) > (1LL << 60) || comp_sum > (1LL << 60)) {
            flags[c & 1] = 1;
          } else {
            MaxPlus f;
            f.p = comp;
            f.q = has ? dsp_mine + comp : MAXPLUS_NONE;
            f = maxplus_scan(f, lane);
            const long long cmp_mine = max(cmp + f.p, f.q);
            MaxPlus h;
            h.p = leg;
            h.q = has ? cmp_mine + leg : MAXPLUS_NONE;
            h = maxplus_scan(h, lane);
            const long long cmb_mine = max(cmb + h.p, h.q);
            if (c == 1) dsp1 = __shfl_sync(FULL_MASK, dsp_mine, 0);
            dsp = __shfl_sync(FULL_MASK, dsp_mine, kend - 1);
            cmp = __shfl_sync(FULL_MASK, cmp_mine, kend - 1);
            cmb = __shfl_sync(FULL_MASK, cmb_mine, kend - 1);
            const long long run = prefix_sum64(served_mine, lane);
            if (has) {
              prefix_overlap[(size_t)b * k_stride + k0 + lane] = JOBS ? leg : cmb_mine;
              prefix_unserved[(size_t)b * k_stride + k0 + lane] = JOBS ? comp : total - (served_sum + run);
            }
            served_sum += __shfl_sync(FULL_MASK, run, 31);
          }
        }
      } else if (c % BATCH_CHUNKS == 0 || c == chunks) {
        settle_times(k_settled, c & 1);
        k_settled = c * CHUNK;
        barrier();   // the maxima have been read and cleared
      }
    }
    if (c == chunks) break;

    // ---- replay chunk c ----
    const int kend = min(CHUNK, K - c * CHUNK);
    const unsigned char* from = stage + (c & 1) * stage_bytes + skew;
    if (kend < CHUNK) {   // the last chunk: matchings beyond the schedule send nothing along the diagonal
      if (in)
        for (int q = kend; q < CHUNK; ++q) const_cast<unsigned char*>(from)[q * N + row] = (unsigned char)row;
      barrier();
    }
    const int dk_mine = dk_next;
    if (__any_sync(FULL_MASK, dk_mine < 0) && lane == 0) flags[c & 1] = 1;
    my_durs[lane] = NARROW ? min(max(dk_mine, 0), 65535) : max(dk_mine, 0);
    __syncwarp();
    if (c + 1 < chunks) {
      fetch(c + 1, std::false_type{});
      const int k = (c + 1) * CHUNK + lane;
      dk_next = k < K ? db[k] : 0;
    }
    const unsigned stamp = 1u << ((MARK_BUFFERS == 1 ? c : c >> 1) & 1);   // differs from what the buffer holds
    unsigned dest_at = smem_addr(from) + (in ? row : 0);
    unsigned mark_base = smem_addr(base + L.marks) + (MARK_BUFFERS == 1 ? 0 : c & 1) * CHUNK * L.mark_stride + mark_at;
    if constexpr (CLUSTER) mark_base = address_in_cta(mark_base, 0);
    const unsigned cell_base = smem_addr(cells);
    int g_mine = 0;
    unsigned s_lo = 0u, s_hi = 0u;
#pragma unroll 1
    for (int q0 = 0; q0 < CHUNK; q0 += 8) {
      unsigned j[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) j[q] = load_u8(dest_at + q * N);
      dest_at += 8 * N;
      const int4 da = *reinterpret_cast<const int4*>(my_durs + q0), dc = *reinterpret_cast<const int4*>(my_durs + q0 + 4);
      const int dk[8] = {da.x, da.y, da.z, da.w, dc.x, dc.y, dc.z, dc.w};
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        // a bad destination serves nothing and leaves a mark missing
        const unsigned col = min(j[q], (unsigned)N);
        store_u8<CLUSTER>(mark_base + q * L.mark_stride + (EXACT ? col : col * mark_step), stamp);
        const unsigned cell = cell_base + col * (EXACT ? 128u : cell_step);
        const int val = load_entry<NARROW>(cell), sv = min(dk[q], val);
        store_entry<NARROW>(cell, max(val - dk[q], 0));
        const int g = __reduce_max_sync(FULL_MASK, sv);
        if (lane == q0 + q) g_mine = g;
        if constexpr (PREFIX && !JOBS) {
          const unsigned lo = __reduce_add_sync(FULL_MASK, NARROW ? (unsigned)sv : (unsigned)sv & 0xffffu);
          const unsigned hi = NARROW ? 0u : __reduce_add_sync(FULL_MASK, (unsigned)sv >> 16);
          if (lane == q0 + q) { s_lo = lo; s_hi = hi; }
        }
      }
      mark_base += 8 * L.mark_stride;
    }
    if constexpr (PREFIX) {
      if (g_mine > 0) atomicMax(&gmax[(c & 1) * CHUNK + lane], g_mine);
      if constexpr (!JOBS) {
        const unsigned long long s = ((unsigned long long)s_hi << 16) + s_lo;
        if (s != 0ull) atomicAdd(&served[(c & 1) * CHUNK + lane], s);
      }
    } else {
      if (g_mine > 0) atomicMax(&gmax[(c % BATCH_CHUNKS) * CHUNK + lane], g_mine);
    }
  }
  barrier();
  if (chunks > 0 && flags[chunks & 1] != 0) bad = true;   // (found in the last step)

  // ---- demand left over ----
  long long left = 0;
  if (in)
    for (int j = 0; j < N; ++j) left += *reinterpret_cast<const Entry*>(cells + (size_t)j * 128);
  left = warp_sum64(left);
  if (lane == 0 && left != 0) atomicAdd(reinterpret_cast<unsigned long long*>(&totals[1]), (unsigned long long)left);
  barrier();
  if (t == 0) {
    if constexpr (!PREFIX) dur_sum = totals[2];
    left = totals[1];
    if (dur_sum > (1LL << 40)) bad = true;
    totals[3] = bad ? 1 : 0;
    if (bad) {
      overlap[b] = serial[b] = idle_ns[b] = idle_tok[b] = unserved[b] = 0;
      status[b] = MOESCHED_ST_BAD_INPUT;
    } else {
      overlap[b] = cmb;
      serial[b] = 2 * dsp + comp_sum;
      idle_ns[b] = K > 0 ? (cmp - dsp1) - comp_sum : 0;
      idle_tok[b] = (long long)N * dur_sum - (total - left);
      unserved[b] = left;
      status[b] = MOESCHED_ST_OK;
    }
  }
  if constexpr (PREFIX) {
    barrier();
    if (rank == 0) {
      const int from = totals[3] != 0 ? 0 : K;
      for (int k = from + t_here; k < k_stride; k += T_HERE) {
        prefix_overlap[(size_t)b * k_stride + k] = -1;
        prefix_unserved[(size_t)b * k_stride + k] = -1;
      }
    }
  }
  if constexpr (CLUSTER) cluster_sync_all();   // CTA 0's memory is in use until here
}

// ---- host side ---------------------------------------------------------------------------

namespace {
struct EvalArgs {
  int B, N;
  const int32_t* demand;
  int k_stride;
  const uint8_t* perm;
  const int32_t *dur, *count;
  moesched_model_t model;
  FastDiv by_gbps;
  long long *overlap, *serial, *idle_ns, *idle_tok, *unserved;
  int32_t* status;
  long long *prefix_overlap, *prefix_unserved;
  cudaStream_t stream;
};
size_t eval_smem(int N, int warps, bool narrow, bool cluster, bool prefix, int buffers) {
  const int slabs = cluster ? warps : narrow ? (N + 63) / 64 : (N + 31) / 32;
  const int T = 32 * warps * (cluster ? 2 : 1);
  return eval_layout(N, T, slabs, warps, prefix, buffers, mark_gap(narrow, buffers, !prefix && N == 64 && T == 64)).total;
}

template <int WARPS, bool NARROW, bool CLUSTER, int BUFFERS>
cudaError_t launch_eval_with(const EvalArgs& a, bool jobs, int only_class) {
  const bool prefix = a.prefix_overlap != nullptr;
  Geometry ge;
  ge.cluster = CLUSTER;
  ge.threads_per_cta = 32 * WARPS;
  ge.wpb = 1;                                    // matrices per CTA
  if (WARPS == 1) { ge.wpb = a.B >= 4 * sm_count() ? 4 : 1; ge.threads_per_cta = 32 * ge.wpb; }
  ge.smem = eval_smem(a.N, WARPS, NARROW, CLUSTER, prefix, BUFFERS) * ge.wpb;
  const bool full = a.N == 32 * WARPS * (CLUSTER ? 2 : 1);
#define MOESCHED_GO(P, J, F)                                                                                         \
  return launch_warp_kernel(eval_kernel<WARPS, NARROW, CLUSTER, P, J, F, BUFFERS>, ge, a.B, a.stream, a.B, a.N,      \
                            a.demand, a.k_stride, a.perm, a.dur, a.count, a.model, a.by_gbps, a.overlap, a.serial,   \
                            a.idle_ns, a.idle_tok, a.unserved, a.status, a.prefix_overlap, a.prefix_unserved, only_class)
  if (prefix && jobs) MOESCHED_GO(true, true, false);
  if (prefix) MOESCHED_GO(true, false, false);
  if constexpr (!CLUSTER && (BUFFERS == 2 || WARPS == 2))   // (128 and 256 ranks never have one buffer here)
    if (full) MOESCHED_GO(false, false, true);
  MOESCHED_GO(false, false, false);
#undef MOESCHED_GO
}

// One buffer for the marks leaves room for up to a third more matrices per SM, which is of use where the SMs then hold the whole batch
// at once (B200, schedules of six matchings per rank: 600 x 112 ranks 86.0 -> 69.4 us, with prefix scores 126.6 -> 89.5; 300 x 140 111.7 ->
// 95.1 and 161.5 -> 111.7). Otherwise it may as well leave a longer tail (550 x 129, 32 matchings, three at a time instead of two 27.0 ->
// 33.8; 833 x 112, 28 matchings, 25.4 -> 27.6). Where an SM holds a single matrix either way, the prefix scores are faster with one (256
// ranks 134.1 -> 130.5 us), the scores as a whole with two (86.4, 87.0). Only 16-bit entries come here: 32-bit ones are for
// batches that are held at once.
template <int WARPS, bool NARROW, bool CLUSTER>
cudaError_t launch_eval_as(const EvalArgs& a, bool jobs, int only_class) {
  if constexpr (NARROW) {
    const bool prefix = a.prefix_overlap != nullptr;
    auto held = [&](int buffers) {   // matrices per SM
      return (int)((SMEM_LIMIT + 1024) / (eval_smem(a.N, WARPS, true, false, prefix, buffers) + 1024));
    };
    const int one = held(1), two = held(2);
    const long long per_sm = (a.B + sm_count() - 1) / sm_count();
    if (one == 1 ? prefix : per_sm <= one && per_sm > two) return launch_eval_with<WARPS, NARROW, CLUSTER, 1>(a, jobs, only_class);
  }
  return launch_eval_with<WARPS, NARROW, CLUSTER, 2>(a, jobs, only_class);
}
}  // namespace

cudaError_t run_eval(int B, int N, const int32_t* demand, int k_stride, const uint8_t* perm, const int32_t* dur,
                     const int32_t* count, const moesched_model_t& model, long long* overlap, long long* serial,
                     long long* idle_ns, long long* idle_tok, long long* unserved, int32_t* status,
                     long long* prefix_overlap, long long* prefix_unserved, cudaStream_t stream, bool jobs) {
  const EvalArgs a{B, N, demand, k_stride, perm, dur, count, model, make_fastdiv(model.link_gbps), overlap, serial,
                   idle_ns, idle_tok, unserved, status, prefix_overlap, prefix_unserved, stream};
  if (N <= 32) return launch_eval_as<1, false, false>(a, jobs, 0);
  const int warps = N <= 64 ? 2 : N <= 128 ? 4 : 8;
  const size_t as_int32 = eval_smem(N, warps, false, false, prefix_overlap != nullptr, 2);
  // As in the greedy path: 32-bit entries at once where the whole batch is resident that way, else 16-bit entries first and
  // then the matrices that do not fit them (over a 2-CTA cluster where one CTA cannot hold the matrix).
  int only_class = 0;
  if (as_int32 > SMEM_LIMIT || B > (long long)sm_count() * (long long)(SMEM_LIMIT / (as_int32 + 1024))) {
    cudaError_t e = warps == 2   ? launch_eval_as<2, true, false>(a, jobs, 0)
                    : warps == 4 ? launch_eval_as<4, true, false>(a, jobs, 0)
                                 : launch_eval_as<8, true, false>(a, jobs, 0);
    if (e != cudaSuccess) return e;
    only_class = CLASS_I32;
  }
  if (as_int32 > SMEM_LIMIT) return launch_eval_as<4, false, true>(a, jobs, only_class);
  return warps == 2   ? launch_eval_as<2, false, false>(a, jobs, only_class)
         : warps == 4 ? launch_eval_as<4, false, false>(a, jobs, only_class)
                      : launch_eval_as<8, false, false>(a, jobs, only_class);
}

}  // namespace moesched
