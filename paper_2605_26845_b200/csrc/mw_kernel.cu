// Greedy max-weight decomposition (paper Sec. 3.2), one warp per demand matrix.
//
// Each greedy step solves one assignment problem on the residual matrix R by shortest augmenting paths on
// cost = -R (a Jonker-Volgenant style search, column duals v warm-started from the previous step), marks the edges that
// are tight under the optimal duals and hands that graph to the Peeler (peel.cuh), which returns the lexicographically
// smallest optimal permutation. The matched entries are then served whole; the largest one is the matching's duration.
//
// What bounds it: the column scans of the shortest-path searches, one after the other (160 per matching at N = 64), each
// a chain of a warp minimum, a load of the settled column's row and a relaxation; a full GPU is bound by
// their instructions. The search therefore holds every candidate as ONE sortable word, distance above "column is
// matched" above the row (or column) to go on with, wherever distances fit 23 bits: one minimum over the warp then gives the
// distance, whether the path ends there, and the row to scan next.
#include <type_traits>

#include "peel.cuh"

namespace moesched {

// STORE of the residual matrix: 0 int32 in this CTA's shared memory, 1 int32 split over a 2-CTA cluster, 2 16-bit entries.
template <int STORE>
struct Residual {
  using T = typename std::conditional<STORE == 2, unsigned short, int>::type;
  T* near_;
  T* far_;
  int N, split;
  __device__ __forceinline__ T* row(int r) const {
    if constexpr (STORE == 1) return r < split ? near_ + r * N : far_ + (r - split) * N;
    else return near_ + r * N;
  }
};

// Shared memory of one warp next to the matrix and the Peeler's: the assignment by rows and columns, predecessors of the
// running search, and a scratch word per row or column.
struct AssignShared {
  int* urow;         // [row] row dual
  unsigned* claim;   // [row or column]
  short* x;          // [row] column
  unsigned* pred;    // [column] row from which the running search reached it, and that row's column << 16
};
__host__ __device__ inline size_t assign_smem_bytes(int N) {
  return 3 * align16((size_t)N * 4) + align16((size_t)N * 2);
}
// With eight words it lies in the Peeler's search levels: the assignment is done with once the tight edges are in the table,
// before the first search, and the levels take 32 bytes a rank, so that a matrix of 232 ranks still fits as int32.
__host__ __device__ inline size_t state_smem_bytes(int N, int W) {
  return peel_smem_bytes(N, W) + (W == 8 ? 0 : assign_smem_bytes(N));
}
__device__ __forceinline__ AssignShared assign_shared(unsigned char* p, int N) {
  const size_t words = align16((size_t)N * 4);
  AssignShared a;
  a.urow = reinterpret_cast<int*>(p);
  a.claim = reinterpret_cast<unsigned*>(p + words);
  a.pred = reinterpret_cast<unsigned*>(p + 2 * words);
  a.x = reinterpret_cast<short*>(p + 3 * words);
  return a;
}

// A column's tag is its number while it is free and TAG_MATCHED | its row once it is matched, so that free columns win ties
// and a minimum that carries a tag along names the row to be scanned next. Rows are tagged likewise where columns choose.
constexpr unsigned TAG_MATCHED = 0x100u;
constexpr unsigned TAG_MASK = 0x1ffu;
constexpr int TAG_BITS = 9;
// Narrow matrices: distances, which lie within 3 C of zero (C the largest entry), and tag fit one word. Wide ones: so does,
// nearly always, the distance from the row's dual, which no column of the search undercuts; it saturates at FAR, and a search
// that gets there is done over with distances of their own.
constexpr int NARROW_BIAS = 1 << 22;
constexpr int NARROW_MAX_ENTRY = NARROW_BIAS / 4;
constexpr unsigned NONE = 0xffffffffu;
constexpr unsigned FAR = (1u << (32 - TAG_BITS)) - 1u;

__device__ __forceinline__ unsigned packed(int dist, unsigned tag) { return ((unsigned)(dist + NARROW_BIAS) << TAG_BITS) | tag; }
__device__ __forceinline__ int packed_dist(unsigned k) { return (int)(k >> TAG_BITS) - NARROW_BIAS; }

// Smallest distance over the warp with the smallest tag among equals, in two steps (wide matrices). INF32: there is none.
template <int W>
__device__ __forceinline__ void nearest(const int (&d)[W], const unsigned (&tag)[W], int& dist, unsigned& who) {
  int m = INF32;
#pragma unroll
  for (int s = 0; s < W; ++s) m = min(m, d[s]);
  dist = __reduce_min_sync(FULL, m);
  unsigned t = NONE;
#pragma unroll
  for (int s = 0; s < W; ++s)
    if (d[s] == dist) t = min(t, tag[s]);
  who = __reduce_min_sync(FULL, t);
}

// One assignment problem. The column duals v carry over from the previous greedy step (weights only decreased, so they
// are still feasible); they are shifted so that the largest is zero. Every column of the previous optimum was tight for its
// row, so v lies within [-C, 0], C the largest entry, and row duals (row minima of cost - v) within [-C, 0] too.
//   1. Rows: each names the column of its smallest reduced cost; a column goes to the lowest row that names it.
//   2. Columns left free: each raises its dual to the largest feasible value, min over the rows of cost - row dual (within
//      [-C, C]), where it becomes tight for a row; if that row is free the two are matched. (N = 64 workload: 15 instead of
//      21 rows left, 161 instead of 225 column scans per matching.)
//   3. Rows left over are inserted one by one by a shortest-path search that settles one column per scan, free columns
//      first among equals, and moves the duals of the settled columns.
// Distances lie within [-2 C, 3 C]. On return sh.x and sh.urow hold the assignment and the row duals. False if a
// search ran out of columns (an inconsistency).
template <int W, int STORE, bool WIDE>
__device__ __forceinline__ bool solve_assignment(const Residual<STORE>& R, int N, int lane, const AssignShared& sh,
                                                 int (&v)[W], unsigned (&work)[MOESCHED_WORK_FIELDS]) {
  bool in[W];
  int vmax = -INF32;
#pragma unroll
  for (int s = 0; s < W; ++s) {
    in[s] = s * 32 + lane < N;
    if (in[s]) vmax = max(vmax, v[s]);
  }
  vmax = __reduce_max_sync(FULL, vmax);
  unsigned tag[W], base[W];   // of the lane's columns; base: packed(-v, tag), so that base - (entry << TAG_BITS) is a key
#pragma unroll
  for (int s = 0; s < W; ++s) {
    v[s] -= vmax;
    tag[s] = (unsigned)(s * 32 + lane);
    base[s] = in[s] ? packed(-v[s], tag[s]) : NONE;
    if (in[s]) sh.claim[s * 32 + lane] = NONE;
  }
  // ---- 1. rows name columns, several at a time; lane l keeps what rows l, l + 32, ... found ----
  // (Eight instead of four with three and four words: 300 x 96 ranks 3.27 -> 3.23 ms, 60 x 72 ranks 1.92 -> 1.87; four instead of two with
  // more: 100 x 160 ranks 4.43 -> 4.57.)
  constexpr int ROWS = W <= 4 ? 8 : 2;
  int u[W];
  unsigned named[W];
#pragma unroll
  for (int w = 0; w < W; ++w) {
    unsigned k_mine = 0u;
    u[w] = 0;
    named[w] = 0u;
    for (int q0 = 0; q0 < 32 && w * 32 + q0 < N; q0 += ROWS) {   // (the last row again beyond the end)
      if constexpr (WIDE) {
#pragma unroll
        for (int q = 0; q < ROWS; ++q) {
          const auto* row = R.row(min(w * 32 + q0 + q, N - 1));
          int d[W], dist;
          unsigned who;
#pragma unroll
          for (int s = 0; s < W; ++s) d[s] = in[s] ? -(int)row[s * 32 + lane] - v[s] : INF32;
          nearest<W>(d, tag, dist, who);
          if (lane == q0 + q) { u[w] = dist; named[w] = who; }
        }
      } else {
        unsigned k[ROWS];
#pragma unroll
        for (int q = 0; q < ROWS; ++q) {
          const auto* row = R.row(min(w * 32 + q0 + q, N - 1));
          k[q] = NONE;
#pragma unroll
          for (int s = 0; s < W; ++s) k[q] = min(k[q], base[s] - ((unsigned)(in[s] ? row[s * 32 + lane] : 0) << TAG_BITS));
        }
#pragma unroll
        for (int q = 0; q < ROWS; ++q) {
          k[q] = __reduce_min_sync(FULL, k[q]);
          if (lane == q0 + q) k_mine = k[q];
        }
      }
    }
    if constexpr (!WIDE) {
      u[w] = packed_dist(k_mine);
      named[w] = k_mine & 0xffu;
    }
  }
  work[WK_TIGHT] += N;
  __syncwarp();
#pragma unroll
  for (int s = 0; s < W; ++s) {
    if (in[s]) {
      sh.urow[s * 32 + lane] = u[s];
      atomicMin(&sh.claim[MS_AT((int)named[s], N)], (unsigned)(s * 32 + lane));
    }
  }
  __syncwarp();
  bool row_free[W];
  unsigned owner[W];
#pragma unroll
  for (int s = 0; s < W; ++s) {
    row_free[s] = in[s] && sh.claim[MS_AT((int)named[s], N)] != (unsigned)(s * 32 + lane);
    if (in[s] && !row_free[s]) sh.x[s * 32 + lane] = (short)named[s];
    owner[s] = in[s] ? sh.claim[s * 32 + lane] : 0u;
  }
  __syncwarp();
  // the rows as the free columns see them: packed(-u, tag of the row), or just the tag
#pragma unroll
  for (int s = 0; s < W; ++s) {
    if (in[s]) {
      if (owner[s] != NONE) tag[s] = TAG_MATCHED | owner[s];
      const unsigned rt = (row_free[s] ? 0u : TAG_MATCHED) | (unsigned)(s * 32 + lane);
      sh.claim[s * 32 + lane] = WIDE ? rt : packed(-u[s], rt);
    }
  }
  __syncwarp();
  // ---- 2. free columns raise their duals ----
  // (Rows in flight: 16 instead of 4 with one-word keys of two words 317 -> 311 us for one plan of 16 matchings, of one word 592 x 16 ranks
  // 66.3 -> 63.7 us and 592 x 32 267 -> 256; below 16 ranks, where the rows go one by one then, 592 x 12 41.1 -> 42.2. 8 instead of as few as
  // the compiler took for entries beyond 23 bits 2.18 -> 2.10 ms, 60 x 72 ranks.)
  {
    int best[W];
    unsigned by[W];
    if constexpr (WIDE) {
#pragma unroll
      for (int s = 0; s < W; ++s) { best[s] = INF32; by[s] = NONE; }
#pragma unroll 8
      for (int i = 0; i < N; ++i) {
        const auto* row = R.row(i);
        const int ui = sh.urow[i];
        const unsigned ti = sh.claim[i];
#pragma unroll
        for (int s = 0; s < W; ++s) {
          const int t = -(int)(in[s] ? row[s * 32 + lane] : 0) - ui;
          if (t < best[s] || (t == best[s] && ti < by[s])) { best[s] = t; by[s] = ti; }
        }
      }
    } else {
      unsigned k[W];
#pragma unroll
      for (int s = 0; s < W; ++s) k[s] = NONE;
#pragma unroll (W <= 2 ? 16 : 4)
      for (int i = 0; i < N; ++i) {
        const auto* row = R.row(i);
        const unsigned from = sh.claim[i];
#pragma unroll
        for (int s = 0; s < W; ++s) k[s] = min(k[s], from - ((unsigned)(in[s] ? row[s * 32 + lane] : 0) << TAG_BITS));
      }
#pragma unroll
      for (int s = 0; s < W; ++s) {
        best[s] = packed_dist(k[s]);
        by[s] = k[s] & TAG_MASK;
      }
    }
    __syncwarp();
#pragma unroll
    for (int s = 0; s < W; ++s)
      if (in[s]) sh.claim[s * 32 + lane] = NONE;
    __syncwarp();
    bool asks[W];
#pragma unroll
    for (int s = 0; s < W; ++s) {
      const bool is_free = in[s] && tag[s] < TAG_MATCHED;
      if (is_free) v[s] = best[s];
      asks[s] = is_free && by[s] < TAG_MATCHED;
      if (asks[s]) atomicMin(&sh.claim[MS_AT((int)by[s], N)], (unsigned)(s * 32 + lane));
    }
    __syncwarp();
#pragma unroll
    for (int s = 0; s < W; ++s) {
      if (asks[s] && sh.claim[by[s]] == (unsigned)(s * 32 + lane)) {
        tag[s] = TAG_MATCHED | by[s];
        sh.x[by[s]] = (short)(s * 32 + lane);
      }
      if (in[s] && sh.claim[s * 32 + lane] != NONE) row_free[s] = false;
    }
  }
  unsigned left[W];
#pragma unroll
  for (int s = 0; s < W; ++s) left[s] = __ballot_sync(FULL, row_free[s]);
  work[WK_SKIP] += N;   // (rows left over are taken off again below)
  __syncwarp();
  // ---- 3. shortest augmenting paths ----
  while (any_bit<W>(left)) {
    const int f = first_of<W>(left);
    clear_bit<W>(left, f);
    work[WK_SKIP]--;
    work[WK_AUG]++;
    int pred[W], settled_at[W], mu;
    unsigned closed[W], who;   // closed: all ones for a settled column; who: tag of the column reached
#pragma unroll
    for (int s = 0; s < W; ++s) {
      pred[s] = f;
      settled_at[s] = 0;
      closed[s] = in[s] ? 0u : NONE;
    }
    // Candidates are keys, distance above tag. A settled column's key is all ones from then on; `closed` keeps new keys from
    // undercutting it. There is a free column as long as there is a free row, so a search always ends at one.
    unsigned key[W], k;
    const auto* first = R.row(MS_AT(f, N));
    const int off = sh.urow[MS_AT(f, N)];
    if constexpr (WIDE) {
#pragma unroll
      for (int s = 0; s < W; ++s)
        key[s] = (min((unsigned)(-(int)(in[s] ? first[s * 32 + lane] : 0) - v[s] - off), FAR) << TAG_BITS) | tag[s] | closed[s];
    } else {
#pragma unroll
      for (int s = 0; s < W; ++s) {
        base[s] = ((unsigned)-v[s] << TAG_BITS) + tag[s];
        key[s] = (base[s] + ((unsigned)(NARROW_BIAS - (in[s] ? (int)first[s * 32 + lane] : 0)) << TAG_BITS)) | closed[s];
      }
    }
    // AHEAD: the row is asked for before it is known whether the search goes on (a free column's number is a row's number
    // too), so that the load and the test overlap: 148 x 256 ranks 42.9 -> 36.5 ms, 20 x 200 ranks 61.1 -> 54.4 ms, 1024 x 16 ranks
    // 99 -> 95 us; with two words (4.8 -> 5.3 ms, 4096 x 64 ranks) and four (20.6 -> 22.1 ms, 1024 x 128) it does not pay.
    // With two or three words the whole row is asked for after the test, then used: 4.83 -> 4.56 ms, one plan of 16 matchings
    // 415 -> 389 us; with four to six that costs registers (20.1 -> 20.9 ms), and asking ahead is no better there (100 x 160 ranks
    // 8.3 -> 9.1 ms).
    constexpr bool AHEAD = W == 1 || W > 6;
    while (true) {   // every scan settles one more column
      k = key[0];
#pragma unroll
      for (int s = 1; s < W; ++s) k = min(k, key[s]);
      k = __reduce_min_sync(FULL, k);
      work[WK_SCAN]++;
      const int i = MS_AT((int)(AHEAD ? min(k & 0xffu, (unsigned)(N - 1)) : k & 0xffu), N);   // (no row if k is NONE)
      const auto* row = R.row(i);
      int ui, entry[W];
      auto fetch = [&] {   // (the empty statements keep the loads where they are)
        ui = sh.urow[i];
        asm volatile("" : "+r"(ui));
#pragma unroll
        for (int s = 0; s < W; ++s) entry[s] = in[s] ? (int)row[s * 32 + lane] : 0;
#pragma unroll
        for (int s = 0; s < W; ++s) asm volatile("" : "+r"(entry[s]));
      };
      if constexpr (AHEAD) fetch();
      if ((k & TAG_MATCHED) == 0u || k >= (WIDE ? FAR << TAG_BITS : NONE)) break;
      if constexpr (W == 2 || W == 3) fetch();
      if constexpr (W >= 4 && W <= 6) ui = sh.urow[i];
#pragma unroll
      for (int s = 0; s < W; ++s) {
        if (key[s] == k) {   // (rows differ, so only the settled column has this key)
          settled_at[s] = (int)(k >> TAG_BITS);
          key[s] = closed[s] = NONE;
        }
        if constexpr (W >= 4 && W <= 6) entry[s] = in[s] ? (int)row[s * 32 + lane] : 0;
        unsigned nk;
        if constexpr (WIDE)
          nk = (min((unsigned)((int)(k >> TAG_BITS) - v[s] - ui - entry[s]), FAR) << TAG_BITS) | tag[s] | closed[s];
        else
          nk = ((k & ~TAG_MASK) + base[s] - ((unsigned)ui << TAG_BITS) - ((unsigned)entry[s] << TAG_BITS)) | closed[s];
        if (nk < key[s]) pred[s] = i;
        key[s] = min(key[s], nk);
      }
    }
    who = k & TAG_MASK;
    mu = (int)(k >> TAG_BITS);
    if constexpr (!WIDE) {
      if (k == NONE) return false;
      mu -= NARROW_BIAS;
#pragma unroll
      for (int s = 0; s < W; ++s) settled_at[s] -= NARROW_BIAS;
    } else {
      mu += off;
#pragma unroll
      for (int s = 0; s < W; ++s) settled_at[s] += off;
      if (k >= FAR << TAG_BITS) {   // too far for a key
        int d[W];
#pragma unroll
        for (int s = 0; s < W; ++s) {
          pred[s] = f;
          closed[s] = in[s] ? 0u : NONE;
          d[s] = in[s] ? -(int)first[s * 32 + lane] - v[s] : INF32;
        }
        while (true) {   // every scan settles one more column
          nearest<W>(d, tag, mu, who);
          work[WK_SCAN]++;
          if (mu == INF32) return false;
          if (who < TAG_MATCHED) break;
          const int i = MS_AT((int)(who & 0xffu), N);
          const auto* row = R.row(i);
          const int h = sh.urow[i] - mu;
#pragma unroll
          for (int s = 0; s < W; ++s) {
            if (tag[s] == who) {
              closed[s] = NONE;
              settled_at[s] = mu;
              d[s] = INF32;
            }
            if (closed[s] == 0u) {
              const int nd = -(int)row[s * 32 + lane] - v[s] - h;
              if (nd < d[s]) { d[s] = nd; pred[s] = i; }
            }
          }
        }
      }
    }
    int j = MS_AT((int)who, N);
    // (Loads first, stores when they have come back, and the next step of the path is on its way before it is known whether there is
    // one: an augmentation costs 400 instead of 700 cycles at N = 64. One plan of 16 matchings 357 -> 323 us, 1024 x 128 ranks 17.9 ->
    // 16.2 ms, 256 x 256 ranks 65.4 -> 63.5 ms. The flip names the rows of its columns itself: 323 -> 319 us, 16.2 -> 16.0, 63.5 -> 62.6;
    // only entries beyond 23 bits lose, 60 x 72 ranks 2.16 -> 2.25 ms.)
    int at[W], ud[W];
#pragma unroll
    for (int s = 0; s < W; ++s) {
      at[s] = in[s] ? (int)sh.x[MS_AT(pred[s], N)] : 0;
      ud[s] = in[s] ? sh.urow[tag[s] & 0xffu] : 0;   // (of no interest for a free column)
    }
#pragma unroll
    for (int s = 0; s < W; ++s)
      if (in[s]) sh.pred[s * 32 + lane] = (unsigned)pred[s] | (unsigned)(pred[s] == f ? 0 : at[s]) << 16;
    __syncwarp();   // (also: the scans have read the row duals)
    unsigned back = sh.pred[j];
    // settled columns move their dual so that the shortest-path tree stays tight, and their rows' duals with them
#pragma unroll
    for (int s = 0; s < W; ++s) {
      if (in[s] && closed[s] != 0u) {
        v[s] += settled_at[s] - mu;
        sh.urow[tag[s] & 0xffu] = ud[s] + mu - settled_at[s];
      }
    }
    sh.urow[f] = mu;   // every lane
    // flip the path back to row f (every lane makes every update)
    for (int it = 0; it <= N; ++it) {
      const int i = MS_AT((int)(back & 0xffffu), N), before = MS_AT((int)(back >> 16), N);
      back = sh.pred[before];
      sh.x[i] = (short)j;
#pragma unroll
      for (int s = 0; s < W; ++s) tag[s] = j == s * 32 + lane ? TAG_MATCHED | (unsigned)i : tag[s];
      if (i == f) break;
      j = before;
    }
    __syncwarp();
  }
  return true;
}

// Tight edges under the optimal duals, row by row into the position table: entry (r, c) is tight iff its reduced cost
// equals the row's dual. One vote per 32 columns gives a row's edges as a set. highest: the highest row adjacent to each of
// the lane's columns.
template <int W, int STORE>
__device__ __forceinline__ void tight_graph(const Residual<STORE>& R, int N, int lane, const AssignShared& sh,
                                            const int (&v)[W], const PosTable<W>& tab, int (&highest)[W]) {
#pragma unroll
  for (int s = 0; s < W; ++s) highest[s] = -1;
  // Several at a time (the last one again beyond the end), all sums before the first vote: 1024 x 16 ranks 95 -> 90 us.
  constexpr int ROWS = W <= 4 ? 8 : 4;
  for (int r0 = 0; r0 < N; r0 += ROWS) {
    PosEntry<W> e[ROWS];
    int at[ROWS], sum[ROWS][W];
#pragma unroll
    for (int q = 0; q < ROWS; ++q) {
      const int r = min(r0 + q, N - 1);
      const auto* row = R.row(r);
      const int ur = sh.urow[r];
      e[q].row8 = (unsigned)r << 8;
      at[q] = MS_AT((int)sh.x[r], N);
#pragma unroll
      for (int s = 0; s < W; ++s) {
        const int c = s * 32 + lane;
        sum[q][s] = c < N ? (int)row[c] + v[s] + ur : 1;
        if (sum[q][s] == 0) highest[s] = r;
      }
    }
#pragma unroll
    for (int q = 0; q < ROWS; ++q) {
#pragma unroll
      for (int s = 0; s < W; ++s) e[q].a[s] = __ballot_sync(FULL, sum[q][s] == 0);
    }
#pragma unroll
    for (int q = 0; q < ROWS; ++q) tab.store(at[q], e[q]);
  }
  __syncwarp();
}

// STORE 2 leaves a matrix with entries beyond 16 bits alone, its status marked CLASS_I32, for a launch with another STORE
// and only_class set, which handles nothing else.
// COUNT: the per-matrix work counters are wanted (register increments the compiler drops otherwise).
template <int W, int STORE, bool COUNT>
__global__ void __launch_bounds__(128) mw_kernel(int B, int N, const int32_t* __restrict__ demand, int k_max,
                                                 uint8_t* __restrict__ perm, int32_t* __restrict__ dur,
                                                 int32_t* __restrict__ count, int32_t* __restrict__ residual,
                                                 int32_t* status, long long* __restrict__ work_out, int only_class) {
  constexpr bool CLUSTER = STORE == 1;
  using T = typename Residual<STORE>::T;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b = CLUSTER ? (int)(blockIdx.x >> 1) : (int)(blockIdx.x * (blockDim.x >> 5) + warp);
  if (b >= B) return;   // (a cluster grid has exactly two CTAs per matrix)
  if (only_class != 0 && status[b] != only_class) return;   // both CTAs of a cluster see the same class
  Residual<STORE> R;
  R.N = N;
  R.split = CLUSTER ? (N + 1) / 2 : N;
  const size_t mat_bytes = align16((size_t)R.split * N * sizeof(T));
  unsigned char* base = smem_raw + (size_t)warp * (mat_bytes + state_smem_bytes(N, W));
  R.near_ = R.far_ = reinterpret_cast<T*>(base);
  Peeler<W, int, false> pl;
  pl.reset(base + mat_bytes, N, lane);
  const AssignShared sh = assign_shared(base + mat_bytes + (W == 8 ? table_bytes(N, W) : peel_smem_bytes(N, W)), N);
  if constexpr (CLUSTER) {
    R.far_ = reinterpret_cast<T*>(map_to_cta(reinterpret_cast<int*>(R.near_), 1));
    cluster_sync_all();
    if (cluster_ctarank() != 0) { cluster_epilogue<true>(); return; }   // lends its shared memory until the end
  }

  unsigned work[MOESCHED_WORK_FIELDS];
#pragma unroll
  for (int q = 0; q < MOESCHED_WORK_FIELDS; ++q) work[q] = 0u;

  // ---- matrix into shared memory; validate, find the largest entry, count the non-zero entries ----
  int nnz = 0, mx = 0;
  {
    const int32_t* D = demand + (size_t)b * N * N;
    int neg = 0;
#pragma unroll
    for (int s = 0; s < W; ++s) {
      const int c = s * 32 + lane;
      if (c < N) {
#pragma unroll 8
        for (int r = 0; r < N; ++r) {
          const int val = D[(size_t)r * N + c];
          neg |= val < 0;
          mx = max(mx, val);
          nnz += val != 0;
          R.row(r)[c] = (T)val;
        }
      }
    }
    neg = __any_sync(FULL, neg);
    mx = neg ? INF32 : __reduce_max_sync(FULL, mx);
    nnz = __reduce_add_sync(FULL, nnz);
    __syncwarp();
    if (STORE == 2 && mx > 65535) {
      if (lane == 0) status[b] = CLASS_I32;
      return;
    }
  }
  int st_code = mx > MOESCHED_MW_MAX_ENTRY ? MOESCHED_ST_BAD_INPUT : MOESCHED_ST_OK;
  int k = 0;

  if (st_code == MOESCHED_ST_OK) {
    const bool wide = STORE != 2 && mx > NARROW_MAX_ENTRY;
    int v[W];
#pragma unroll
    for (int s = 0; s < W; ++s) v[s] = 0;
    uint8_t* pout = perm + (size_t)b * k_max * N;
    int32_t* dout = dur + (size_t)b * k_max;
    while (k < k_max && nnz > 0) {
      bool ok;
      if (wide) ok = solve_assignment<W, STORE, STORE != 2>(R, N, lane, sh, v, work);
      else ok = solve_assignment<W, STORE, false>(R, N, lane, sh, v, work);
      if (!ok) { st_code = MOESCHED_ST_INTERNAL; break; }
      int highest[W];
      tight_graph<W, STORE>(R, N, lane, sh, v, pl.tab, highest);
      unsigned left[W];
      pl.adopt(highest, left);
      pl.canonicalise(0u, left, work);
      // serve: the heaviest matched pair sets the duration; matched entries are sent whole
      int dmax = 0, served = 0;
#pragma unroll
      for (int s = 0; s < W; ++s) {
        if (pl.valid(s)) {
          const int r = MS_AT((int)(pl.key[s] >> 8), N);
          T* p = R.row(r) + s * 32 + lane;
          const int val = *p;
          dmax = max(dmax, val);
          served += val != 0;
          *p = (T)0;
          pout[r] = (uint8_t)(s * 32 + lane);
        }
      }
      dmax = __reduce_max_sync(FULL, dmax);
      nnz -= __reduce_add_sync(FULL, served);
      if (lane == 0) dout[k] = dmax;
      __syncwarp();
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
  if (residual != nullptr && st_code != MOESCHED_ST_BAD_INPUT) {
    int32_t* ro = residual + (size_t)b * N * N;
    for (int r = 0; r < N; ++r) {
      const T* rp = R.row(r);
      for (int c = lane; c < N; c += 32) ro[(size_t)r * N + c] = rp[c];
    }
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

static size_t mw_smem_per_warp(int N, int W, int store) {
  const int rows = store == 1 ? (N + 1) / 2 : N;
  return align16((size_t)rows * N * (store == 2 ? 2 : 4)) + state_smem_bytes(N, W);
}

template <int STORE>
static cudaError_t launch_mw(int B, int N, const int32_t* demand, int k_max, uint8_t* perm, int32_t* dur,
                             int32_t* count, int32_t* residual, int32_t* status, long long* work, int only_class,
                             cudaStream_t stream) {
  Geometry ge = plan_geometry(N);
  ge.cluster = STORE == 1;
  ge.wpb = STORE == 0 && N <= 32 ? 4 : 1;   // several small matrices share a CTA so that an SM can hold 64 warps
  ge.smem = mw_smem_per_warp(N, ge.cpl, STORE) * ge.wpb;
#define MOESCHED_GO(C)                                                                                             \
  do {                                                                                                             \
    if (work != nullptr)                                                                                           \
      return launch_warp_kernel(mw_kernel<C, STORE, true>, ge, B, stream, B, N, demand, k_max, perm, dur, count,   \
                                residual, status, work, only_class);                                               \
    return launch_warp_kernel(mw_kernel<C, STORE, false>, ge, B, stream, B, N, demand, k_max, perm, dur, count,    \
                              residual, status, work, only_class);                                                 \
  } while (0)
  if constexpr (STORE == 1) {
    MOESCHED_GO(8);
  } else {
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
  }
#undef MOESCHED_GO
}

cudaError_t run_mw(int B, int N, const int32_t* demand, int k_max, uint8_t* perm, int32_t* dur, int32_t* count,
                   int32_t* residual, int32_t* status, long long* work, cudaStream_t stream) {
  const size_t as_int32 = mw_smem_per_warp(N, plan_geometry(N).cpl, 0);
  // Shared memory limits how many matrices an SM holds. Where all of them fit half of it as int32 (the Birkhoff kernel often
  // runs beside), one launch takes every matrix; otherwise they are held as 16-bit entries, and a second launch takes those that do not fit (as int32,
  // over a 2-CTA cluster where one CTA cannot hold the matrix).
  if (N <= 32 || (as_int32 <= SMEM_LIMIT && (size_t)((B + sm_count() - 1) / sm_count()) * (as_int32 + 1024) <= SMEM_LIMIT / 2))
    return launch_mw<0>(B, N, demand, k_max, perm, dur, count, residual, status, work, 0, stream);
  cudaError_t e = launch_mw<2>(B, N, demand, k_max, perm, dur, count, residual, status, work, 0, stream);
  if (e != cudaSuccess) return e;
  if (as_int32 > SMEM_LIMIT)
    return launch_mw<1>(B, N, demand, k_max, perm, dur, count, residual, status, work, CLASS_I32, stream);
  return launch_mw<0>(B, N, demand, k_max, perm, dur, count, residual, status, work, CLASS_I32, stream);
}

}  // namespace moesched
