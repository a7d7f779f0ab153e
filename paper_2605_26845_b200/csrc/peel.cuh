// One warp peels perfect matchings off one matrix (the Birkhoff-von Neumann loop, paper Sec. 3.1): the matching, its
// support graph and the searches that keep the matching lexicographically smallest. Shared by the integer and the
// real-valued decomposition.
//
// Layout. Column c is "position" c: lane c % 32, slot c / 32 of the warp. A position holds the ROW matched to its
// column: the row's number, the columns the row is adjacent to (a bit mask of W words), and the value of the matched
// entry. A set of positions is therefore a set of columns and a set of rows at once, and one vote per slot turns
// "which lanes qualify" into that set in every lane's registers:
//   * a search level -- which rows are adjacent to a column of the frontier -- is W AND-ORs and one vote per slot, with
//     no reduction over the warp (a vote costs a quarter of a reduction);
//   * the lowest column a row may take is the lowest bit of (its adjacency & the set reached): no search over lanes;
//   * a search record (the set of rows that could reach the searched one) stays with the position and is void as soon
//     as one of its positions changes hands.
// When a row moves to another column its mask and number move to another lane: a table in shared memory (one entry
// per position, rewritten by every lane with the same values, so that a lane reads back its own stores) makes them
// available to all lanes with one vector load. An entry is overwritten only once every lane has read what it held: a
// vote keeps the lanes together but orders no memory, so shift(), exchange() and drop_edges() begin with a warp barrier
// (three matrices of N = 100 41.3 -> 41.8 ms; barrier and stores at their end 42.0).
// (What a search leaves in the history is likewise read before the rows are moved, and so before the next search.)
// The matched values live in registers; the matrix in memory is touched only where a row moves (the value of the pair
// that is given up goes back, the value of the new pair is fetched, and is not needed before the end of the step).
// Against a layout that keeps, per column, the set of adjacent rows (rows stay where they are, a level needs an
// OR-reduction per word, every choice of a column a minimum over the warp): see bvn_kernel.cu for the times.
#pragma once

#include "common.cuh"

namespace moesched {

// ---- sets of positions ------------------------------------------------------------------------

// 1 << n, and 0 for n outside 0 .. 31 (the shift of the machine clamps; the language leaves it open)
__device__ __forceinline__ unsigned one_shl(int n) {
#ifdef __CUDACC__
  unsigned r;
  asm("shl.b32 %0, 1, %1;" : "=r"(r) : "r"(n));
  return r;
#else   // (the CPU tests)
  return n < 0 || n > 31 ? 0u : 1u << n;
#endif
}
template <int W>
__device__ __forceinline__ void single_mask(int q, unsigned (&m)[W]) {
#pragma unroll
  for (int w = 0; w < W; ++w) m[w] = one_shl(q - 32 * w);
}
// The lowest member of a non-empty set, as a set and as a number. (Isolating the bit and asking for the position of the
// highest one is one slow operation; reversing the word and counting zeros would be two.)
template <int W>
__device__ __forceinline__ int first_of(const unsigned (&m)[W], unsigned (&single)[W]) {
  unsigned v = m[W - 1];
  int base = (W - 1) * 32;
#pragma unroll
  for (int k = W - 2; k >= 0; --k) {
    base = m[k] != 0u ? k * 32 : base;
    v = m[k] != 0u ? m[k] : v;
  }
  v &= 0u - v;
#pragma unroll
  for (int w = 0; w < W; ++w) single[w] = base == w * 32 ? v : 0u;
  return base + 31 - __clz(v);
}
template <int W>
__device__ __forceinline__ int first_of(const unsigned (&m)[W]) {
  unsigned ignored[W];
  return first_of<W>(m, ignored);
}
// the set {0 .. q-1} from the set {q}
template <int W>
__device__ __forceinline__ void below_mask(const unsigned (&single)[W], unsigned (&m)[W]) {
  if constexpr (W == 2) {
    const unsigned long long v = as64(single) - 1ull;
    m[0] = (unsigned)v;
    m[1] = (unsigned)(v >> 32);
  } else {
    bool above = false;   // a lower word holds q
#pragma unroll
    for (int w = 0; w < W; ++w) {
      m[w] = above ? 0u : single[w] - 1u;
      above = above || single[w] != 0u;
    }
  }
}

// ---- the position table -----------------------------------------------------------------------

// A row as the searches see it. Row numbers are kept shifted left by 8, so that row | position is one sortable word.
template <int W>
struct PosEntry {
  unsigned a[W];   // columns adjacent to the row
  unsigned row8;   // row << 8
};
// With eight words the row numbers lie apart, behind the masks: a padded entry would take 48 bytes, and a matrix of 230 to 232
// ranks held as int32 next to the table would no longer fit one CTA (148 greedy ones of 232 ranks 55.8 -> 76.6 ms over two).
__host__ __device__ constexpr int table_words(int W) { return W == 1 ? 2 : W == 8 ? 8 : (W + 4) / 4 * 4; }   // per entry
__host__ __device__ inline size_t table_bytes(int N, int W) {
  return align16((size_t)N * table_words(W) * 4) + (W == 8 ? align16((size_t)N * 4) : 0);
}
template <int W>
struct PosTable {
  static constexpr int WORDS = table_words(W);
  static constexpr int WHOLE = W / 4 * 4;   // words of the mask that fill groups of 16 bytes
  unsigned* base;
  unsigned* rows;   // eight words only
  __device__ __forceinline__ PosEntry<W> load(int q) const {
    const unsigned* p = base + q * WORDS;
    PosEntry<W> e;
    if constexpr (W == 1) {
      const uint2 v = *reinterpret_cast<const uint2*>(p);
      e.a[0] = v.x; e.row8 = v.y;
    } else {
#pragma unroll
      for (int k = 0; k < WHOLE; k += 4) {
        const uint4 v = *reinterpret_cast<const uint4*>(p + k);
        e.a[k] = v.x; e.a[k + 1] = v.y; e.a[k + 2] = v.z; e.a[k + 3] = v.w;
      }
      if constexpr (W == 8) {
        e.row8 = rows[q];
      } else if constexpr (W % 4 == 0) {
        e.row8 = p[W];
      } else if constexpr (W % 4 == 1) {
        const uint2 v = *reinterpret_cast<const uint2*>(p + WHOLE);
        e.a[WHOLE] = v.x; e.row8 = v.y;
      } else {
        const uint4 v = *reinterpret_cast<const uint4*>(p + WHOLE);
        e.a[WHOLE] = v.x; e.a[WHOLE + 1] = v.y;
        if constexpr (W % 4 == 3) { e.a[WHOLE + 2] = v.z; e.row8 = v.w; }
        else e.row8 = v.z;
      }
    }
    return e;
  }
  // every lane stores the same entry
  __device__ __forceinline__ void store(int q, const PosEntry<W>& e) const {
    unsigned* p = base + q * WORDS;
    if constexpr (W == 1) {
      *reinterpret_cast<uint2*>(p) = make_uint2(e.a[0], e.row8);
    } else {
#pragma unroll
      for (int k = 0; k < WHOLE; k += 4)
        *reinterpret_cast<uint4*>(p + k) = make_uint4(e.a[k], e.a[k + 1], e.a[k + 2], e.a[k + 3]);
      if constexpr (W == 8) rows[q] = e.row8;
      else if constexpr (W % 4 == 0) p[W] = e.row8;
      else if constexpr (W % 4 == 1) *reinterpret_cast<uint2*>(p + WHOLE) = make_uint2(e.a[WHOLE], e.row8);
      else if constexpr (W % 4 == 2) *reinterpret_cast<uint4*>(p + WHOLE) = make_uint4(e.a[WHOLE], e.a[WHOLE + 1], e.row8, 0u);
      else *reinterpret_cast<uint4*>(p + WHOLE) = make_uint4(e.a[WHOLE], e.a[WHOLE + 1], e.a[WHOLE + 2], e.row8);
    }
  }
};

// Shared memory of one warp: position table, then the search levels (0 .. N).
__host__ __device__ inline size_t peel_smem_bytes(int N, int W) {
  return table_bytes(N, W) + align16((size_t)(N + 1) * W * 4);
}

// The matrix in memory: rows [0, split) at near_, the rest in the partner CTA of a cluster (CLUSTER only).
template <typename V, bool CLUSTER>
struct PeelMatrix {
  V* near_;
  V* far_;
  int S, split;
  __device__ __forceinline__ V* cell(int r, int c) const {
    if constexpr (CLUSTER) return (r < split ? near_ + r * S : far_ + (r - split) * S) + c;
    else return near_ + (r * S + c);
  }
};

template <int W, typename V, bool CLUSTER>
struct Peeler {
  int N, lane;
  PeelMatrix<V, CLUSTER> mem;
  PosTable<W> tab;
  unsigned* hist;
  unsigned key[W];      // row at the lane's position s, and the position: row << 8 | position; 0 beyond N
  unsigned A[W][W];     // A[s]: columns adjacent to that row
  V val[W];             // value of the entry of row vrow[s] in the lane's column s
  int vrow[W];
  // Lower columns that the row is adjacent to and that hold a higher row: how many there are (a row with none cannot move
  // to a lower column). Negative: searched in vain; `rec` holds the rows that could reach it, and it cannot move before
  // one of them has moved. UNKNOWN and more: such a record has become void.
  int chance[W];
  unsigned rec[W][W];
  unsigned broken[W];   // positions whose pair is nominal only: the column is free and the row has lost its entry
  int broken_count;
  static constexpr int UNKNOWN = 1 << 16, IN_VAIN = -(1 << 16);

  __device__ __forceinline__ bool valid(int s) const { return s * 32 + lane < N; }
  // whether the lane's position s is in the set
  __device__ __forceinline__ bool mine(const unsigned (&set)[W], int s) const { return (set[s] & (1u << lane)) != 0u; }

  // Up to six words, the tests of all words are evaluated before the first vote, so that the votes follow one another and
  // their latencies overlap, in place of a test and a vote in turn: one matrix of N = 64 8.13 -> 7.84 ms, three of N = 100
  // 41.0 -> 39.7, 1024 of N = 128 18.7 -> 18.4, 100 of N = 160 13.4 -> 12.0. (With eight words, what this keeps alive costs more: 33.5 -> 34.7.)
  static constexpr bool VOTES_LAST = W <= 6;
  // A row that has moved is read back from the table by the lane that it has moved to. Up to six words, where the row is needed again
  // sooner than the load returns, that lane selects it from the copy that all lanes have. (Selecting, with seven and eight words:
  // 100 of N = 224 334 ms, reading back 307; 256 of N = 256 531 and 530; with two words 10.6 and 11.9 for 1024 of N = 64.)
  static constexpr bool RELOAD = W >= 7;
  // The chances of a row that has moved are counted, or it is just looked at when its turn comes: a look in vain costs the same few
  // operations per word for any W, counting grows with it (100 of N = 160 158.6 -> 154.7 ms, 100 of N = 192 171.4 -> 168.9, 256 of
  // N = 256 530 -> 520, but one of N = 64 7.48 -> 7.75; with four words there is nothing in it).
  static constexpr bool COUNTED = W <= 4;
  // A branch that all lanes take together costs about 20 cycles of the chain, so the ways out of a search lead straight to what comes
  // next instead of through a common test (one of N = 64 7.84 -> 7.47 ms, 4096 27.1 -> 25.9, 256 of N = 256 530 -> 514). Likewise:
  // the first level, where 67 % of the searches of 16 ranks, 44 % of 64 and 31 % of 128 end, is taken apart and followed by the exchange
  // (1024 of N = 16 271 -> 267 us, one of N = 64 7.47 -> 7.24 ms, 148 of N = 96 27.1 -> 26.4, 100 of N = 192 168.9 -> 165.3; 1024 of N = 128
  // 123.7 -> 124.9; with eight words the code that this adds costs more: 514 -> 581);
  static constexpr bool FIRST_APART = W <= 6;
  // a first level without members has a way of its own (267 -> 261 us, 4096 of N = 64 26.0 -> 25.7 ms; 100 of N = 160 153.9 -> 158.3);
  static constexpr bool NONE_APART = W <= 2;
  // the lowest column wanted is found before it is known whether there is one (one of N = 64 7.20 -> 7.18 ms, 1024 10.48 -> 10.41, 148
  // of N = 96 26.5 -> 26.4, 1024 of N = 128 124.9 -> 123.5; 1024 of N = 16 261 -> 265 us, 100 of N = 160 153.8 -> 157.8 ms).
  static constexpr bool WANT_EARLY = W >= 2 && W <= 4;

  // positions whose row is higher than that of key k
  __device__ __forceinline__ void rows_above(unsigned k, unsigned (&out)[W]) const {
    bool yes[W];
#pragma unroll
    for (int s = 0; s < W; ++s) {
      yes[s] = key[s] > (k | 0xffu);
      if (!VOTES_LAST) out[s] = __ballot_sync(FULL, yes[s]);
    }
    if (VOTES_LAST) {
#pragma unroll
      for (int s = 0; s < W; ++s) out[s] = __ballot_sync(FULL, yes[s]);
    }
  }

  __device__ __forceinline__ void reset(unsigned char* smem, int N_, int lane_) {
    N = N_;
    lane = lane_;
    tab.base = reinterpret_cast<unsigned*>(smem);
    tab.rows = tab.base + (size_t)N * PosTable<W>::WORDS;
    hist = reinterpret_cast<unsigned*>(smem + table_bytes(N, W));
    broken_count = N;
#pragma unroll
    for (int s = 0; s < W; ++s) {
      key[s] = 0u;
      val[s] = V(0);
      vrow[s] = 0;
      broken[s] = N >= (s + 1) * 32 ? 0xffffffffu : (N <= s * 32 ? 0u : (1u << (N - s * 32)) - 1u);
      chance[s] = valid(s) ? 0 : IN_VAIN;
#pragma unroll
      for (int w = 0; w < W; ++w) A[s][w] = rec[s][w] = 0u;
    }
  }

  // Row r with adjacency e.a starts out at the position of its own number (so every lower position holds a lower row: no
  // chances); the pair is nominal until it is repaired.
  __device__ __forceinline__ void seat(int r, const PosEntry<W>& e) {
    tab.store(r, e);
#pragma unroll
    for (int s = 0; s < W; ++s) {
      if (r == s * 32 + lane) {
        key[s] = (unsigned)(r << 8 | r);
        vrow[s] = r;
        val[s] = *mem.cell(r, r);
#pragma unroll
        for (int w = 0; w < W; ++w) A[s][w] = e.a[w];
      }
    }
  }

  // Takes over a complete matching from the table, as the graph of a new problem. A row cannot move unless a row above it
  // (highest: the highest one adjacent to the lane's column) could take its column. Nor can it unless it lies on a cycle: rows
  // that are adjacent to no column but their own leave the graph, then those that were adjacent to the columns of these alone,
  // and so on. What is `left` holds all cycles, and a rotation moves rows within it only. (The tight edges of a greedy step are
  // hardly more than a tree, and nearly all searches were in vain. N = 64: 12 passes and 7 search levels instead of 39 levels,
  // one plan of 16 matchings 395 -> 358 us, 1024 x 128 ranks 20.0 -> 17.8 ms.)
  __device__ __forceinline__ void adopt(const int (&highest)[W], unsigned (&left)[W]) {
    broken_count = 0;
    const unsigned low = (1u << lane) - 1u;
#pragma unroll
    for (int s = 0; s < W; ++s) {
      key[s] = 0u;
      chance[s] = IN_VAIN;
#pragma unroll
      for (int w = 0; w < W; ++w) A[s][w] = rec[s][w] = 0u;
      if (valid(s)) {
        const PosEntry<W> e = tab.load(s * 32 + lane);
        key[s] = e.row8 | (unsigned)(s * 32 + lane);
        unsigned lower = e.a[s] & low;
#pragma unroll
        for (int w = 0; w < W; ++w) {
          A[s][w] = e.a[w];
          if (w < s) lower |= e.a[w];
        }
        chance[s] = highest[s] <= (int)(e.row8 >> 8) ? IN_VAIN : lower != 0u ? UNKNOWN : 0;
      }
      left[s] = 0xffffffffu;   // (columns beyond N are adjacent to no row)
    }
    __syncwarp();
    unsigned gone = 1u;
    // (If no row may move, there is nothing to keep from being searched: a vote that pays with one word, where hardly a step of few
    // ranks has such a row, 64 x 2 ranks 4.07 -> 3.79 us, two matchings; with three 994 -> 1035, 592 x 96.)
    if constexpr (W == 1) gone = __ballot_sync(FULL, chance[0] > 0);
    while (gone != 0u) {   // every pass takes a row out of `left`
      gone = 0u;
#pragma unroll
      for (int s = 0; s < W; ++s) {
        unsigned o = A[s][s] & left[s] & ~(1u << lane);
#pragma unroll
        for (int w = 0; w < W; ++w)
          if (w != s) o |= A[s][w] & left[w];
        const unsigned stay = __ballot_sync(FULL, o != 0u) & left[s];
        gone |= stay ^ left[s];
        left[s] = stay;
      }
    }
#pragma unroll
    for (int s = 0; s < W; ++s)
      if (!mine(left, s)) chance[s] = IN_VAIN;
  }

  // reaches[s]: the row at position s is adjacent to column q (single: the set {q}), which lies below its own.
  __device__ __forceinline__ void adjacent_from_above(const unsigned (&single)[W], bool (&reaches)[W]) const {
    const unsigned low = (1u << lane) - 1u;
#pragma unroll
    for (int s = 0; s < W; ++s) {
      unsigned t = A[s][s] & single[s] & low;
#pragma unroll
      for (int w = 0; w < s; ++w) t |= A[s][w] & single[w];
      reaches[s] = t != 0u;
    }
  }
  // The owners of the positions of a set take over what the table says.
  __device__ __forceinline__ void reload(const unsigned (&set)[W]) {
#pragma unroll
    for (int s = 0; s < W; ++s) {
      if (mine(set, s)) {
        const PosEntry<W> e = tab.load(s * 32 + lane);
        key[s] = e.row8 | (unsigned)(s * 32 + lane);
#pragma unroll
        for (int w = 0; w < W; ++w) A[s][w] = e.a[w];
      }
    }
  }
  // The owner of position q (single: the set {q}) takes over row e.
  __device__ __forceinline__ void settle(const unsigned (&single)[W], const PosEntry<W>& e, int its_chance) {
#pragma unroll
    for (int s = 0; s < W; ++s) {
      if (mine(single, s)) {
        key[s] = e.row8 | (unsigned)(s * 32 + lane);
        chance[s] = its_chance;
#pragma unroll
        for (int w = 0; w < W; ++w) A[s][w] = e.a[w];
      }
    }
  }

  // Row e takes column q (single: the set {q}) from row old8 >> 8: the table, the owner's registers, and the chances of
  // the rows between the two that are adjacent to q and sit above it.
  __device__ __forceinline__ void shift(int q, const unsigned (&single)[W], const PosEntry<W>& e, unsigned old8) {
    __syncwarp();   // the entry of q, and the levels that led there, have been read
    tab.store(q, e);
    const unsigned now = e.row8 | 0xffu, before = old8 | 0xffu;
    const int change = e.row8 > old8 ? 1 : -1;
    unsigned under[W];
    below_mask<W>(single, under);
    bool reaches[W];
    adjacent_from_above(single, reaches);
    int own = COUNTED ? 0 : UNKNOWN;
    unsigned higher[W];
    if (VOTES_LAST && COUNTED) rows_above(now, higher);
#pragma unroll
    for (int s = 0; s < W; ++s) {
      const bool above = key[s] > now;
      if (reaches[s] && above != (key[s] > before)) chance[s] += change;
      if constexpr (COUNTED) own += __popc((VOTES_LAST ? higher[s] : __ballot_sync(FULL, above)) & e.a[s] & under[s]);
    }
    if constexpr (RELOAD) {
      reload(single);
#pragma unroll
      for (int s = 0; s < W; ++s)
        if (mine(single, s)) chance[s] = own;
    } else {
      settle(single, e, own);
    }
  }

  // One search level: the positions of `alive` whose row is adjacent to a column of F become the new F. Returns the new
  // members ORed together.
  __device__ __forceinline__ unsigned grow(unsigned (&F)[W], unsigned (&alive)[W]) const {
    unsigned b[W];
    bool yes[W];
#pragma unroll
    for (int s = 0; s < W; ++s) {
      unsigned o = 0u;
#pragma unroll
      for (int w = 0; w < W; ++w) o |= A[s][w] & F[w];
      yes[s] = o != 0u;
      if (!VOTES_LAST) b[s] = __ballot_sync(FULL, yes[s]);
    }
    if (VOTES_LAST) {
#pragma unroll
      for (int s = 0; s < W; ++s) b[s] = __ballot_sync(FULL, yes[s]);
    }
    unsigned any = 0u;
#pragma unroll
    for (int s = 0; s < W; ++s) {
      F[s] = b[s] & alive[s];
      alive[s] &= ~b[s];
      any |= F[s];
    }
    return any;
  }

  // Row i (entry e at position p, single: root) and row u (entry f at position q, single: target), i below u, change
  // places: what a walk of one step comes to, and most walks are. `settled`: no column below q that row i is adjacent to
  // holds a row above it.
  __device__ __forceinline__ void exchange(int p, const unsigned (&root)[W], const PosEntry<W>& e, int q,
                                           const unsigned (&target)[W], const PosEntry<W>& f, bool settled = true) {
    __syncwarp();   // both entries, and the levels that led there, have been read
    tab.store(q, e);
    tab.store(p, f);
    const unsigned ki = e.row8 | 0xffu, ku = f.row8 | 0xffu;
    unsigned under[W];
    below_mask<W>(root, under);
    bool reaches_p[W], reaches_q[W];
    adjacent_from_above(root, reaches_p);
    adjacent_from_above(target, reaches_q);
    int own = COUNTED ? 0 : UNKNOWN;
    unsigned higher[W];
    if (VOTES_LAST && COUNTED) rows_above(ku, higher);
#pragma unroll
    for (int s = 0; s < W; ++s) {
      const bool above = key[s] > ku;
      if constexpr (COUNTED) own += __popc((VOTES_LAST ? higher[s] : __ballot_sync(FULL, above)) & f.a[s] & under[s]);
      if (!above && key[s] > ki) {   // between the two: column q now holds a lower row, column p a higher one
        if (reaches_q[s]) --chance[s];
        if (reaches_p[s]) ++chance[s];
      }
    }
    if constexpr (RELOAD) {
      unsigned both[W];
#pragma unroll
      for (int w = 0; w < W; ++w) both[w] = root[w] | target[w];
      reload(both);
#pragma unroll
      for (int s = 0; s < W; ++s) {
        if (mine(target, s)) chance[s] = settled ? 0 : UNKNOWN;
        if (mine(root, s)) chance[s] = own;
      }
    } else {
      settle(target, e, settled ? 0 : UNKNOWN);
      settle(root, f, own);
    }
    unsigned P[W];
#pragma unroll
    for (int w = 0; w < W; ++w) P[w] = root[w] | target[w];
    void_records(P);
  }

  // Row e (of position p, single: root) takes column q (single: target), which its search has reached at `level`; the row
  // displaced there takes a column of the level before that it is adjacent to (there is one: that is how it was
  // reached), the lowest or the lowest of those with a higher row, and so on down to p, the only column of level 0.
  __device__ __forceinline__ void walk(int p, const unsigned (&root)[W], PosEntry<W> e, int q, unsigned (&target)[W], int level,
                                       bool settled) {
    unsigned P[W];
    PosEntry<W> f = tab.load(q);
    if constexpr (!FIRST_APART) {
      if (level == 1) {
        exchange(p, root, e, q, target, f, settled);
        return;
      }
    }
#pragma unroll
    for (int w = 0; w < W; ++w) P[w] = 0u;
    while (true) {
      shift(q, target, e, f.row8);
#pragma unroll
      for (int w = 0; w < W; ++w) P[w] |= target[w];
      e = f;
      if (level == 0) break;
      --level;
      unsigned h[W];
      hist_load<W>(hist, level, h);
#pragma unroll
      for (int w = 0; w < W; ++w) h[w] = level == 0 ? root[w] : h[w] & e.a[w];
      if constexpr (W <= 6) {
        // rather a column that the row can have without displacing a lower one: that row would be searched again (N = 128:
        // 4.5 instead of 5.2 searches per matching, 23.5 -> 19.4 ms over 1024 x 3000 matchings; N = 64 27.9 -> 27.5 ms;
        // 100 x N = 192 17.0 -> 16.1 ms; with seven and eight words the votes cost what the searches save)
        unsigned G[W], some = 0u;
        rows_above(e.row8, G);
#pragma unroll
        for (int w = 0; w < W; ++w) {
          G[w] &= h[w];
          some |= G[w];
        }
#pragma unroll
        for (int w = 0; w < W; ++w) h[w] = some != 0u && level != 0 ? G[w] : h[w];
      }
      q = (int)min((unsigned)first_of<W>(h, target), (unsigned)(N - 1));
      f = tab.load(q);
    }
    void_records(P);
  }

  // Records that contain a row that has moved are void.
  __device__ __forceinline__ void void_records(const unsigned (&P)[W]) {
#pragma unroll
    for (int s = 0; s < W; ++s) {
      unsigned v = 0u;
#pragma unroll
      for (int w = 0; w < W; ++w) v |= rec[s][w] & P[w];
      if (chance[s] < 0 && v != 0u) chance[s] = UNKNOWN;
    }
  }

  // Search from the columns F over the rows of `alive`, level by level into the history, until a row at a column of `target`
  // is reached (true) or nothing more is. `level`: the last level with members.
  __device__ __forceinline__ bool search(unsigned (&F)[W], unsigned (&alive)[W], const unsigned (&target)[W], int& level,
                                         unsigned& levels, unsigned& pops) const {
    while (true) {   // every level takes its members out of `alive`
      unsigned hit;
      if (!step(F, alive, target, hit, levels, pops)) return false;
      ++level;
      if (hit != 0u) return true;
      hist_store<W>(hist, level, F);
    }
  }
  // One level of it; whether it has members. hit: not zero if one of them is the one searched for.
  __device__ __forceinline__ bool step(unsigned (&F)[W], unsigned (&alive)[W], const unsigned (&target)[W], unsigned& hit,
                                       unsigned& levels, unsigned& pops) const {
    const unsigned any = grow(F, alive);
    ++levels;
    hit = 0u;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      pops += __popc(F[w]);
      hit |= F[w] & target[w];
    }
    return any != 0u;
  }

  // ---- repair: every row that lost its entry gets a column again ----------------------------------
  // Rows below r0, the row that lost its entry, keep their columns if at all possible: the columns that can be handed to
  // r0 without touching them are found by a forward search from the free column over the rows above r0 (a row adjacent to
  // a column of the previous level could move there and release its own). r0 takes the lowest such column it is adjacent
  // to, which is its column in the lexicographically smallest matching of the new graph, and the rows on the way
  // move one step each towards the free column. Several free rows at once, and a row that needs rows below it, go through
  // repair_any(). Rows below lo8 >> 8 have their final column. False: some row cannot be matched any more (the matching of
  // the others is unchanged).
  __device__ __forceinline__ bool repair(unsigned& lo8, unsigned (&work)[MOESCHED_WORK_FIELDS]) {
    unsigned alive[W];
    int searched = -1;   // levels of a search that found nothing for the only free row
    if (broken_count == 1) {
      const int p = MS_AT(first_of<W>(broken), N);
      const PosEntry<W> e = tab.load(p);
      unsigned F[W], want[W], target[W], any = 0u;
      if (VOTES_LAST) rows_above(e.row8, alive);
#pragma unroll
      for (int s = 0; s < W; ++s) {
        if (!VOTES_LAST) alive[s] = __ballot_sync(FULL, key[s] > (e.row8 | 0xffu));   // the rows above r0
        F[s] = broken[s];
        want[s] = e.a[s] & alive[s];
        any |= want[s];
      }
      if (any != 0u) {
        int q = MS_AT(first_of<W>(want, target), N), level = 0;
        unsigned pops = 0u, hit1;
        bool hit;
        if constexpr (FIRST_APART) {
          const bool some = step(F, alive, target, hit1, work[WK_SCAN], pops);
          if (some && hit1 != 0u) {
            work[WK_AUG]++;
            work[WK_TIGHT]++;
            exchange(p, broken, e, q, target, tab.load(q));
            lo8 = min(lo8, e.row8 + 0x100u);
            broken_count = 0;
            return true;
          }
          hit = false;
          if (some) {
            level = 1;
            hist_store<W>(hist, 1, F);
            hit = search(F, alive, target, level, work[WK_SCAN], pops);
          }
        } else {
          hit = search(F, alive, target, level, work[WK_SCAN], pops);
        }
        if (!hit) {
          any = 0u;
#pragma unroll
          for (int w = 0; w < W; ++w) { want[w] &= ~alive[w]; any |= want[w]; }
          if (any != 0u) {   // the next best column
            q = MS_AT(first_of<W>(want, target), N);
            level = level_of_row<W>(hist, level, q, lane);
          }
        }
        if (hit || any != 0u) {
          work[WK_AUG] += level;
          work[WK_TIGHT]++;
          walk(p, broken, e, q, target, level, hit);
          lo8 = min(lo8, e.row8 + 0x100u);   // r0 has its final column; the rows that moved lie above it
          broken_count = 0;
          return true;
        }
        // (with more words, what this keeps alive costs more than the search: N = 8 1.28 -> 1.15 us a matching, N = 100
        // 4.39 -> 4.46, N = 256 17.9 -> 23.2)
        if constexpr (W == 1) searched = level;
      }
    }
    return repair_any(lo8, searched, alive, work);
  }

  // The general case: free rows lowest first, each from all free columns. A row that is adjacent to none of the columns that
  // can be released above it: the highest row below r0 that could move to one of them is admitted, the search continues from
  // its column, and so on: the path disturbs as few low rows as possible, and lo8 drops to the lowest row it moves.
  // searched >= 0: the only free row has been searched for so many levels; `left` are the rows above it that were not reached.
  __device__ __forceinline__ bool repair_any(unsigned& lo8, int searched, const unsigned (&left)[W],
                                             unsigned (&work)[MOESCHED_WORK_FIELDS]) {
    for (; broken_count > 0; --broken_count) {
      unsigned k = 0xffffffffu;
#pragma unroll
      for (int s = 0; s < W; ++s)
        if (mine(broken, s)) k = min(k, key[s]);
      k = __reduce_min_sync(FULL, k);
      const int p = MS_AT((int)(k & 0xffu), N);
      PosEntry<W> e = tab.load(p);
      const unsigned r8 = e.row8;
      unsigned above[W], alive[W], F[W], target[W], admitted[W], can[W], any = 0u;
      if (VOTES_LAST) rows_above(r8, above);
#pragma unroll
      for (int s = 0; s < W; ++s) {
        if (!VOTES_LAST) above[s] = __ballot_sync(FULL, key[s] > (r8 | 0xffu));
        F[s] = broken[s];
        alive[s] = searched >= 0 ? left[s] : above[s] & ~F[s];
        can[s] = e.a[s] & (above[s] | F[s]);
        any |= can[s];
        target[s] = admitted[s] = 0u;
      }
      int q = any != 0u ? MS_AT(first_of<W>(can, target), N) : 0, level = max(searched, 0);
      hist_store<W>(hist, 0, F);
      bool lowered = false, settled = intersects<W>(F, target);
      unsigned pops = 0u;
      while (!settled) {
        if (searched < 0) settled = search(F, alive, target, level, work[WK_SCAN], pops);
        if (settled) break;
        searched = -1;
        unsigned released[W];
        any = 0u;
#pragma unroll
        for (int w = 0; w < W; ++w) {
          released[w] = broken[w] | admitted[w] | (above[w] & ~alive[w]);
          can[w] = e.a[w] & released[w];
          any |= can[w];
        }
        if (any != 0u) {   // the lowest released column r0 is adjacent to
          q = first_of<W>(can, target);
          level = level_of_row<W>(hist, level, MS_AT(q, N), lane);
          break;
        }
        k = 0u;
#pragma unroll
        for (int s = 0; s < W; ++s) {
          unsigned o = 0u;
#pragma unroll
          for (int w = 0; w < W; ++w) o |= A[s][w] & released[w];
          if (o != 0u && key[s] < r8 && !mine(admitted, s) && valid(s)) k = max(k, key[s] + 0x100u);
        }
        k = __reduce_max_sync(FULL, k);
        if (k == 0u) return false;
        lowered = true;
        single_mask<W>((int)(k & 0xffu), F);
        ++level;
        hist_store<W>(hist, level, F);
        settled = intersects<W>(F, e.a);   // r0 is adjacent to the admitted row's own column
        q = settled ? (int)(k & 0xffu) : q;
#pragma unroll
        for (int w = 0; w < W; ++w) {
          admitted[w] |= F[w];
          if (settled) target[w] = F[w];
        }
      }
      unsigned P[W], lowest8 = r8;
#pragma unroll
      for (int w = 0; w < W; ++w) P[w] = 0u;
      while (true) {
        const PosEntry<W> old = tab.load(MS_AT(q, N));
        shift(q, target, e, old.row8);
#pragma unroll
        for (int w = 0; w < W; ++w) P[w] |= target[w];
        lowest8 = min(lowest8, e.row8);
        e = old;
        if (level == 0) break;
        --level;
        work[WK_AUG]++;
        unsigned h[W];
        hist_load<W>(hist, level, h);
        if (lowered) {   // an admitted row may move to a column of ANY earlier level; the levels still fall strictly
          for (int d = 0; d < level; ++d) {
            unsigned hd[W];
            hist_load<W>(hist, d, hd);
#pragma unroll
            for (int w = 0; w < W; ++w) h[w] |= hd[w];
          }
        }
#pragma unroll
        for (int w = 0; w < W; ++w) h[w] &= e.a[w];
        q = (int)min((unsigned)first_of<W>(h, target), (unsigned)(N - 1));
        if (lowered) level = level_of_row<W>(hist, level, MS_AT(q, N), lane);
      }
      work[WK_BATCH] += lowered ? 1u : 0u;
      work[WK_TIGHT] += lowered ? 0u : 1u;
      lo8 = min(lo8, lowered ? lowest8 : r8 + 0x100u);
      // the free column q is taken now; its own free row, if that is another one than r0, sits at p until its turn comes
#pragma unroll
      for (int w = 0; w < W; ++w) broken[w] &= ~target[w];
      if (q != p) {
        single_mask<W>(p, target);
        shift(p, target, e, r8);
#pragma unroll
        for (int w = 0; w < W; ++w) P[w] |= target[w];
      }
      void_records(P);
    }
    return true;
  }

  // ---- lexicographically smallest perfect matching over the rows from lo8 >> 8 up -------------------
  // Rows below have their final column. A row i can only move to a lower column if one of those it is adjacent to holds
  // a row above i. A backward search from i's own column -- who could take the column of a row already reached -- runs until
  // it reaches the row at the lowest such column (nothing lower can be had) or is exhausted; the lowest column reached is
  // taken and the matching rotated along the cycle. (lo8 rises with every row looked at.)
  __device__ __forceinline__ void canonicalise(unsigned lo8, unsigned (&work)[MOESCHED_WORK_FIELDS]) {
    unsigned all[W];
#pragma unroll
    for (int w = 0; w < W; ++w) all[w] = 0xffffffffu;
    canonicalise(lo8, all, work);
  }
  // (all cycles lie within `left`)
  __device__ __forceinline__ void canonicalise(unsigned lo8, const unsigned (&left)[W], unsigned (&work)[MOESCHED_WORK_FIELDS]) {
    while (true) {
      unsigned k = 0xffffffffu;
#pragma unroll
      for (int s = 0; s < W; ++s)
        if (chance[s] > 0 && key[s] >= lo8) k = min(k, key[s]);
      k = __reduce_min_sync(FULL, k);
      if (k == 0xffffffffu) return;
      const int p = MS_AT((int)(k & 0xffu), N);
      k |= 0xffu;
      lo8 = k + 1u;
      const PosEntry<W> e = tab.load(p);
      unsigned root[W], alive[W], F[W], want[W], target[W], any = 0u;
      single_mask<W>(p, root);
      below_mask<W>(root, want);
      if (VOTES_LAST) rows_above(k, alive);
#pragma unroll
      for (int s = 0; s < W; ++s) {
        if (!VOTES_LAST) alive[s] = __ballot_sync(FULL, key[s] > k);   // the rows above
        alive[s] &= left[s];
        want[s] &= e.a[s] & alive[s];
        any |= want[s];
        F[s] = root[s];
      }
      int q = 0, level = FIRST_APART ? 1 : 0;
      if constexpr (WANT_EARLY) q = first_of<W>(want, target);   // (meaningless if there is none)
      if (any == 0u) {   // (after a record has become void) none: counted from here on
#pragma unroll
        for (int s = 0; s < W; ++s)
          if (mine(root, s)) chance[s] = 0;
        continue;
      }
      work[WK_SWEEP]++;
      work[WK_POP]++;
      if constexpr (!WANT_EARLY) q = first_of<W>(want, target);
      q = MS_AT(q, N);
      bool hit = false;
      if constexpr (FIRST_APART) {
        unsigned hit1;
        const bool some = step(F, alive, target, hit1, work[WK_LEVEL], work[WK_POP]);
        if (NONE_APART && !some) {   // nobody can take its column
#pragma unroll
          for (int s = 0; s < W; ++s) {
            if (mine(root, s)) {
              chance[s] = IN_VAIN;
#pragma unroll
              for (int w = 0; w < W; ++w) rec[s][w] = root[w];
            }
          }
          continue;
        }
        if ((NONE_APART || some) && hit1 != 0u) {
          work[WK_ROT]++;
          exchange(p, root, e, q, target, tab.load(q));
          continue;
        }
        if (NONE_APART || some) {
          hist_store<W>(hist, 1, F);
          hit = search(F, alive, target, level, work[WK_LEVEL], work[WK_POP]);
        }
      } else {
        hit = search(F, alive, target, level, work[WK_LEVEL], work[WK_POP]);
      }
      if (!hit) {
        any = 0u;
#pragma unroll
        for (int w = 0; w < W; ++w) { want[w] &= ~alive[w]; any |= want[w]; }
        if (any == 0u) {
          // the row stays put until one of the rows that can reach it changes column
          rows_above(k, want);
#pragma unroll
          for (int w = 0; w < W; ++w) want[w] = (want[w] & left[w] & ~alive[w]) | root[w];
#pragma unroll
          for (int s = 0; s < W; ++s) {
            if (mine(root, s)) {
              chance[s] = IN_VAIN;
#pragma unroll
              for (int w = 0; w < W; ++w) rec[s][w] = want[w];
            }
          }
          continue;
        }
        q = MS_AT(first_of<W>(want, target), N);   // the next best column
        level = level_of_row<W>(hist, level, q, lane);
      }
      work[WK_ROT] += level;
      walk(p, root, e, q, target, level, hit);
    }
  }

  // The values of the pairs as they are now: what a lane holds for a pair given up goes back to memory.
  __device__ __forceinline__ void fetch_values() {
#pragma unroll
    for (int s = 0; s < W; ++s) {
      const int r = (int)(key[s] >> 8);
      if (r != vrow[s]) {
        *mem.cell(MS_AT(vrow[s], N), s * 32 + lane) = val[s];
        val[s] = *mem.cell(MS_AT(r, N), s * 32 + lane);
        vrow[s] = r;
      }
    }
  }

  // The smallest matched value has been subtracted and the pairs of `zero` (bit s of the lane) have vanished: takes their
  // edges out and returns how many there were (uniform).
  __device__ __forceinline__ int drop_edges(unsigned zero) {
    broken_count = 0;
    __syncwarp();   // every lane is done with the entries as they were
#pragma unroll
    for (int s = 0; s < W; ++s) {
      const bool z = (zero >> s) & 1u;
      if (z) {
        A[s][s] &= ~(1u << lane);
        tab.base[(s * 32 + lane) * PosTable<W>::WORDS + s] = A[s][s];
      }
      broken[s] = __ballot_sync(FULL, z);
      broken_count += __popc(broken[s]);
    }
    __syncwarp();   // the table entries above were written by their owners alone
    return broken_count;
  }
};

}  // namespace moesched
