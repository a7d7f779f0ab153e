// The lexicographically smallest perfect matching of a graph of at most SMALL_MAX_N ranks, kept up to date while edges
// vanish: one warp, no searches.
//
// Which sets of columns the rows i .. N-1 can fill is a bitmap F_i over all 2^N sets. F_i follows from F_{i+1}: a set can be
// filled if taking one of row i's columns out of it leaves one that can. Columns 0 .. 4 number a bit within a lane's word, columns
// 5 and up the lane, so that taking a column out is a shift by a constant or a shuffle, for all sets at once. The matching is then
// read off from row 0 up: a row takes the lowest of its columns that leaves a set which the rows after it can fill; lane c looks at
// column c.
// After edges have vanished, F has changed only for their rows and lower ones (the recomputation stops where it comes out as
// before), rows below the lowest of them keep their columns if that can still be completed, and once the rows above the
// highest of them see the columns left that they saw before, they keep theirs too. (N = 8: 1.8 bitmaps recomputed and 3.9 rows read
// off per matching.)
//
// What bounds it: the chain of shuffle, shift and vote per row read off, 175 cycles, and of 270 cycles per bitmap, with the
// branches between them. Against the searches of peel.cuh, complete decompositions, back to back in a CUDA graph, B200, for 1, 592 and
// 4096 matrices: N = 1 1.95 -> 1.24 us, 2.61 -> 1.93, 4.19 -> 2.39; N = 4 7.8 -> 6.3, 9.3 -> 6.6, 19.4 -> 13.5; N = 6 20.6 -> 18.6, 25.6 -> 20.3,
// 49.4 -> 41.1; N = 8 39.1 -> 38.7, 43.4 -> 41.0, 96.9 -> 93.3. At eight ranks it ends there: 10000 matrices 198 and 199 us, 40000 727 and
// 741; from nine ranks on the instructions (4096 of N = 10 169 and 207).
#pragma once

#include "common.cuh"

namespace moesched {

constexpr int SMALL_MAX_N = 8;

template <int N>
struct SmallMatcher {
  static constexpr unsigned ALL = (1u << N) - 1u;
  int lane;
  unsigned rows;              // rows adjacent to the lane's column
  int row;                    // the row matched to it
  unsigned left[N];           // columns that the rows before i leave
  unsigned F[N + 1];          // F[0] is not used

  // sets of the bitmap that have column c (c < 5)
  __host__ __device__ static constexpr unsigned having(int c) {
    return c == 0 ? 0xaaaaaaaau : c == 1 ? 0xccccccccu : c == 2 ? 0xf0f0f0f0u : c == 3 ? 0xff00ff00u : 0xffff0000u;
  }

  __device__ __forceinline__ void begin(int lane_, unsigned rows_) {
    lane = lane_;
    rows = rows_;
    row = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) F[i] = left[i] = 0u;
    F[N] = lane == 0 ? 1u : 0u;   // the empty set
  }

  // F[i] from F[i + 1]; whether it has changed.
  __device__ __forceinline__ bool fill(int i, unsigned after, unsigned& mine) const {
    const unsigned cols = __ballot_sync(FULL, (rows >> i) & 1u);
    unsigned now = 0u;
#pragma unroll
    for (int c = 0; c < N; ++c) {
      const unsigned has = 0u - ((cols >> c) & 1u);
      if (c < 5) now |= (after << (1 << (c < 5 ? c : 0))) & (has & having(c));
      else now |= __shfl_xor_sync(FULL, after, 1 << (c >= 5 ? c - 5 : 0)) & (has & (0u - ((unsigned)(lane >> (c >= 5 ? c - 5 : 0)) & 1u)));
    }
    const bool changed = now != mine;
    mine = now;
    return __any_sync(FULL, changed);
  }

  // Row i takes its column out of S, if it can have one.
  __device__ __forceinline__ void take(int i, unsigned after, unsigned& S) {
    const unsigned rest = S & ~(1u << lane);
    const unsigned word = __shfl_sync(FULL, after, (int)(rest >> 5));
    unsigned b = __ballot_sync(FULL, (word >> (rest & 31u)) & (S >> lane) & (rows >> i) & 1u);
    b &= 0u - b;
    row = (b >> lane) & 1u ? i : row;
    S &= ~b;
  }

  // The matching of the graph without the edges that the rows `gone` have lost (all rows: without anything known before).
  // False: there is no perfect matching any more.
  __device__ __forceinline__ bool update(unsigned gone, bool first_time) {
    switch (31 - __clz(gone)) {
#define MOESCHED_FILL(I)                                                            \
  case I:                                                                           \
    if constexpr (I >= 1 && I < N) {                                                \
      if (!fill(I, F[I + 1], F[I]) && (gone & ((1u << I) - 1u)) == 0u) break;       \
    }                                                                               \
    [[fallthrough]];
      MOESCHED_FILL(7) MOESCHED_FILL(6)
      MOESCHED_FILL(5) MOESCHED_FILL(4) MOESCHED_FILL(3) MOESCHED_FILL(2) MOESCHED_FILL(1)
#undef MOESCHED_FILL
      default: break;
    }
    // Rows below the lowest of `gone` keep their columns if that can be completed. If not, so do those below the highest row that can.
    int from = first_time ? 0 : __ffs(gone) - 1;
    for (int attempt = 0; attempt < 2; ++attempt) {
      unsigned S = ALL & ~__ballot_sync(FULL, !first_time && row < from);
      bool as_before = false;
      switch (from) {
#define MOESCHED_TAKE(I)                                                            \
  case I:                                                                           \
    if constexpr (I < N) {                                                          \
      as_before = !first_time && S == left[I] && (gone >> I) == 0u;                 \
      if (as_before) break;                                                         \
      left[I] = S;                                                                  \
      take(I, F[I + 1], S);                                                         \
    }                                                                               \
    [[fallthrough]];
        MOESCHED_TAKE(0) MOESCHED_TAKE(1) MOESCHED_TAKE(2) MOESCHED_TAKE(3) MOESCHED_TAKE(4) MOESCHED_TAKE(5)
        MOESCHED_TAKE(6) MOESCHED_TAKE(7)
#undef MOESCHED_TAKE
        default: break;
      }
      if (as_before || S == 0u) return true;
      if (from == 0) return false;
      // The first row had nothing to take, and `left` is as before for it and the rows below.
      int can = 0;
#pragma unroll
      for (int i = 1; i < N; ++i) {
        const unsigned L = left[i];
        const unsigned word = __shfl_sync(FULL, F[i], (int)(L >> 5));
        if (i < from && ((word >> (L & 31u)) & 1u) != 0u) can = i;
      }
      from = can;
    }
    return false;
  }
};


}  // namespace moesched
