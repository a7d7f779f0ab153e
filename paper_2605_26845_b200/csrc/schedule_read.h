// What the scoring kernel reads of a schedule array, as plain arithmetic (no CUDA in here: the CPU tests compile it too).
#pragma once

namespace moesched {

// A matrix's schedule is read in groups of 16 aligned bytes, the first of which begins `skew` bytes before it. That may be
// part of the matrix before; where fewer than `skew` bytes of the array precede the schedule, the group would begin before
// the array, and only the part from the schedule's first byte on is read.
#ifdef __CUDACC__
__host__ __device__
#endif
inline bool begins_before_the_array(long long ahead, int skew) {
  return ahead < skew;
}

}  // namespace moesched
