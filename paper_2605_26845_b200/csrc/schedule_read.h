// What the scoring kernel reads of a schedule array, as plain arithmetic (no CUDA in here: the CPU tests compile it too).
#pragma once

namespace moesched {

struct ByteSpan {
  int from, to;   // bytes [from, to) of a group of 16
};

// A chunk of `bytes` bytes that begins `ahead` bytes into the array (15 stands for all above) is read in groups of 16 aligned bytes; the group that
// begins `at` bytes after the chunk's first byte (at > -16) is read in this span. A group may reach back into what precedes
// the chunk as long as that belongs to the array; where it would begin before the array it is read from the chunk's
// first byte on. Nothing behind the chunk is read.
#ifdef __CUDACC__
__host__ __device__
#endif
inline ByteSpan group_span(int ahead, int bytes, int at) {
  ByteSpan s;
  s.from = at + ahead < 0 ? -at : 0;
  s.to = bytes - at < 16 ? bytes - at : 16;
  return s;
}

}  // namespace moesched
