// The Peeler (csrc/peel.cuh) and the SmallMatcher (csrc/small.cuh) on the CPU: one thread per lane, votes and reductions through a
// barrier of the 32 threads. The lanes really run apart between two such operations, so a lane that overwrites shared memory which
// another has still to read shows in the result. Reads N, k_max and a balanced N x N matrix from standard input (int32), writes the
// number of matchings, then coefficients and permutations: by the Peeler, or by the SmallMatcher with the argument "small". With the
// argument "adopt" the matrix is a graph, followed by a column for each row that make a matching of it, and the lexicographically
// smallest matching is written (one, with coefficient 0): the Peeler as the greedy decomposition enters it.
#include <barrier>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <thread>
#include <vector>

#include <cuda_runtime.h>

static std::barrier<> lanes(32);
static unsigned slots[32];
static thread_local int self;
static thread_local unsigned noise;

static void together() {
  lanes.arrive_and_wait();
  noise = noise * 1664525u + 1013904223u;   // lanes go on one after the other, in an order that changes
  if (noise >> 31) std::this_thread::yield();
  for (volatile unsigned n = noise >> 22; n > 0; n = n - 1) {}
}
static void __syncwarp() { together(); }
template <typename F>
static unsigned combine(unsigned v, F f) {
  slots[self] = v;
  together();
  unsigned r = slots[0];
  for (int l = 1; l < 32; ++l) r = f(r, slots[l]);
  together();
  return r;
}
static unsigned __ballot_sync(unsigned, bool p) {
  return combine(p ? 1u << self : 0u, [](unsigned a, unsigned b) { return a | b; });
}
static unsigned __reduce_min_sync(unsigned, unsigned v) {
  return combine(v, [](unsigned a, unsigned b) { return a < b ? a : b; });
}
static unsigned __reduce_max_sync(unsigned, unsigned v) {
  return combine(v, [](unsigned a, unsigned b) { return a > b ? a : b; });
}
static unsigned __reduce_add_sync(unsigned, unsigned v) {
  return combine(v, [](unsigned a, unsigned b) { return a + b; });
}
static unsigned __reduce_or_sync(unsigned, unsigned v) {
  return combine(v, [](unsigned a, unsigned b) { return a | b; });
}
static bool __any_sync(unsigned m, bool p) { return __ballot_sync(m, p) != 0u; }
static unsigned __shfl_sync(unsigned, unsigned v, int from) {
  slots[self] = v;
  together();
  const unsigned r = slots[from & 31];
  together();
  return r;
}
static unsigned __shfl_xor_sync(unsigned m, unsigned v, int bits) { return __shfl_sync(m, v, self ^ bits); }
static int __popc(unsigned v) { return __builtin_popcount(v); }
static int __clz(unsigned v) { return v ? __builtin_clz(v) : 32; }
static int __ffs(unsigned v) { return __builtin_ffs((int)v); }
template <typename A, typename B>
static auto min(A a, B b) { return a < b ? a : b; }
template <typename A, typename B>
static auto max(A a, B b) { return a > b ? a : b; }
static size_t __cvta_generic_to_shared(const void* p) { return (size_t)p; }   // (these two are only named)
static unsigned long long __umul64hi(unsigned long long a, unsigned long long) { return a; }

#include "peel.cuh"
#include "small.cuh"

using namespace moesched;

static int N, k_max, found;
static std::vector<int> matrix, coef, column_of;
static std::vector<unsigned char> perm, memory;

template <int W>
static void lane_main(int lane) {   // the loop of the Birkhoff kernel without the padding
  self = lane;
  noise = 2654435761u * (lane + 1);
  Peeler<W, int, false> pl;
  pl.mem.near_ = pl.mem.far_ = matrix.data();
  pl.mem.S = pl.mem.split = N;
  pl.reset(memory.data(), N, lane);
  int left = 0, k = 0;
  for (int r = 0; r < N; ++r) {
    PosEntry<W> e;
    e.row8 = (unsigned)r << 8;
    for (int s = 0; s < W; ++s) {
      const int c = s * 32 + lane;
      e.a[s] = __ballot_sync(FULL, c < N && matrix[r * N + c] > 0);
      left += __popc(e.a[s]);
    }
    pl.seat(r, e);
  }
  __syncwarp();
  unsigned work[MOESCHED_WORK_FIELDS] = {};
  for (; left > 0 && k < k_max; ++k) {
    unsigned lo8 = (unsigned)N << 8;
    if (!pl.repair(lo8, work)) break;
    if (k == 0) lo8 = 0u;
    pl.canonicalise(lo8, work);
    pl.fetch_values();
    unsigned least = 0xffffffffu, zero = 0u;
    for (int s = 0; s < W; ++s)
      if (pl.valid(s)) least = min(least, (unsigned)pl.val[s]);
    least = __reduce_min_sync(FULL, least);
    for (int s = 0; s < W; ++s) {
      pl.val[s] -= (int)least;
      if (pl.valid(s)) {
        if (pl.val[s] == 0) zero |= 1u << s;
        perm[(size_t)k * N + (pl.key[s] >> 8) % 256] = (unsigned char)(s * 32 + lane);
      }
    }
    left -= pl.drop_edges(zero);
    if (lane == 0) coef[k] = (int)least;
  }
  if (lane == 0) found = k;
}

template <int W>
static void lane_adopt(int lane) {   // the greedy kernel, from the graph of tight edges on
  self = lane;
  noise = 2654435761u * (lane + 1);
  Peeler<W, int, false> pl;
  pl.reset(memory.data(), N, lane);
  int highest[W];
  for (int s = 0; s < W; ++s) highest[s] = -1;
  for (int r = 0; r < N; ++r) {
    PosEntry<W> e;
    e.row8 = (unsigned)r << 8;
    for (int s = 0; s < W; ++s) {
      const int c = s * 32 + lane;
      const bool edge = c < N && matrix[r * N + c] > 0;
      if (edge) highest[s] = r;
      e.a[s] = __ballot_sync(FULL, edge);
    }
    pl.tab.store(column_of[r], e);
  }
  __syncwarp();
  unsigned left[W], work[MOESCHED_WORK_FIELDS] = {};
  pl.adopt(highest, left);
  pl.canonicalise(0u, left, work);
  for (int s = 0; s < W; ++s)
    if (pl.valid(s)) perm[(pl.key[s] >> 8) % 256] = (unsigned char)(s * 32 + lane);
  if (lane == 0) found = 1;
}

template <int N>
static void lane_small(int lane) {   // the loop of the kernel for few ranks without the padding
  self = lane;
  noise = 2654435761u * (lane + 1);
  unsigned rows = 0u;
  for (int r = 0; r < N; ++r)
    if (lane < N && matrix[r * N + lane] > 0) rows |= 1u << r;
  SmallMatcher<N> m;
  m.begin(lane, rows);
  int left = (int)__reduce_add_sync(FULL, (unsigned)__popc(rows)), k = 0;
  unsigned gone = SmallMatcher<N>::ALL;
  for (; left > 0 && k < k_max; ++k) {
    if (!m.update(gone, k == 0)) break;
    int* cell = lane < N ? &matrix[m.row % N * N + lane] : nullptr;
    const unsigned least = __reduce_min_sync(FULL, cell ? (unsigned)*cell : 0xffffffffu);
    if (cell) *cell -= (int)least;
    const unsigned lost = cell && *cell == 0 ? 1u << m.row : 0u;
    m.rows &= ~lost;
    gone = __reduce_or_sync(FULL, lost);
    left -= __popc(gone);
    if (cell) perm[(size_t)k * N + m.row % N] = (unsigned char)lane;
    if (lane == 0) coef[k] = (int)least;
  }
  if (lane == 0) found = k;
}

int main(int argc, char** argv) {
  const char* what = argc > 1 ? argv[1] : "";
  int head[2];
  if (std::fread(head, 4, 2, stdin) != 2) return 1;
  N = head[0];
  k_max = head[1];
  matrix.resize((size_t)N * N);
  if (std::fread(matrix.data(), 4, matrix.size(), stdin) != matrix.size()) return 1;
  if (!std::strcmp(what, "adopt")) {
    column_of.resize(N);
    if (std::fread(column_of.data(), 4, N, stdin) != (size_t)N) return 1;
  }
  coef.resize(k_max);
  perm.resize((size_t)k_max * N + 256);
  const int W = (N + 31) / 32;
  memory.resize(peel_smem_bytes(N, W) + 64);
  using Lane = void (*)(int);
  const Lane birkhoff[] = {lane_main<1>, lane_main<2>, lane_main<3>, lane_main<4>, lane_main<5>, lane_main<6>, lane_main<7>, lane_main<8>};
  const Lane adopt[] = {lane_adopt<1>, lane_adopt<2>, lane_adopt<3>, lane_adopt<4>, lane_adopt<5>, lane_adopt<6>, lane_adopt<7>, lane_adopt<8>};
  const Lane small[] = {lane_small<1>, lane_small<2>, lane_small<3>, lane_small<4>, lane_small<5>, lane_small<6>, lane_small<7>, lane_small<8>};
  const Lane run = !std::strcmp(what, "adopt") ? adopt[W - 1] : !std::strcmp(what, "small") ? small[N - 1] : birkhoff[W - 1];
  std::vector<std::thread> warp;
  for (int lane = 0; lane < 32; ++lane) warp.emplace_back(run, lane);
  for (auto& t : warp) t.join();
  std::fwrite(&found, 4, 1, stdout);
  std::fwrite(coef.data(), 4, found, stdout);
  std::fwrite(perm.data(), 1, (size_t)found * N, stdout);
  return 0;
}
