// The Peeler (csrc/peel.cuh) on the CPU: one thread per lane, votes and reductions through a barrier of the 32 threads. The
// lanes really run apart between two such operations, so a lane that overwrites shared memory which another has still to read
// shows in the result. Reads N, k_max and a balanced N x N matrix from standard input (int32), writes the number of
// matchings, then coefficients and permutations.
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

using namespace moesched;

static int N, k_max, found;
static std::vector<int> matrix, coef;
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

int main() {
  int head[2];
  if (std::fread(head, 4, 2, stdin) != 2) return 1;
  N = head[0];
  k_max = head[1];
  matrix.resize((size_t)N * N);
  if (std::fread(matrix.data(), 4, matrix.size(), stdin) != matrix.size()) return 1;
  coef.resize(k_max);
  perm.resize((size_t)k_max * N + 256);
  const int W = (N + 31) / 32;
  memory.resize(peel_smem_bytes(N, W) + 64);
  std::vector<std::thread> warp;
  for (int lane = 0; lane < 32; ++lane)
    warp.emplace_back(W == 1 ? lane_main<1> : W == 2 ? lane_main<2> : W == 3 ? lane_main<3> : lane_main<8>, lane);
  for (auto& t : warp) t.join();
  std::fwrite(&found, 4, 1, stdout);
  std::fwrite(coef.data(), 4, found, stdout);
  std::fwrite(perm.data(), 1, (size_t)found * N, stdout);
  return 0;
}
