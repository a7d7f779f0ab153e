"""Which bytes of a schedule array the scoring kernel reads: csrc/schedule_read.h, compiled for the CPU."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "schedule_read.h"
// All chunks (32 matchings) of all matrices of a batch of schedules of stride K, of which `used` matchings are read, in
// an array that begins `offset` bytes after a multiple of 16: returns 0 if every used byte is read and none outside.
static int faults(int B, int N, int K, int used, int offset) {
  std::vector<int> read((size_t)B * K * N, 0);
  for (int b = 0; b < B; ++b)
    for (int c = 0; c * 32 < used; ++c) {
      const long long ahead = (long long)b * K * N + (long long)c * 32 * N;
      const int bytes = (used - c * 32 < 32 ? used - c * 32 : 32) * N, skew = (int)((offset + ahead) & 15);
      for (int g = 0; g * 16 < bytes + skew; ++g) {
        const int at = g * 16 - skew;   // offset of the group from the chunk's first byte
        const bool cut = at < 0 && c == 0 && moesched::begins_before_the_array(ahead, skew);
        const int from = cut ? skew : 0, to = bytes - at < 16 ? bytes - at : 16;
        for (int q = from; q < to; ++q) {
          const long long byte = ahead + at + q;
          if (byte < 0 || byte >= ahead + bytes) return 1;
          ++read[byte];
        }
      }
    }
  for (int b = 0; b < B; ++b)
    for (int i = 0; i < used * N; ++i)
      if (read[(size_t)b * K * N + i] == 0) return 2;
  return 0;
}
int main() {
  for (int N : {1, 2, 3, 4, 5, 7, 8, 15, 16, 17, 33, 64, 100, 255, 256})
    for (int K : {1, 2, 3, 4, 15, 31, 32, 33, 65})
      for (int used : {1, K / 2, K - 1, K})
        for (int offset = 0; offset < 16; ++offset) {
          if (used < 1) continue;
          const int f = faults(N == 1 ? 40 : 18, N, K, used, offset);
          if (f != 0) { std::printf("N %d, stride %d, %d used, offset %d: fault %d\n", N, K, used, offset, f); return 1; }
        }
  return 0;
}
"""


def test_nothing_outside_the_schedules_is_read(tmp_path):
    src, exe = tmp_path / "read.cpp", tmp_path / "read"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-I", os.path.join(ROOT, "paper_2605_26845_b200", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    done = subprocess.run([str(exe)], capture_output=True, text=True)
    assert done.returncode == 0, done.stdout
