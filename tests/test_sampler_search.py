"""The shared-memory search of sample_rows_kernel, walked on the host with the kernel's own index arithmetic
(netmax_search.h): every probe stays inside the row it belongs to, over all numbers of workers the kernel takes (every one to
4096, every seventh beyond), and the draw is the one plain counting gives -- also for u = 2^32 - 1, which no threshold is above."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2009_05766_b200", "csrc")

PROGRAM = r"""
#include <algorithm>
#include <cstdio>
#include <vector>
#include "netmax_search.h"
using namespace netmax;

static uint64_t state = 88172645463325252ull;
static uint32_t word() { state ^= state << 13; state ^= state >> 7; state ^= state << 17; return (uint32_t)(state >> 16); }

int main() {
  long draws = 0;
  for (uint32_t M = 128; M <= 16384; M += (M < 4096 ? 1 : 7)) {
    const uint32_t h = sample_levels(M), padded = (M + 15u) & ~15u;
    for (int rows : {2, 4})
      if (padded > sample_stride(M, rows) || (1u << h) > sample_tree(M, rows)) return std::printf("rows overlap, M = %u\n", M), 1;
    for (uint32_t last : {M - 1, M / 2, 0u}) {  // the row's last positive entry: thresholds are at the top from there on
      std::vector<uint32_t> row(padded, 0xFFFFFFFFu), tree(1u << h, 0u);
      std::vector<int> set(1u << h, 0);
      for (uint32_t j = 0; j < last; ++j) row[j] = word();
      std::sort(row.begin(), row.begin() + last);
      for (uint32_t j = 1; j < (1u << h); ++j) {
        const uint32_t n = sample_node(j, h, (uint32_t)__builtin_ctz(j));
        if (n == 0 || n >= (1u << h) || set[n]++) return std::printf("node %u of M = %u\n", n, M), 1;
        tree[n] = 16u * j <= M ? row[16u * j - 1u] : 0xFFFFFFFFu;
      }
      for (uint32_t u : {0u, 1u, word(), word(), row[last / 2], row[last / 2] - 1u, row[(M - 1) / 16 * 16], 0xFFFFFFFEu, 0xFFFFFFFFu}) {
        uint32_t at = 1;
        for (uint32_t l = 0; l < h; ++l) at = 2u * at + (tree[at] <= u ? 1u : 0u);
        at = 16u * sample_block(at, h, M);
        for (uint32_t s = 8; s > 0; s >>= 1) {
          if (at + s - 1 >= padded) return std::printf("M = %u, u = %u: probe at %u of a row of %u\n", M, u, at + s - 1, padded), 1;
          if (row[at + s - 1] <= u) at += s;
        }
        const uint32_t count = (uint32_t)(std::upper_bound(row.begin(), row.begin() + M, u) - row.begin());
        if (std::min(at, last) != std::min(count, last)) return std::printf("M = %u, u = %u: drew %u\n", M, u, std::min(at, last)), 1;
        ++draws;
      }
    }
  }
  std::printf("%ld\n", draws);
  return 0;
}
"""


def test_every_probe_stays_in_its_row_and_draws_what_counting_gives(tmp_path):
    src, exe = tmp_path / "search.cpp", tmp_path / "search"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    done = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert done.returncode == 0, done.stdout
    assert int(done.stdout) > 100_000
