"""How a GEMM over all tokens is cut into slabs (csrc/slab_plan.h, host arithmetic): the same cost as a scan of every count, and
few counts looked at, because the library plans at every call."""

import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_23353_b200", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <random>
#include "slab_plan.h"
using isopo::plan_slab;

static int64_t cost(int64_t blocks, int64_t per, int64_t tiles, int64_t slots, int64_t overhead) {
  return ((blocks + per - 1) / per * tiles + slots - 1) / slots * (per + overhead);
}

int main() {
  std::mt19937_64 rng(1);
  auto log_int = [&](int64_t top) {
    int bits = 1;
    while ((int64_t)1 << bits <= top) ++bits;
    return std::min<int64_t>(top, 1 + (int64_t)(rng() >> 1) % ((int64_t)1 << (1 + rng() % bits)));
  };
  int64_t looked_most = 0;
  for (int k = 0; k < 20000; ++k) {
    const int64_t blocks = log_int(20000), tiles = log_int(3000), slots = 1 + rng() % 600, overhead = rng() % 20;
    const int64_t most = k % 3 == 0 ? log_int(4000) : std::min<int64_t>((blocks + 7) / 8, std::max<int64_t>(8, 8 * slots / tiles));
    const int64_t per = plan_slab(blocks, tiles, slots, overhead, most);
    const int64_t top = std::max<int64_t>(1, std::min(most, blocks));
    if (per < 1 || per > blocks || (blocks + per - 1) / per > top) return printf("slab of %ld in %ld blocks, at most %ld\n", (long)per, (long)blocks, (long)most), 1;
    int64_t best = INT64_MAX;
    for (int64_t n = 1; n <= top; ++n) best = std::min(best, cost(blocks, (blocks + n - 1) / n, tiles, slots, overhead));
    if (cost(blocks, per, tiles, slots, overhead) != best)
      return printf("blocks %ld tiles %ld slots %ld most %ld: %ld against %ld\n", (long)blocks, (long)tiles, (long)slots, (long)most,
                    (long)cost(blocks, per, tiles, slots, overhead), (long)best), 1;
    // counts looked at under the library's own limits: eight waves, or eight counts of layers with more tiles than slots
    if (k % 3) {
      int64_t looked = 0;
      for (int64_t n = 0; n < top; ++looked) n = std::min(top, (((n + 1) * tiles + slots - 1) / slots) * slots / tiles);
      looked_most = std::max(looked_most, looked);
    }
  }
  printf("%ld\n", (long)looked_most);
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("slab_plan")
    src, exe = d / "main.cpp", d / "main"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return exe


def test_same_cost_as_a_scan_of_every_count(program):
    r = subprocess.run([str(program)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout) <= 9
