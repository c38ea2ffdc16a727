// How a GEMM over all tokens is cut into token slabs.  Host arithmetic only: no CUDA, so that it can be tested by itself.
#pragma once

#include <stdint.h>

#include <algorithm>

namespace isopo {

// The tokens come in `blocks`; every slab of them is `tiles` work units; `slots` units run at one time.  Returns the blocks per
// slab whose waves of units take least, a wave costing its slab and `overhead` blocks (pipeline fill, adding the tile), for at
// most `most` slabs; equal costs go to the fewer slabs.  Only the largest count of every number of waves can be the best, and
// only those are looked at: a scan of all counts took 15 us of the host at 300,000 tokens of a layer of one tile.
inline int64_t plan_slab(int64_t blocks, int64_t tiles, int64_t slots, int64_t overhead, int64_t most) {
  most = std::max<int64_t>(1, std::min(most, blocks));
  int64_t best_per = blocks, best = INT64_MAX;
  for (int64_t n = 0; n < most;) {
    const int64_t waves = ((n + 1) * tiles + slots - 1) / slots;
    n = std::min(most, waves * slots / tiles);
    const int64_t per = (blocks + n - 1) / n, used = (blocks + per - 1) / per;
    const int64_t cost = (used * tiles + slots - 1) / slots * (per + overhead);
    if (cost < best) { best = cost; best_per = per; }
  }
  return best_per;
}

}  // namespace isopo
