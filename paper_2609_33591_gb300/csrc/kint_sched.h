// Static item schedule of a persistent kernel, computed on the host (kint_sched_build.h) and
// passed as a launch parameter.  Plain data.
#pragma once
#include <cstdint>

namespace kint {

// CTA c takes the items idx[off[c]] .. idx[off[c+1] - 1] in that order.  n == 0: no schedule, the snake
// order (snake_item) instead.  A schedule travels in each launch's parameters (4.7 KB), which bounds its
// items.  Above the bound every head's longest block comes first again, and the tiles are read from
// DRAM for each block: 256 heads of T=2048 at d=128 (4096 items) take 722 us in pass 2 and 1208 in dQ
// against 124 and 231 for 64 heads, 384 heads of T=1024 under 3xTF32 568 in dQ against 131 for 96.
constexpr int SCHED_MAX_CTAS = 304, SCHED_MAX_ITEMS = 2048;
struct Sched {
  int n;
  uint16_t off[SCHED_MAX_CTAS + 1];
  uint16_t idx[SCHED_MAX_ITEMS];
};

}  // namespace kint
