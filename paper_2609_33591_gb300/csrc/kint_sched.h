// Static item schedule of a persistent kernel, computed on the host (kint_sched_build.h) and
// passed as a launch parameter.  Plain data.
#pragma once
#include <cstdint>

namespace kint {

// CTA c takes the items idx[off[c]] .. idx[off[c+1] - 1] in that order.  n == 0: no schedule, the snake
// order (snake_item) instead.  2048 items: 16 heads of 16384 rows.
constexpr int SCHED_MAX_CTAS = 304, SCHED_MAX_ITEMS = 2048;
struct Sched {
  int n;
  uint16_t off[SCHED_MAX_CTAS + 1];
  uint16_t idx[SCHED_MAX_ITEMS];
};

}  // namespace kint
