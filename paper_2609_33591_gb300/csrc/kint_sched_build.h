// Host side of the item schedules: which kernels have one, how it is built, and the store of the
// schedules built so far.  Plain C++, no CUDA.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <tuple>
#include <utility>
#include <vector>

#include "kint_sched.h"

namespace kint {

// Items are (block, head) pairs, item = block * BH + head, the longest blocks first: query blocks of
// the forward passes and dQ, key blocks of the single-pass backward and dK.
enum SchedKind { SCHED_STATS = 0, SCHED_MAIN = 1, SCHED_FUSED = 2, SCHED_DQ = 3, SCHED_DK = 4 };

// Heads go in groups whose tiles (what every item of a head streams) fit in this share of the
// 129 MB L2, all items of a group before the next group's; with every head's longest item first
// the tiles were read from DRAM again for each block.  Between 24 and 72 MB the times are the
// same within 2 %.  B=4 H=16 T=2048 d=128 (200 MB of tiles in dQ and dK): pass 1 78 -> 75 us,
// pass 2 136 -> 124, dQ 248 -> 232, dK 238 -> 231; B=8 H=12 T=1024 3xTF32 dQ 147 -> 132,
// dK 131 -> 127.  Not the single-pass backward, where groups of 16 to 48 of 96 heads gave nothing.
// A call somewhat above the limit is split too, although one group balances the CTAs better: softmax
// at B=8 H=12 T=1024 (50 MB of tiles in pass 2, longest CTA 1.14 of the mean against 1.10) took 186.1 us
// forward and backward in two groups, 186.9 in one.
constexpr double kGroupBytes = 48e6;

// What a schedule depends on.  nqt: 64-row query tiles (kinds whose items are key blocks; else 0);
// hg: the heads per group that kGroupBytes gives, hg_min: the fewest that leave no CTA without items.
struct SchedKey {
  int kind, nitems, ngrid, BH, nqb, nqt, hg, hg_min;
  bool operator<(const SchedKey& o) const {
    return std::tie(kind, nitems, ngrid, BH, nqb, nqt, hg, hg_min) <
           std::tie(o.kind, o.nitems, o.ngrid, o.BH, o.nqb, o.nqt, o.hg, o.hg_min);
  }
};

// head_bytes: bytes of one tensor of a head in the precision the kernel reads (hi and lo parts).
inline SchedKey sched_key(int kind, int nitems, int ngrid, int BH, int nqb, int nqt, double head_bytes) {
  const bool keys = kind == SCHED_FUSED || kind == SCHED_DK;
  const int tensors = kind == SCHED_FUSED ? 0 : kind == SCHED_STATS ? 1 : kind == SCHED_MAIN ? 2 : 3;
  const int ng = (int)std::ceil(tensors * head_bytes * BH / kGroupBytes);
  // at least as many items as CTAs in a group (a group of one head of 128 blocks on 152 SMs took
  // 5 % longer than groups of two)
  const int hg_min = std::min(BH, (ngrid + nqb - 1) / nqb);
  const int hg = ng <= 1 ? BH : std::max(hg_min, (BH + ng - 1) / ng);
  return SchedKey{kind, nitems, ngrid, BH, nqb, keys ? nqt : 0, hg, hg_min};
}

// The schedule of a key: longest processing time first.  An item costs a + tiles (a = its fixed
// cost in tiles: operand loads, epilogue, measured per CTA), and a group's items in decreasing cost
// each go to the CTA with the least work so far, ties to the lower CTA.  Of the group sizes from hg
// down to half of it, the one whose longest CTA is shortest.
// A build runs in the first call of every new shape (a ragged batch meets new lengths all the time),
// so it is kept to tens of microseconds; a search of all CTAs for each item took 0.5 to 4 ms per
// kernel (forward and backward at B=4 H=16 d=128, T = 1027 .. 2435: the first call of a length took
// 1.4 ms more than the next ones, now 0.1).  Work is counted in units that make every cost a whole number, and the CTAs stand in
// buckets by their work, one bit per CTA: the least work never falls, and no CTA is ahead of it by
// more than one item's cost, so a ring of that many buckets holds them all.
inline void build_sched(const SchedKey& k, Sched& out) {
  // units per tile and fixed cost in units: 2.6 tiles for pass 2, 4 for dQ and dK, 2 for the others
  const bool keys = k.kind == SCHED_FUSED || k.kind == SCHED_DK;
  const int upt = k.kind == SCHED_MAIN ? 5 : 1;
  const int fixed = k.kind == SCHED_MAIN ? 13 : (k.kind == SCHED_DQ || k.kind == SCHED_DK) ? 4 : 2;
  // tiles of block b: 64-row query tiles of a key block, 64-key tiles of dQ's query blocks, 128-key
  // blocks of the forward passes'
  auto cost = [&](int b) {
    return fixed + upt * (keys ? k.nqt - 2 * b : (k.nqb - b) * (k.kind == SCHED_DQ ? 2 : 1));
  };
  const int words = (k.ngrid + 63) / 64;
  int ring = 64;
  while (ring <= cost(0)) ring *= 2;
  std::vector<uint64_t> bucket((size_t)ring * words);
  // (CTA of the i-th item in the order of the groups, and that order's group size)
  std::vector<uint16_t> who(k.nitems), best(k.nitems);
  int best_hg = 0, best_span = 0;
  auto for_items = [&](int hg, auto&& f) {  // groups, then blocks, then the group's heads
    for (int h0 = 0, i = 0; h0 < k.BH; h0 += hg)
      for (int b = 0; b < k.nqb; ++b)
        for (int h = h0; h < std::min(k.BH, h0 + hg); ++h, ++i) f(i, b, h);
  };
  for (int ng = (k.BH + k.hg - 1) / k.hg, hg = k.hg, last = 0; best_hg == 0 || (2 * hg >= k.hg && hg >= k.hg_min);
       ++ng, hg = (k.BH + ng - 1) / ng) {
    if (hg != last) {
      last = hg;
      std::fill(bucket.begin(), bucket.end(), 0);
      for (int c = 0; c < k.ngrid; ++c) bucket[c / 64] |= 1ull << (c % 64);
      int least = 0, span = 0;
      for_items(hg, [&](int i, int b, int) {
        uint64_t* w = nullptr;
        int j = 0;
        for (;; ++least) {  // the least work with a CTA, and its lowest CTA
          w = &bucket[(size_t)(least & (ring - 1)) * words];
          for (j = 0; j < words && w[j] == 0; ++j) {
          }
          if (j < words) break;
        }
        const uint64_t bit = w[j] & (~w[j] + 1);
        w[j] ^= bit;
        const int load = least + cost(b);
        bucket[(size_t)(load & (ring - 1)) * words + j] |= bit;
        span = std::max(span, load);
        who[i] = (uint16_t)(64 * j + __builtin_ctzll(bit));
      });
      if (best_hg == 0 || span < best_span) {
        best.swap(who);
        best_hg = hg;
        best_span = span;
      }
    }
    if (k.hg == k.BH || hg <= 1) break;
  }
  std::memset(&out, 0, sizeof(out));
  out.n = k.nitems;
  for (int i = 0; i < k.nitems; ++i) ++out.off[best[i] + 1];
  for (int c = 0; c < k.ngrid; ++c) out.off[c + 1] = (uint16_t)(out.off[c + 1] + out.off[c]);
  std::vector<uint16_t> pos(out.off, out.off + k.ngrid);
  for_items(best_hg, [&](int i, int b, int h) { out.idx[pos[best[i]]++] = (uint16_t)(b * k.BH + h); });
}

// The schedules built so far, kMax of them: a further one takes the place of the oldest (a call that
// holds that one keeps it alive), so how a shape runs does not depend on the shapes before it.  A
// call at d = 128 or under 3xTF32 uses four, so the store serves 256 such shapes without building
// again, in 5 MB.  A schedule is built outside the lock (two threads may build the same one; the
// first to finish is kept), so that a call never waits for another's build.
class SchedStore {
 public:
  using Ptr = std::shared_ptr<const Sched>;
  static constexpr size_t kMax = 1024;
  static Ptr none() {
    static const Sched z{};
    return Ptr(std::shared_ptr<void>(), &z);
  }
  // The schedule of `k`; none where one does not apply, and where memory ran out (the snake order gives
  // the same results).
  Ptr get(const SchedKey& k) noexcept {
    if (k.ngrid >= k.nitems || k.ngrid > SCHED_MAX_CTAS || k.nitems > SCHED_MAX_ITEMS) return none();
    try {
      {
        std::lock_guard<std::mutex> lk(mu_);
        const auto it = map_.find(k);
        if (it != map_.end()) return it->second;
      }
      auto s = std::make_shared<Sched>();
      build_sched(k, *s);
      std::lock_guard<std::mutex> lk(mu_);
      const auto it = map_.find(k);
      if (it != map_.end()) return it->second;
      if (age_.size() < kMax) {
        age_.push_back(k);
      } else {
        map_.erase(age_[oldest_]);
        age_[oldest_] = k;
        oldest_ = (oldest_ + 1) % kMax;
      }
      return map_.emplace(k, std::move(s)).first->second;
    } catch (...) {
      return none();
    }
  }
  size_t size() {
    std::lock_guard<std::mutex> lk(mu_);
    return map_.size();
  }

 private:
  std::mutex mu_;
  std::map<SchedKey, Ptr> map_;
  std::vector<SchedKey> age_;  // the stored keys, in a ring from the oldest on once it is full
  size_t oldest_ = 0;
};

}  // namespace kint
