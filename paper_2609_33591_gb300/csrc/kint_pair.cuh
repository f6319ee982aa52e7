// Product pipeline shared by the dQ and dK kernels at d = 128 and under 3xTF32.  Both form, per
// tile of 64 rows,
//   S = A1 X^T,  g = A2 Y^T,  acc += dS XT^T     (dQ: A1 = Q, A2 = dO, X = K, Y = V, XT = K^T;
//                                                 dK: A1 = K, A2 = V, X = Q, Y = dO, XT = Q^T)
// with A1, A2 the 128 rows of the item (hi, lo under 3xTF32).
//
// TMEM: A1 [0, 128), two score buffers S_b | g_b at 128 + 128 b, the accumulators from 384 on.
// A2 is read from shared memory, so that two 64-row score buffers fit: with both operands in
// TMEM one fitted, and products and element work took turns; two 32-row buffers instead made
// products of N = 32, which take as long as those of N = 64 (48-55 cycles against 33-48).
// smem: A2 at sm_a (also the next item's A1 on its way into TMEM, once the last g has read
// A2); rings of X, Y and XT tiles at sm_x, sm_y, sm_xt (nx, ny, nxt slots of tile_bytes each),
// freed one by one as the product that reads each completes: three separate rings, because
// 192 KB hold no two stages of all three.  dK's row records have a ring of their own.
// Warps: a producer for A1, A2, X, Y and the records, one for XT, an MMA warp for S, g and one
// for acc, each on another SM sub-partition.
#pragma once
#include <type_traits>

#include "kint_bwd_common.cuh"

namespace kint {

// Item order of a kernel: a host schedule for the pair pipeline, the snake order otherwise (at
// d = 64 the snake order measured better: MinMax dQ 67.5 against 72 us).
template <bool PAIR>
using ItemOrder = std::conditional_t<PAIR, Sched, SnakeOrder>;

constexpr int PAIR_T = 64;  // rows per tile

// The item's operand rows [orow, orow + 128) and its nt tiles, from row row0, of head bh.
struct PairItem {
  int bh, orow, row0, nt;
  bool ok;
};

struct PairBars {
  uint64_t *fullX, *emptyX, *fullY, *emptyY, *fullT, *emptyT;  // [2] tile landed / read by its product
  uint64_t *fullR, *emptyR;   // [2] records landed / read by every compute warp (dK)
  uint64_t *sfull, *pready, *accdone;  // [2] S_b, g_b computed / dS stored / read by acc
  uint64_t *done;   // every product of the item complete
  uint64_t *kst;    // A1 staged in smem
  uint64_t *ops;    // A1 in TMEM (the staging area free)
  uint64_t *v;      // A2 landed
  uint64_t *vfree;  // the item's last g complete
  uint64_t *drain;  // clean-up commits of the two MMA warps
};
constexpr int PAIR_NBARS = 28;

__device__ __forceinline__ PairBars pair_bars(uint64_t* b) {
  return PairBars{b,      b + 2,  b + 4,  b + 6,  b + 8,  b + 10, b + 12, b + 14, b + 16,
                  b + 18, b + 20, b + 22, b + 23, b + 24, b + 25, b + 26, b + 27};
}
__device__ __forceinline__ void pair_init(const PairBars& B, int compute_warps) {
  for (int s = 0; s < 2; ++s) {
    mbar_init(&B.fullX[s], 1);
    mbar_init(&B.emptyX[s], 1);
    mbar_init(&B.fullY[s], 1);
    mbar_init(&B.emptyY[s], 1);
    mbar_init(&B.fullT[s], 1);
    mbar_init(&B.emptyT[s], 1);
    mbar_init(&B.fullR[s], 1);
    mbar_init(&B.emptyR[s], compute_warps);
    mbar_init(&B.sfull[s], 1);
    mbar_init(&B.pready[s], compute_warps);
    mbar_init(&B.accdone[s], 1);
  }
  mbar_init(B.done, 1);
  mbar_init(B.kst, 1);
  mbar_init(B.ops, compute_warps);
  mbar_init(B.v, 1);
  mbar_init(B.vfree, 1);
  mbar_init(B.drain, 2);
}

// The natural maps (64-row boxes) of A1, A2, X, Y and the transposed one of X, hi and lo.
struct PairMaps {
  const CUtensorMap *a1, *a1_lo, *a2, *a2_lo, *x, *x_lo, *y, *y_lo, *xt, *xt_lo;
};

// Producer of A1, A2, X, Y and (rec_load, when REC) the tile's records: get(n) is the CTA's
// n-th item, rec_load(item, tile, dst, bar) issues a tile's records.
template <bool REC, class Get, class RecLoad>
__device__ __forceinline__ void pair_producer(const Params& p, const PairMaps& m, const PairBars& B, uint8_t* sm,
                                              Get get, RecLoad rec_load) {
  const int D = p.d, parts = p.x3 ? 2 : 1, tile = PAIR_T * D * 4, ops = 128 * D * 4;
  int n = 0, gx = 0, gy = 0, gr = 0, na = 0, nv = 0;  // item; loads issued of each kind
  RingPos x, y, r;
  bool ok = true;
  auto load_a = [&](const CUtensorMap* hi, const CUtensorMap* lo, uint64_t* bar, const PairItem& it) {
    mbar_arrive_expect_tx(bar, parts * ops);
    load_rows_tile_boxed(sm + p.sm_a, hi, bar, D, 128, PAIR_T, 0, it.orow, it.bh);
    if (p.x3) load_rows_tile_boxed(sm + p.sm_a + ops, lo, bar, D, 128, PAIR_T, 0, it.orow, it.bh);
  };
  auto load_t = [&](uint8_t* dst, const CUtensorMap* hi, const CUtensorMap* lo, uint64_t* bar, int row, int bh) {
    mbar_arrive_expect_tx(bar, parts * tile);
    load_rows_tile(dst, hi, bar, D, PAIR_T, 0, row, bh);
    if (p.x3) load_rows_tile(dst + tile, lo, bar, D, PAIR_T, 0, row, bh);
  };
  PairItem it = get(0);
  if (it.ok) {
    load_a(m.a1, m.a1_lo, B.kst, it);
    ++na;
  }
  while (it.ok && ok) {
    for (int t = 0; t < it.nt; ++t) {
      const int row = it.row0 + t * PAIR_T;
      if (gx >= p.nx && !mbar_wait_warp(&B.emptyX[x.i], x.ph ^ 1u, p.wait_ns, p.status, DEV_ERR_TIMEOUT_MMA)) {
        ok = false;
        break;
      }
      load_t(sm + p.sm_x + x.i * parts * tile, m.x, m.x_lo, &B.fullX[x.i], row, it.bh);
      x.next(p.nx);
      ++gx;
      if (gy >= p.ny && !mbar_wait_warp(&B.emptyY[y.i], y.ph ^ 1u, p.wait_ns, p.status, DEV_ERR_TIMEOUT_MMA)) {
        ok = false;
        break;
      }
      load_t(sm + p.sm_y + y.i * parts * tile, m.y, m.y_lo, &B.fullY[y.i], row, it.bh);
      y.next(p.ny);
      ++gy;
      if constexpr (REC) {
        if (gr >= 2 && !mbar_wait_warp(&B.emptyR[r.i], r.ph ^ 1u, p.wait_ns, p.status, DEV_ERR_TIMEOUT_SYNC)) {
          ok = false;
          break;
        }
        rec_load(it, row, sm + p.sm_rec + r.i * p.rec_bytes, &B.fullR[r.i]);
        r.next(2);
        ++gr;
      }
      if (t == 0) {  // A2, once A1 has gone from the staging area into TMEM
        if (!mbar_wait_warp(B.ops, n & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_SYNC)) {
          ok = false;
          break;
        }
        load_a(m.a2, m.a2_lo, B.v, it);
        ++nv;
      }
    }
    if (!ok) break;
    const PairItem nx = get(n + 1);
    if (nx.ok) {  // the next item's A1, once the last g has read A2
      if (!mbar_wait_warp(B.vfree, n & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_MMA)) {
        ok = false;
        break;
      }
      load_a(m.a1, m.a1_lo, B.kst, nx);
      ++na;
    }
    it = nx;
    ++n;
  }
  // clean-up: the last loads issued have landed
  drain_ring(B.fullX, x, gx, p.nx, p.wait_ns, p.status);
  drain_ring(B.fullY, y, gy, p.ny, p.wait_ns, p.status);
  if (REC) drain_ring(B.fullR, r, gr, 2, p.wait_ns, p.status);
  if (na > 0) mbar_wait_warp(B.kst, (na - 1) & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA);
  if (nv > 0) mbar_wait_warp(B.v, (nv - 1) & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA);
}

// Producer of the XT tiles.
template <class Get>
__device__ __forceinline__ void pair_producer_t(const Params& p, const PairMaps& m, const PairBars& B, uint8_t* sm,
                                                Get get) {
  const int D = p.d, parts = p.x3 ? 2 : 1, tile = PAIR_T * D * 4;
  int g = 0;
  RingPos s;
  bool ok = true;
  for (int n = 0; ok; ++n) {
    const PairItem it = get(n);
    if (!it.ok) break;
    for (int t = 0; t < it.nt; ++t, ++g, s.next(p.nxt)) {
      const int row = it.row0 + t * PAIR_T;
      if (g >= p.nxt && !mbar_wait_warp(&B.emptyT[s.i], s.ph ^ 1u, p.wait_ns, p.status, DEV_ERR_TIMEOUT_MMA)) {
        ok = false;
        break;
      }
      uint8_t* dst = sm + p.sm_xt + s.i * parts * tile;
      mbar_arrive_expect_tx(&B.fullT[s.i], parts * tile);
      load_rows_tile(dst, m.xt, &B.fullT[s.i], PAIR_T, D, row, 0, it.bh);
      if (p.x3) load_rows_tile(dst + tile, m.xt_lo, &B.fullT[s.i], PAIR_T, D, row, 0, it.bh);
    }
  }
  drain_ring(B.fullT, s, g, p.nxt, p.wait_ns, p.status);
}

// MMA warp of S and g.
template <class Get>
__device__ __forceinline__ void pair_mma_sg(const Params& p, const PairBars& B, const uint8_t* sm, Get get) {
  const int D = p.d, parts = p.x3 ? 2 : 1, tile = PAIR_T * D * 4;
  const uint8_t* a2 = sm + p.sm_a;
  const uint8_t* a2l = a2 + 128 * D * 4;
  int g = 0;
  RingPos x, y, b;
  bool ok = true;
  for (int n = 0; ok; ++n) {
    const PairItem it = get(n);
    if (!it.ok) break;
    ok = mbar_wait_warp(B.ops, n & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_SYNC);
    if (ok) tc_fence_after();
    for (int t = 0; t < it.nt && ok; ++t, ++g, x.next(p.nx), y.next(p.ny), b.next(2)) {
      // the buffer's dS has been read by acc of two tiles ago
      if (g >= 2 && !mbar_wait_warp(&B.accdone[b.i], b.ph ^ 1u, p.wait_ns, p.status, DEV_ERR_TIMEOUT_MMA)) ok = false;
      if (ok) ok = mbar_wait_warp(&B.fullX[x.i], x.ph, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA);
      if (!ok) break;
      tc_fence_after();
      const uint32_t cS = 128u + 128u * (uint32_t)b.i, cG = cS + 64u;
      const uint8_t* xs = sm + p.sm_x + x.i * parts * tile;
      if (p.x3) {
        mma_tmem_smem(cS, D, xs, PAIR_T, D, false);        // A1_lo X_hi
        mma_tmem_smem(cS, 0, xs + tile, PAIR_T, D, true);  // A1_hi X_lo
        mma_tmem_smem(cS, 0, xs, PAIR_T, D, true);         // A1_hi X_hi
      } else {
        mma_tmem_smem(cS, 0, xs, PAIR_T, D, false);
      }
      mma_commit(&B.emptyX[x.i]);
      if (t == 0) ok = mbar_wait_warp(B.v, n & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA);
      if (ok) ok = mbar_wait_warp(&B.fullY[y.i], y.ph, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA);
      if (!ok) break;
      tc_fence_after();
      const uint8_t* ys = sm + p.sm_y + y.i * parts * tile;
      if (p.x3) {
        mma_smem_smem(cG, a2l, ys, PAIR_T, D, false);
        mma_smem_smem(cG, a2, ys + tile, PAIR_T, D, true);
        mma_smem_smem(cG, a2, ys, PAIR_T, D, true);
      } else {
        mma_smem_smem(cG, a2, ys, PAIR_T, D, false);
      }
      mma_commit(&B.emptyY[y.i]);
      mma_commit(&B.sfull[b.i]);
      if (t + 1 == it.nt) mma_commit(B.vfree);
    }
  }
  drain_mma(B.drain, p.wait_ns, p.status);  // clean-up: no product still writes TMEM
}

// MMA warp of acc: acc(cS, cG, XT tile, first tile of the item).
template <class Get, class Acc>
__device__ __forceinline__ void pair_mma_acc(const Params& p, const PairBars& B, const uint8_t* sm, Get get, Acc acc) {
  const int D = p.d, parts = p.x3 ? 2 : 1, tile = PAIR_T * D * 4;
  RingPos s, b;
  bool ok = true;
  for (int n = 0; ok; ++n) {
    const PairItem it = get(n);
    if (!it.ok) break;
    for (int t = 0; t < it.nt; ++t, s.next(p.nxt), b.next(2)) {
      if (!mbar_wait_warp(&B.pready[b.i], b.ph, p.wait_ns, p.status, DEV_ERR_TIMEOUT_SYNC) ||
          !mbar_wait_warp(&B.fullT[s.i], s.ph, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t cS = 128u + 128u * (uint32_t)b.i;
      acc(cS, cS + 64u, sm + p.sm_xt + s.i * parts * tile, t == 0);
      mma_commit(&B.emptyT[s.i]);
      mma_commit(&B.accdone[b.i]);
    }
    if (ok) mma_commit(B.done);
  }
  drain_mma(B.drain, p.wait_ns, p.status);
}

// A compute thread's columns [c0, c0 + nc) of its row (TMEM lane) of the staged A1, into TMEM;
// handed to the MMA warp and the producer through ops.  n: the CTA's n-th item.
__device__ __forceinline__ bool pair_ops_to_tmem(const Params& p, const PairBars& B, const uint8_t* sm, int n, int row,
                                                 int c0, int nc) {
  const bool ok = mbar_wait(B.kst, n & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA);
  if (ok) {
#pragma unroll 1
    for (int c = c0; c < c0 + nc; c += 16) {
      staged16_to_tmem(0, 0, sm + p.sm_a, row, c);
      if (p.x3) staged16_to_tmem(0, p.d, sm + p.sm_a + 128 * p.d * 4, row, c);
    }
  }
  tmem_st_wait();
  tc_fence_before();
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(B.ops);
  return ok;
}

}  // namespace kint
