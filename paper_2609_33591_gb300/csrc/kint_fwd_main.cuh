// Pass 2 of the forward (App. A): reconstruction of the weights on the row's grid,
// normalization and P V, as a template; its instantiations are split over two
// translation units that compile in parallel.
#pragma once
#include <cfloat>
#include "kint_dev.cuh"
#include "kint_launch.h"

namespace kint {

// Thread roles of k_fwd_main: NG groups of eight compute warps, then two MMA warps and the K
// (and Q, and output stores) and V^T producer warps.  NG = 2: one CTA per SM; NG = 1: two CTAs
// per SM, so that one item's start and epilogue run under the other's tiles.  The last
// warpgroup (MMA and producers) gives registers to the compute warpgroups: launched at 96
// (80) per thread, it keeps 64 (48) and they take 104 (96).
template <int NG>
struct MainT {
  static constexpr int NCOMP = 256 * NG, NTHR = NCOMP + 128;
  static constexpr int MMA_W = NCOMP / 32, MMA2_W = MMA_W + 1, KPROD_W = MMA_W + 2, VPROD_W = MMA_W + 3;
  static constexpr int REG_LAUNCH = NG == 2 ? 96 : 80, REG_COMP = NG == 2 ? 104 : 96, REG_AUX = NG == 2 ? 64 : 48;
  static constexpr int CTAS = 2 / NG, TMEM_COLS = 512 / CTAS;
  static_assert(NCOMP * REG_COMP + 128 * REG_AUX <= NTHR * REG_LAUNCH, "register shares exceed the launch allocation");
};
// Slots of the ring that carries the tiles' chunk sums to the V^T producer (a power of two, at
// least the score buffers plus the V^T slots: see sum_rows).
constexpr int CSR_M = 8;
constexpr int BK_M = 64;  // keys per tile

// ---------------------------------------------------------------------------
// Element work on one chunk of W keys of one row: the grid position u = acc * k1 + c0, the
// decisions (r, t, Nearest, FWM tail) and the weights w^L = e_r + t (e_{r+1} - e_r),
// w^N = (t >= 1/2 ? e_{r+1} : e_r), by table lookups in place of the exponential.
// MODE 0: a1 = forward weight; 1: also a2 = w^L for O_lerp; 2: a1 = w^L.
// Positions and round-down adds go two keys to an instruction (f32x2: the same roundings
// per element), because the pass is bound by issue slots and latency, not by its pipes.
// ---------------------------------------------------------------------------
template <int CAL, int REC, int MODE, bool DIAG, int W>
__device__ __forceinline__ void fwd_chunk(const float (&v)[W], float (&a1)[W], float (&a2)[W], int j0, int i,
                                          const RowGrid& g, float Kf, uint32_t tab, float sk1, float sc0,
                                          float& wm_acc, float& wl_acc) {
#pragma unroll
  for (int jj = 0; jj < W; jj += 2) {
    float wm[2], wl[2] = {0.f, 0.f};
    const float2 vv = make_float2(v[jj], v[jj + 1]);
    if constexpr (CAL == CAL_SOFTMAX || CAL == CAL_EXP8) {
      const float2 x = fma2(vv, make_float2(sk1, sk1), make_float2(sc0, sc0));
      wm[0] = ex2_approx(x.x);  // e^{s - M} (App. A, Softmax)
      wm[1] = ex2_approx(x.y);
      if constexpr (CAL == CAL_EXP8) {
        wm[0] = e4m3_rn(wm[0]);  // E4M3(e^{s - M})
        wm[1] = e4m3_rn(wm[1]);
      }
    } else if constexpr (CAL == CAL_EXPB) {
      float zb;
      wm[0] = bf16_exp_weight(__fadd_rn(__fmul_rn(vv.x, g.k1), g.c0), zb);  // bf16(e^{bf16(s - M)})
      wm[1] = bf16_exp_weight(__fadd_rn(__fmul_rn(vv.y, g.k1), g.c0), zb);
    } else if constexpr (CAL == CAL_FWM) {
      // v = 2u = acc * 2k1 + 2c0 (sk1, sc0) clamped to [-1, 2K]; floor(v) = q = 2r + [t >= 1/2]
      // indexes the half-bin table {alpha, beta, w^N} by the float bits of its round-down (entry q
      // at tab + 24 bits: sixteen neighbouring entries share no bank), with the tail (u < 0) on the two zero entries below q = 0:
      // w^L = alpha + v beta, w^N = the Nearest endpoint.  Same decisions as decode_u.
      constexpr bool need_wn = REC == REC_NEAREST && MODE != 2;
      constexpr bool need_wl = REC == REC_LERP || MODE != 0;
      float2 x = fma2(vv, make_float2(sk1, sk1), make_float2(sc0, sc0));
      x.x = fminf(fmaxf(x.x, -1.0f), Kf);  // Kf = 2K here
      x.y = fminf(fmaxf(x.y, -1.0f), Kf);
      const float2 q = add2_rd(x, make_float2(kMagic, kMagic));
      const uint32_t aa[2] = {tab + __float_as_uint(q.x) * kLineStride, tab + __float_as_uint(q.y) * kLineStride};
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const float vc = k ? x.y : x.x;
        if constexpr (need_wl) {
          const float2 e = lds_f2(aa[k]);
          wl[k] = __fmaf_rn(vc, e.y, e.x);
        }
        if constexpr (need_wn) wm[k] = lds_f32(aa[k] + 8u);
        else wm[k] = wl[k];
      }
    } else if constexpr (CAL == CAL_MINMAX && REC == REC_NEAREST && MODE == 0) {
      // only the Nearest endpoint: v = 2u (sk1, sc0) clamped to [0, 2K], q = floor(v), and the
      // row's table of e_{(q + 1) / 2} by q, rows 512 bytes apart (0x4B000000 * 512 = 0 mod 2^32)
      float2 x = fma2(vv, make_float2(sk1, sk1), make_float2(sc0, sc0));
      x.x = fminf(fmaxf(x.x, 0.0f), Kf);
      x.y = fminf(fmaxf(x.y, 0.0f), Kf);
      const float2 q = add2_rd(x, make_float2(kMagic, kMagic));
      wm[0] = lds_f32(tab + (__float_as_uint(q.x) << 9));
      wm[1] = lds_f32(tab + (__float_as_uint(q.y) << 9));
    } else {
      const float2 u = fma2(vv, make_float2(g.k1, g.k1), make_float2(g.c0, g.c0));
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const float uk = k ? u.y : u.x;
        float t, rf;
        uint32_t rb;
        decode_u(uk, Kf, t, rb, rf);
        // MinMax: this row's table, rows 1024 bytes apart; FWMR: one shared table, entries 8 bytes apart
        float2 e = lds_f2(fwm_like(CAL) ? tab + rb * 8u : tab + rb * 1024u);
        if constexpr (CAL == CAL_FWMR) {
          // below the window: the continued grid (negative r)
          const BelowPair bp = resolved_below(uk, g.hl, g.b0l);
          const bool below = uk < 0.0f;
          t = below ? bp.t : t;
          e = below ? make_float2(bp.e0, bp.e1) : e;
        }
        wl[k] = __fmaf_rn(t, __fsub_rn(e.y, e.x), e.x);
        const float wn = (t >= 0.5f) ? e.y : e.x;
        wm[k] = (REC == REC_NEAREST) ? wn : wl[k];
      }
    }
    if constexpr (DIAG) {
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const bool ok = (j0 + jj + k) <= i;
        wm[k] = ok ? wm[k] : 0.f;
        wl[k] = ok ? wl[k] : 0.f;
      }
    }
    if constexpr (MODE != 2) wm_acc = __fadd_rn(__fadd_rn(wm_acc, wm[0]), wm[1]);
    if constexpr (MODE != 0) wl_acc = __fadd_rn(__fadd_rn(wl_acc, wl[0]), wl[1]);
    a1[jj] = (MODE == 2) ? wl[0] : wm[0];
    a1[jj + 1] = (MODE == 2) ? wl[1] : wm[1];
    if constexpr (MODE == 1) {
      a2[jj] = wl[0];
      a2[jj + 1] = wl[1];
    }
  }
}

// Decision codes of one chunk for kint_attn_debug_bins (not on the timed path, but
// inlined into the main loop: the calibration is a template parameter so that each
// instantiation carries only its own branch).
template <int CAL, int W>
__device__ void fwd_debug_codes(const Params& p, const float (&v)[W], int j0, int i, int bh, const RowGrid& g,
                                float sk1, float sc0) {
  if (i >= p.T) return;
  for (int jj = 0; jj < W; ++jj) {
    const int j = j0 + jj;
    if (j >= p.T) break;
    uint8_t cb = 255, ci = 255;
    if (j <= i) {
      if constexpr (CAL == CAL_EXP8) {
        cb = ci = (uint8_t)e4m3_code(e4m3_rn(ex2_approx(__fmaf_rn(v[jj], sk1, sc0))));
      } else if constexpr (CAL == CAL_EXPB) {
        float zb;
        const float w = bf16_exp_weight(__fadd_rn(__fmul_rn(v[jj], g.k1), g.c0), zb);
        cb = (uint8_t)bf16_low_byte(zb);
        ci = (uint8_t)bf16_low_byte(w);
      } else if (CAL == CAL_SOFTMAX || g.nogrid) {
        cb = ci = 253;
      } else {
        const float u = __fmaf_rn(v[jj], g.k1, g.c0);
        float t, rf;
        uint32_t rb;
        decode_u(u, (float)p.Kint, t, rb, rf);
        if (CAL == CAL_FWM && u < 0.0f) {
          cb = ci = 254;
        } else if constexpr (CAL == CAL_FWMR) {
          // resolved: indices run below zero, stored as index + 128 saturated to [0, 252]
          const int r = u < 0.0f ? (int)floorf(u) : (int)rf;
          const float tt = u < 0.0f ? __fsub_rn(u, floorf(u)) : t;
          const int l = r + (tt >= 0.5f ? 1 : 0);
          ci = (uint8_t)min(max(r + 128, 0), 252);
          cb = (uint8_t)min(max(l + 128, 0), 252);
        } else {
          const int r = (int)rf;
          ci = (uint8_t)r;
          cb = (uint8_t)(r + (t >= 0.5f ? 1 : 0));
        }
      }
    }
    const size_t idx = ((size_t)bh * p.T + i) * p.T + j;
    if (p.bins) p.bins[idx] = cb;
    if (p.ivals) p.ivals[idx] = ci;
  }
}

// ---------------------------------------------------------------------------
// k_fwd_main.  Work items are (128-row query block, head) pairs, longest blocks first; a
// CTA takes the items sched_item(sch, 0), sched_item(sch, 1), ...  An item's keys come in
// 64-key tiles (an even number of them, except where the sequence ends).  Tile and stage
// counters run on across items, so the next item's first tiles load under the current
// epilogue.
//   compute warps: the groups take the tiles in turn; thread t of a group owns query row t % 128
//     (its TMEM lane) and 32 of the tile's keys.  While one group does the element work of
//     tile t, the products of tile t + 1 run and the other group (NG = 1: the other CTA)
//     works.  They also copy the next item's Q into TMEM (q_tmem) ahead of the epilogue, so
//     that its first S products run under the epilogue and S reads only K from shared memory.
//   MMA_WARP: S_b = Q K^T up to nbuf - 1 tiles ahead, P V of each tile once its weights are
//     stored; MMA2_WARP (MODE 1, TF32): P^L V.
//   KPROD / VPROD: K (and Q) tiles and V^T tiles through two rings, so that a K slot is
//     refilled as soon as its S completed and not when its P V has.  KPROD also issues the
//     TMA stores of the previous item's outputs once the ring holds the item's first tiles;
//     VPROD adds up the row sums W from the tiles' chunk sums (sum_rows).
// TMEM: score buffers S_b at [64 b, 64 b + 64), b < nbuf (the weights overwrite their
// scores as MMA operand A); an A2 buffer per group (w^L, or the tf32 lo part of A under
// 3xTF32) after them; O, then O_lerp; Q (hi[, lo]) with q_tmem.
// smem: Q (hi[, lo]) at sm_a (with q_tmem only on its way to TMEM: the next item's Q loads
// under the current item); the K ring at sm_stage0, the V^T ring at sm_v (nstage and
// nstage_v slots of sm_stage_bytes each); grid tables at sm_table; the row sums and the ring
// of chunk sums at sm_rows; the output staging tile(s) at sm_ostage, over the V^T ring
// (ost_alias: d = 128 and 3xTF32) where they do not fit beside it: V^T of the next item is
// the operand needed last, so it is the one that waits for the stores.
//
// What bounds it: at d = 64 the element work's issue slots, the shared-memory cycles that table
// lookups and MMA operands share, and the hand-offs between them; at d = 128 and under
// 3xTF32 the tensor pipe (48-49% active) and its operand loads.  Measured on GB300 (kernel
// alone, cold L2), against one 128-key stage and score buffer where two did not fit and
// eight compute warps: B=8 H=12 T=1024 d=64 FWM K=4 Prob-STE 67.8 -> 66.5 us (within a step 67.1 and
// 67.5: nothing gained there), softmax 46.6 -> 33.7, 3xTF32 144 -> 80; B=4 H=16 T=2048 d=128 FWM Weight-STE 254 -> 134; H=16 T=16384 d=128
// MinMax K=16 LERP 3417 -> 1516.
// ---------------------------------------------------------------------------
// Wait for the K tile in slot `stg`, S_b = Q K^T into score buffer b, commit to bar_s[b]
// (compute warps) and to the slot's bar_emptyK.  aQ: the TMEM column of Q (q_tmem).
template <bool X3>
__device__ __forceinline__ bool main_issue_s(const Params& p, RingPos stg, int b, uint64_t* bar_fullK,
                                             uint64_t* bar_emptyK, uint64_t* bar_s, const uint8_t* st0,
                                             const uint8_t* sQ, uint32_t tmem, uint32_t aQ) {
  const int s = stg.i, D = p.d;
  if (!mbar_wait_warp(&bar_fullK[s], stg.ph, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA)) return false;
  tc_fence_after();
  const uint8_t* sk = st0 + s * p.sm_stage_bytes;
  const uint32_t dcol = tmem + (uint32_t)b * BK_M;
  const int qtile = D * 512, ktile = D * BK_M * 4;
  if (p.q_tmem) {
    if constexpr (X3) {
      mma_tmem_smem(dcol, aQ + D, sk, BK_M, D, false);      // Q_lo K_hi
      mma_tmem_smem(dcol, aQ, sk + ktile, BK_M, D, true);   // Q_hi K_lo
      mma_tmem_smem(dcol, aQ, sk, BK_M, D, true);           // Q_hi K_hi
    } else {
      mma_tmem_smem(dcol, aQ, sk, BK_M, D, false);
    }
  } else if constexpr (X3) {
    mma_smem_smem(dcol, sQ + qtile, sk, BK_M, D, false);
    mma_smem_smem(dcol, sQ, sk + ktile, BK_M, D, true);
    mma_smem_smem(dcol, sQ, sk, BK_M, D, true);
  } else {
    mma_smem_smem(dcol, sQ, sk, BK_M, D, false);
  }
  mma_commit(&bar_s[b]);
  mma_commit(&bar_emptyK[s]);
  return true;
}

// HOOK: the instantiations of the test hook of the first Q wait (kint_test_expire_next_q_wait).  As a
// run-time switch it cost every launch plan up to 0.9 us of 157.
template <int CAL, int REC, int MODE, bool X3, int NG, bool HOOK>
__global__ void __launch_bounds__(MainT<NG>::NTHR, MainT<NG>::CTAS) k_fwd_main(const __grid_constant__ Maps maps, const Params p,
                                                      const __grid_constant__ Sched sch) {
  uint8_t* sm = smem_base();
  using T = MainT<NG>;
  constexpr int NCOMP = T::NCOMP;
  constexpr int parts = X3 ? 2 : 1;
  constexpr bool useA2 = MODE == 1 || X3, split = MODE == 1 && !X3;
  const int D = p.d, Kq = p.Kint, NS = p.nstage, NV = p.nstage_v, nbuf = p.nbuf;
  const int qtile = D * 512, ktile = D * BK_M * 4;
  uint8_t* sQ = sm + p.sm_a;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm + p.sm_bars);
  // Parity tells apart only neighbouring phases of a barrier, so none may complete twice between
  // two waits of one waiter: the next S into buffer b needs P V of the tile before in it, so its
  // weights, so its group's wait; and a group waiting on buffer b has seen a later S than the
  // one that used b before (S products complete in order).
  uint64_t* bar_s = bars;              // [4] S_b computed
  uint64_t* bar_pready = bars + 4;     // [4] the weights of buffer b stored by the tile's eight warps
  uint64_t* bar_pv = bars + 8;         // [NG] the product that read the group's A2 buffer complete
  [[maybe_unused]] uint64_t* bar_never = bars + 11;  // (of the four kept for bar_pv; NG <= 2) nothing arrives
  uint64_t* bar_q = bars + 12;         // Q of the item landed in smem
  uint64_t* bar_qfree = bars + 13;     // smem Q may be reloaded (q_tmem: Q copied into TMEM; else last S complete)
  uint64_t* bar_done = bars + 14;      // every product of the item complete
  uint64_t* bar_ofree = bars + 15;     // O / O_lerp read out of TMEM by every compute warp
  uint64_t* bar_ostg = bars + 16;      // output tile(s) staged by every compute warp
  uint64_t* bar_stfree = bars + 17;    // the staging area read by its stores
  uint64_t* bar_drain = bars + 18;     // MMA_WARP's clean-up commit
  uint64_t* bar_drain2 = bars + 19;    // MMA2_WARP's clean-up commit
  uint64_t* bar_cs = bars + 20;        // [8] a tile's chunk sums are in the ring
  uint64_t* bar_w = bars + 28;         // the item's row sums are published
  uint64_t* bar_fullK = bars + 29;     // [NS] K tile landed
  uint64_t* bar_emptyK = bar_fullK + NS;  // [NS] its S complete
  uint64_t* bar_fullV = bar_emptyK + NS;  // [NV] V^T tile landed
  uint64_t* bar_emptyV = bar_fullV + NV;  // [NV] its P V (and P^L V) complete
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bar_emptyV + NV);
  uint8_t* ostg = sm + p.sm_ostage;
  float* wsum = reinterpret_cast<float*>(sm + p.sm_rows);  // [item parity][W^N, W^L][128]
  float* cring = wsum + 4 * 128;  // [CSR_M][first, second chunk][128] chunk sums, then those of w^L
  const bool alias = p.ost_alias != 0, q_tmem = p.q_tmem != 0;
  // O and O_lerp staged side by side (one use of the area per item), or one after the other
  const bool two_phase = MODE == 1 && p.ost_n == 1;
  const int cA2 = BK_M * nbuf, cO = cA2 + (useA2 ? NG * BK_M : 0), cOL = cO + D, cQ = cOL + (MODE == 1 ? D : 0);
  const int tid = threadIdx.x, warp = warp_id_uniform();

  if (tid == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(&bar_fullK[s], 1);
      mbar_init(&bar_emptyK[s], 1);
    }
    for (int s = 0; s < NV; ++s) {
      mbar_init(&bar_fullV[s], 1);
      mbar_init(&bar_emptyV[s], split ? 2 : 1);
    }
    for (int b = 0; b < 4; ++b) {
      mbar_init(&bar_s[b], 1);
      mbar_init(&bar_pready[b], 8);
      mbar_init(&bar_pv[b], 1);
    }
    for (int b = 0; b < CSR_M; ++b) mbar_init(&bar_cs[b], 8);
    mbar_init(bar_w, 1);
    mbar_init(bar_q, 1);
    mbar_init(bar_qfree, q_tmem ? NCOMP / 32 : 1);
    mbar_init(bar_done, split ? 2 : 1);
    mbar_init(bar_ofree, NCOMP / 32);
    mbar_init(bar_ostg, NCOMP / 32);
    mbar_init(bar_stfree, 1);
    mbar_init(bar_drain, 1);
    mbar_init(bar_drain2, 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(tslot, T::TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_trigger();
  pdl_wait();  // everything below may read what the previous kernel wrote
  // With all 512 columns allocated the allocation starts at lane 0, column 0; a compile-time
  // base keeps the TMEM addresses of the issue paths in uniform registers.
  if (T::CTAS == 1 && threadIdx.x == 0 && *tslot != 0u) dev_flag(p.status, DEV_ERR_BOUNDS);
  const uint32_t tmem = T::CTAS == 1 ? 0u : *tslot;
  auto tiles_of = [&](int qb) { return min(2 * qb + 2, (p.T + BK_M - 1) / BK_M); };

  // (each warpgroup reallocates registers inside its own branch: ahead of a branch that both
  // share, ptxas holds the compute path to the fifth warpgroup's registers too)
  if (warp >= NCOMP / 32) {
    setmaxnreg_dec<T::REG_AUX>();
    if (warp == T::KPROD_W) {
      int g = 0, n = 0, use = 0;  // use: uses of the staging area stored so far
      int nq = 0;                 // Q tiles loaded
      RingPos ld;
      bool ok = true;
      // Q of the next item to load, once smem Q is free
      auto load_q = [&]() -> bool {
        const int item = sched_item(sch, nq);
        if (item >= p.nitems) return true;
        const int it = item_block(p, item), bh_ = item - it * p.BH;
        if (nq > 0 && !mbar_wait_warp(bar_qfree, (nq - 1) & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_SYNC)) return false;
        mbar_arrive_expect_tx(bar_q, parts * qtile);
        load_rows_tile(sQ, &maps.q, bar_q, D, 128, 0, (p.nqb - 1 - it) * 128, bh_);
        if (X3) load_rows_tile(sQ + qtile, &maps.q_lo, bar_q, D, 128, 0, (p.nqb - 1 - it) * 128, bh_);
        ++nq;
        return true;
      };
      // the staging area has been read by the stores issued: it may be written again
      auto release_staging = [&]() {
        tma_store_wait_read();
        if ((tid & 31) == 0) mbar_arrive(bar_stfree);
        __syncwarp();
      };
      // the outputs of item k, from the tiles the compute warps staged
      auto store_outputs = [&](int k) -> bool {
        const int item = sched_item(sch, k), it = item_block(p, item), bh_ = item - it * p.BH;
        const int q0 = (p.nqb - 1 - it) * 128;
        for (int ph = 0; ph < (two_phase ? 2 : 1); ++ph, ++use) {
          if (!mbar_wait_warp(bar_ostg, use & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_SYNC)) return false;
          store_rows_tile_boxed(ostg, (MODE == 2 || ph == 1) ? &maps.out_lerp : &maps.out, D, 64, q0, bh_, false);
          if (MODE == 1 && !two_phase)
            store_rows_tile_boxed(ostg + 128 * D * 4, &maps.out_lerp, D, 64, q0, bh_, false);
          if (two_phase && ph == 0) release_staging();
        }
        return true;
      };
      ok = load_q();
      for (int item = sched_item(sch, n); item < p.nitems && ok; item = sched_item(sch, ++n)) {
        const int it = item_block(p, item), qb = p.nqb - 1 - it, bh = item - it * p.BH, nkt = tiles_of(qb);
        if (!q_tmem && n > 0) ok = load_q();
        for (int kt = 0; kt < nkt && ok; ++kt, ++g, ld.next(NS)) {
          const int s = ld.i;
          if (g >= NS && !mbar_wait_warp(&bar_emptyK[s], ld.ph ^ 1u, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA)) {
            ok = false;
            break;
          }
          uint8_t* dst = sm + p.sm_stage0 + s * p.sm_stage_bytes;
          mbar_arrive_expect_tx(&bar_fullK[s], parts * ktile);
          load_rows_tile(dst, &maps.k, &bar_fullK[s], D, BK_M, 0, kt * BK_M, bh);
          if (X3) load_rows_tile(dst + ktile, &maps.k_lo, &bar_fullK[s], D, BK_M, 0, kt * BK_M, bh);
          if (kt == min(nkt, NS) - 1) {
            // the item's first tiles are on their way: now the next item's Q (this one's went into
            // TMEM before the previous epilogue), and the previous item's outputs
            if (q_tmem) ok = load_q();
            if (n > 0 && ok && !p.debug) {
              ok = store_outputs(n - 1);
              if (alias && ok) release_staging();
            }
          }
        }
        if (n > 0 && !alias && ok && !p.debug) release_staging();
      }
      if (ok && n > 0 && !p.debug) store_outputs(n - 1);
      tma_store_wait_all();
      // clean-up: the last K tiles and Q tile issued have landed
      drain_ring(bar_fullK, ld, g, NS, p.wait_ns, p.status);
      if (nq > 0) mbar_wait_warp(bar_q, (nq - 1) & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA);
    } else if (warp == T::VPROD_W) {
      int g = 0, n = 0, use = 0;
      RingPos ld;
      bool ok = true;
      // The row sums W, in one fixed order whatever the tiling: every 32-key chunk from its first
      // key (the compute threads), the chunks of the even (odd) 64-key tiles of the item in
      // sequence, even + odd.  The backward truncates P = w / W to TF32, where another last
      // bit of W is another P.  Lane l adds up rows l, l + 32, l + 64, l + 96.  A tile is summed
      // before the V^T slot it used is refilled, so the ring cannot be overrun: writing slot
      // G % 8 for tile G needs S(G), so P V(G - nbuf), so V^T(G - nbuf) loaded, so tile
      // G - nbuf - NV summed.
      const int lane = tid & 31;
      float we[4], wo[4], le[4], lo[4];
      int sg = 0, snkt = 0, skt = 0, sn = 0;  // tiles summed; the item being summed: its tiles, those summed, its number
      auto sum_rows = [&]() -> bool {
        const int sl = sg & (CSR_M - 1);
        if (!mbar_wait_warp(&bar_cs[sl], (uint32_t)(sg / CSR_M) & 1u, p.wait_ns, p.status, DEV_ERR_TIMEOUT_SYNC))
          return false;
        if (skt == 0) {
          const int item = sched_item(sch, sn);
          snkt = tiles_of(p.nqb - 1 - item_block(p, item));
#pragma unroll
          for (int k = 0; k < 4; ++k) we[k] = wo[k] = le[k] = lo[k] = 0.f;
        }
        const float* c = cring + sl * 256 + lane;
#pragma unroll
        for (int k = 0; k < 4; ++k) {  // (the tile's parity chooses the sum: swap, so that it is always we)
          const float w = __fadd_rn(__fadd_rn(we[k], c[32 * k]), c[128 + 32 * k]);
          we[k] = wo[k];
          wo[k] = w;
          if constexpr (MODE == 1) {
            const float* cl = c + CSR_M * 256;
            const float l = __fadd_rn(__fadd_rn(le[k], cl[32 * k]), cl[128 + 32 * k]);
            le[k] = lo[k];
            lo[k] = l;
          }
        }
        ++sg;
        if (++skt == snkt) {
          float* w = wsum + (sn & 1) * 256 + lane;
#pragma unroll
          for (int k = 0; k < 4; ++k) {  // (addition commutes: which of the two is the even tiles' does not matter)
            w[32 * k] = __fadd_rn(we[k], wo[k]);
            if constexpr (MODE == 1) w[128 + 32 * k] = __fadd_rn(le[k], lo[k]);
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_w);
          skt = 0;
          ++sn;
        }
        return true;
      };
      for (int item = sched_item(sch, n); item < p.nitems && ok; item = sched_item(sch, ++n)) {
        const int it = item_block(p, item), qb = p.nqb - 1 - it, bh = item - it * p.BH, nkt = tiles_of(qb);
        // with the ring as the previous item's output staging area, its sums come first (the
        // outputs are scaled by them), then its stores
        if (alias && !p.debug && n > 0) {
          while (ok && sg < g) ok = sum_rows();
          for (int ph = 0; ph < (two_phase ? 2 : 1) && ok; ++ph, ++use)
            ok = mbar_wait_warp(bar_stfree, use & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_SYNC);
        }
        for (int kt = 0; kt < nkt && ok; ++kt, ++g, ld.next(NV)) {
          const int s = ld.i;
          while (ok && sg <= g - NV) ok = sum_rows();
          if (!ok || (g >= NV && !mbar_wait_warp(&bar_emptyV[s], ld.ph ^ 1u, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA))) {
            ok = false;
            break;
          }
          uint8_t* dst = sm + p.sm_v + s * p.sm_stage_bytes;
          mbar_arrive_expect_tx(&bar_fullV[s], parts * ktile);
          load_rows_tile(dst, &maps.vt, &bar_fullV[s], BK_M, D, kt * BK_M, 0, bh);
          if (X3) load_rows_tile(dst + ktile, &maps.vt_lo, &bar_fullV[s], BK_M, D, kt * BK_M, 0, bh);
        }
      }
      while (ok && sg < g) ok = sum_rows();
      drain_ring(bar_fullV, ld, g, NV, p.wait_ns, p.status);
    } else if (warp == T::MMA_W) {
      const uint8_t* st0 = sm + p.sm_stage0;
      int n = 0;
      // K slot and buffer of the next S product; V slot, buffer and group of the tile being finished
      RingPos is, ib, cs, cb, cg;
      bool ok = true;
      const int ahead = nbuf - 1;  // S products issued ahead of the tile being finished
      for (int item = sched_item(sch, n); item < p.nitems && ok; item = sched_item(sch, ++n)) {
        const int nkt = tiles_of(p.nqb - 1 - item_block(p, item));
        ok = mbar_wait_warp(q_tmem ? bar_qfree : bar_q, n & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA);
        if (ok) tc_fence_after();
        int ns = 0;  // S products of the item issued
        auto next_s = [&]() {
          ok = main_issue_s<X3>(p, is, ib.i, bar_fullK, bar_emptyK, bar_s, st0, sQ, tmem, tmem + cQ);
          is.next(NS);
          ib.next(nbuf);
          if (++ns == nkt && ok && !q_tmem) mma_commit(bar_qfree);
        };
        while (ok && ns < nkt && ns < ahead) next_s();
        for (int kt = 0; kt < nkt && ok; ++kt, cs.next(NV), cb.next(nbuf), cg.next(NG)) {
          const int b = cb.i, s = cs.i;
          const uint8_t* vt = sm + p.sm_v + s * p.sm_stage_bytes;
          const bool acc = kt > 0;
          // S(kt + ahead): its buffer was last read by P V(kt - 1), which precedes it in issue order
          if (ns < nkt && ns <= kt + ahead) next_s();
          if (!ok) break;
          // V^T landed; the item's first P V overwrites O: the previous item's epilogue must have read it
          if (!mbar_wait_warp(&bar_fullV[s], cs.ph, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA) ||
              (kt == 0 && n > 0 && !mbar_wait_warp(bar_ofree, (n - 1) & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_SYNC))) {
            ok = false;
            break;
          }
          if (!mbar_wait_warp(&bar_pready[b], cb.ph, p.wait_ns, p.status, DEV_ERR_TIMEOUT_SYNC)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t A = tmem + b * BK_M;
          if constexpr (X3) {
            mma_tmem_smem(tmem + cO, tmem + cA2 + cg.i * BK_M, vt, D, BK_M, acc);  // A_lo V_hi (frees A2 first)
            mma_commit(&bar_pv[cg.i]);
            mma_tmem_smem(tmem + cO, A, vt + ktile, D, BK_M, true);  // A_hi V_lo
            mma_tmem_smem(tmem + cO, A, vt, D, BK_M, true);          // A_hi V_hi
          } else {
            mma_tmem_smem(tmem + cO, A, vt, D, BK_M, acc);
          }
          mma_commit(&bar_emptyV[s]);
        }
        if (ok) mma_commit(bar_done);
      }
      drain_mma(bar_drain, p.wait_ns, p.status);  // clean-up: no product still writes TMEM
    } else if (warp == T::MMA2_W) {
      // P^L V of every tile (split only): O_lerp += w^L V once the tile's weights are stored
      if constexpr (split) {
        int n = 0;
        RingPos cs, cb, cg;
        bool ok = true;
        for (int item = sched_item(sch, n); item < p.nitems && ok; item = sched_item(sch, ++n)) {
          const int nkt = tiles_of(p.nqb - 1 - item_block(p, item));
          for (int kt = 0; kt < nkt; ++kt, cs.next(NV), cb.next(nbuf), cg.next(NG)) {
            if (!mbar_wait_warp(&bar_pready[cb.i], cb.ph, p.wait_ns, p.status, DEV_ERR_TIMEOUT_SYNC) ||
                !mbar_wait_warp(&bar_fullV[cs.i], cs.ph, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA) ||
                (kt == 0 && n > 0 && !mbar_wait_warp(bar_ofree, (n - 1) & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_SYNC))) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint8_t* vt = sm + p.sm_v + cs.i * p.sm_stage_bytes;
            mma_tmem_smem(tmem + cOL, tmem + cA2 + cg.i * BK_M, vt, D, BK_M, kt > 0);
            mma_commit(&bar_pv[cg.i]);
            mma_commit(&bar_emptyV[cs.i]);
          }
          if (!ok) break;
          mma_commit(bar_done);
        }
        drain_mma(bar_drain2, p.wait_ns, p.status);  // clean-up: no product still writes TMEM
      }
    }
  } else {
    setmaxnreg_inc<T::REG_COMP>();
    const int row = tid & 127, cq = tid >> 7, cg = cq & 1, grp = cq >> 1, quarter = warp & 3;
    constexpr int NQ = 2 * NG;  // threads per row
    // The warps of a quarter share its 32 rows (their tables and outputs) and meet at this
    // barrier; nothing but the tile hand-offs couples the quarters.
    const int bar_rows = BAR_COMPUTE + 1 + quarter;
    constexpr bool mm_half = CAL == CAL_MINMAX && REC == REC_NEAREST && MODE == 0;
    constexpr bool half = CAL == CAL_FWM || mm_half;
    const float Kf = (float)(half ? 2 * Kq : Kq);
    int n = 0, use = 0;
    int g = 0, gn = grp;  // tiles of the CTA's earlier items; the group's next tile (over all items)
    int own = 0;          // 1 after the group's first tile
    uint32_t gph = 0;     // parity of the group's tiles so far
    int b = grp;          // its score buffer, and the phase of that buffer's barriers
    uint32_t bph = 0;
    bool failed = false;
    // The row extrema of an item, loaded one item ahead.
    int qb = 0, bh = 0;
    float M = 0.f, m = 0.f;
    auto load_extrema = [&](int item, int& qb_, int& bh_, float& M_, float& m_) {
      const int it = item_block(p, item);
      qb_ = p.nqb - 1 - it;
      bh_ = item - it * p.BH;
      const int i = qb_ * 128 + row;
      const size_t rw = (size_t)bh_ * p.T + i;
      M_ = i < p.T ? p.row_max[rw] : 0.0f;
      m_ = (CAL == CAL_MINMAX && i < p.T) ? p.row_min[rw] : 0.0f;
    };
    // The k-th item's Q rows from smem into TMEM (each thread its share of its row's columns),
    // handed to the MMA warp and the K producer through bar_qfree.
    auto q_to_tmem = [&](int k) -> bool {
      const bool ok = mbar_wait(bar_q, k & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA);
      if (ok) {
#pragma unroll 1
        for (int c = cq * (D / NQ); c < (cq + 1) * (D / NQ); c += 16) {
          staged16_to_tmem(tmem, cQ, sQ, row, c);
          if constexpr (X3) staged16_to_tmem(tmem, cQ + D, sQ + qtile, row, c);
        }
      }
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if ((tid & 31) == 0) mbar_arrive(bar_qfree);
      return ok;
    };
    int item = sched_item(sch, 0);
    if (item < p.nitems) {
      load_extrema(item, qb, bh, M, m);
      if (q_tmem) failed = !q_to_tmem(0);
      if constexpr (HOOK) {  // every warp but the first of each quarter waits on
        if (q_tmem && cq > 0) failed = !mbar_wait(bar_never, 0, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA);
      }
    }
    // Tables addressed by the float bits 0x4B000000 + index of the floored position.
    // FWM: one half-bin table of 24-byte line entries, q in [-2, 2K] at sm_table + 24 (q + 2)
    // (0x4B000000 * 24 = 0x08000000 mod 2^32).
    // FWMR: one shared pair table (e_r, e_{r+1}), r = 0 .. K - 1 (rb * 8 = 0x58000000 + 8 r).
    // MinMax: one pair table per row ([K][128], 1024 bytes per r: rb * 1024 wraps to r * 1024),
    // or for Nearest weights alone the endpoints by half bin ([2K + 1][128] floats); a
    // degenerate row's entries are 1, so its weights are 1 whatever the position.
    uint32_t tab = smem_u32(sm + p.sm_table) + (uint32_t)row * (mm_half ? 4u : 8u);
    if constexpr (CAL == CAL_FWM) {
      tab = smem_u32(sm + p.sm_table) + kLineStride * kHalfTail - 0x08000000u;
      if (tid < 2 * Kq + 1 + kHalfTail) {
        const float4 e = fwm_line_entry(p, tid - kHalfTail);
        float* dst = reinterpret_cast<float*>(sm + p.sm_table + tid * kLineStride);
        dst[0] = e.x;
        dst[1] = e.y;
        dst[2] = e.z;
      }
    } else if constexpr (CAL == CAL_FWMR) {
      tab = smem_u32(sm + p.sm_table) + 8u * kFwdTail - 0x58000000u;
      if (tid < Kq)
        *reinterpret_cast<float2*>(sm + p.sm_table + 8 * kFwdTail + tid * 8) =
            make_float2(p.fwm_e[tid], p.fwm_e[tid + 1]);
      if (tid < kFwdTail) *reinterpret_cast<float2*>(sm + p.sm_table + tid * 8) = make_float2(0.f, 0.f);
    }
    // The shared table is written; and a first Q wait that ran out in some warps sends every compute
    // warp past the items, because the others would wait for those at the item's barriers.
    failed = group_any(BAR_COMPUTE, NCOMP, failed);
    while (item < p.nitems && !failed) {
      const int nkt = tiles_of(qb), i = qb * 128 + row;
      const bool row_ok = i < p.T;
      const size_t rw = (size_t)bh * p.T + (row_ok ? i : 0);
      const RowGrid gr = row_grid(p, M, m);
      // softmax: base-2 exponent coefficients; the half-bin forms: the position v = 2u =
      // acc * 2k1 + 2c0 (an exact doubling of u)
      const float sk1 = half ? 2.0f * gr.k1 : p.scale * 1.4426950408889634f;
      const float sc0 = half ? 2.0f * gr.c0 : -M * 1.4426950408889634f;
      // the next item and its extrema, which load under this item's tiles
      const int next = sched_item(sch, n + 1);
      int nqb_ = 0, nbh_ = 0;
      float nM = 0.f, nm = 0.f;
      if (next < p.nitems) load_extrema(next, nqb_, nbh_, nM, nm);
      if constexpr (mm_half) {
        for (int r = cq; r <= Kq; r += NQ) {
          const float e = gr.nogrid ? 1.0f : grid_value(p, gr, r);
          float* t0 = reinterpret_cast<float*>(sm + p.sm_table) + row;
          if (r > 0) t0[(2 * r - 1) * 128] = e;
          t0[2 * r * 128] = e;
        }
      } else if constexpr (CAL == CAL_MINMAX) {
        for (int r = cq; r < Kq; r += NQ) {
          const float2 e = gr.nogrid ? make_float2(1.f, 1.f)
                                     : make_float2(grid_value(p, gr, r), grid_value(p, gr, r + 1));
          *reinterpret_cast<float2*>(sm + p.sm_table + (size_t)r * 1024 + row * 8) = e;
        }
      }
      if constexpr (CAL == CAL_MINMAX) group_sync(bar_rows, 32 * NQ);

      const int i0w = qb * 128 + quarter * 32;  // this warp's first row
      for (; gn - g < nkt; gn += NG, own = 1) {
        const int kt = gn - g;
        if (!mbar_wait(&bar_s[b], bph, p.wait_ns, p.status, DEV_ERR_TIMEOUT_MMA)) {
          failed = true;
          break;
        }
        tc_fence_after();
        // the thread's 32 keys; with an A2 operand as two halves, which bounds the live registers
        // (rolled, because the element work is the instruction cache's largest tenant)
        constexpr int W = useA2 ? 16 : 32;
        const int sl = gn & (CSR_M - 1);
        float cm = 0.f, cl = 0.f;
#pragma unroll 1
        for (int h = 0; h < 32 / W; ++h) {
          const int c0 = cg * 32 + h * W, j0 = kt * BK_M + c0;
          float v[W], a1[W], a2[W];
          tmem_ldw<W>(lane_addr(tmem, b * BK_M + c0), v);
          tmem_ld_wait();
          if (p.debug) fwd_debug_codes<CAL>(p, v, j0, i, bh, gr, sk1, sc0);
          if (j0 > i0w + 31) {  // every key of the chunk lies after every row of the warp
#pragma unroll
            for (int q = 0; q < W; ++q) a1[q] = a2[q] = 0.f;
          } else {
            if (j0 + W - 1 > i0w)
              fwd_chunk<CAL, REC, MODE, true, W>(v, a1, a2, j0, i, gr, Kf, tab, sk1, sc0, cm, cl);
            else
              fwd_chunk<CAL, REC, MODE, false, W>(v, a1, a2, j0, i, gr, Kf, tab, sk1, sc0, cm, cl);
            if constexpr (X3) {
#pragma unroll
              for (int q = 0; q < W; ++q) {
                const float hi = tf32_rna(a1[q]);
                a2[q] = __fsub_rn(a1[q], hi);
                a1[q] = hi;
              }
            }
          }
          tmem_stw<W>(lane_addr(tmem, b * BK_M + c0), a1);
          if constexpr (useA2) {
            // the A2 buffer is an operand of the group's previous tile's product until it completes
            if (h == 0 && own &&
                !mbar_wait(&bar_pv[grp], gph ^ 1u, p.wait_ns, p.status, DEV_ERR_TIMEOUT_MMA)) {
              failed = true;
              break;
            }
            tmem_stw<W>(lane_addr(tmem, cA2 + grp * BK_M + c0), a2);
          }
        }
        cring[sl * 256 + cg * 128 + row] = MODE == 2 ? cl : cm;
        if constexpr (MODE == 1) cring[(CSR_M + sl) * 256 + cg * 128 + row] = cl;
        if (failed) break;
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if ((tid & 31) == 0) {
          mbar_arrive(&bar_pready[b]);
          mbar_arrive(&bar_cs[sl]);
        }
        gph ^= 1u;  // the group's next tile
        b += NG;
        if (b >= nbuf) {  // (nbuf >= 2)
          b -= nbuf;
          bph ^= 1u;
        }
      }
      g += nkt;
      if (!failed) failed = !mbar_wait(bar_done, n & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_MMA);
      tc_fence_after();
      // every S of the item is complete: the next item's Q goes in under the epilogue
      if (!failed && q_tmem && next < p.nitems) failed = !q_to_tmem(n + 1);
      if (!failed) failed = !mbar_wait(bar_w, n & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_SYNC);
      if (!failed && !p.debug && use > 0)  // the staging area's previous stores have read it
        failed = !mbar_wait(bar_stfree, (use - 1) & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_SYNC);
      failed = group_any(bar_rows, 32 * NQ, failed);
      if (failed) break;
      const float Wmt = wsum[(n & 1) * 256 + row];  // (MODE 2: the sum of w^L)
      const float Wlt = MODE == 1 ? wsum[(n & 1) * 256 + 128 + row] : Wmt;
      if (!p.debug) {
        // O = (sum_j w_j V_j) / W (and O_lerp): each thread scales its share of its row's d
        // columns into a swizzled tile for the TMA store
        auto stage_out = [&](uint8_t* tile, int col, float W) {
          const float inv = row_ok ? 1.0f / W : 0.0f;
          for (int c = cq * (D / NQ); c < (cq + 1) * (D / NQ); c += 16) {
            float v[16];
            tmem_ld16(lane_addr(tmem, col + c), v);
            tmem_ld_wait();
#pragma unroll
            for (int q = 0; q < 16; ++q) v[q] *= inv;
            row16_to_staged(tile, row, c, v);
          }
        };
        auto hand_over = [&]() {
          fence_async_smem();
          __syncwarp();
          if ((tid & 31) == 0) mbar_arrive(bar_ostg);
          ++use;
        };
        stage_out(ostg, cO, Wmt);
        if (MODE == 1 && !two_phase) stage_out(ostg + 128 * D * 4, cOL, Wlt);
        if (MODE == 1 && two_phase) {
          hand_over();
          failed = !mbar_wait(bar_stfree, (use - 1) & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_SYNC);
          failed = group_any(bar_rows, 32 * NQ, failed);
          if (failed) break;
          stage_out(ostg, cOL, Wlt);
        }
        // the accumulators go back to the MMA warps for the next item
        tc_fence_before();
        hand_over();
        if ((tid & 31) == 0) mbar_arrive(bar_ofree);
        if (row_ok && cq == 0) {
          if (MODE != 2) p.W[rw] = Wmt;
          if (MODE != 0 && p.W_lerp) p.W_lerp[rw] = Wlt;
        }
      } else {
        tc_fence_before();
        __syncwarp();
        if ((tid & 31) == 0) mbar_arrive(bar_ofree);
      }
      item = next;
      qb = nqb_;
      bh = nbh_;
      M = nM;
      m = nm;
      ++n;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, T::TMEM_COLS);
}

template <int CAL, int REC, int MODE, bool X3, int NG, bool HOOK = false>
static cudaError_t launch_main_n(const Maps& maps, const Params& p, int smem_bytes, cudaStream_t s, const Sched& sch) {
  auto kern = k_fwd_main<CAL, REC, MODE, X3, NG, HOOK>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, dim3((unsigned)p.ngrid), dim3(MainT<NG>::NTHR), smem_bytes, s, maps, p, sch);
}
template <int CAL, int REC, int MODE, bool X3>
static cudaError_t launch_main_t(const Maps& maps, const Params& p, int smem_bytes, cudaStream_t s, const Sched& sch) {
  // one grid with a shared table and one with a table per row (a barrier at the item's start)
  constexpr bool hooked = !X3 && MODE == 0 && ((CAL == CAL_FWM && REC == REC_NEAREST) || (CAL == CAL_MINMAX && REC == REC_LERP));
  if constexpr (hooked) {
    if (p.expire_wait)
      return p.main_groups == 1 ? launch_main_n<CAL, REC, MODE, X3, 1, true>(maps, p, smem_bytes, s, sch)
                                : launch_main_n<CAL, REC, MODE, X3, 2, true>(maps, p, smem_bytes, s, sch);
  }
  if constexpr (!X3 && MODE == 0) {
    if (p.main_groups == 1) return launch_main_n<CAL, REC, MODE, X3, 1>(maps, p, smem_bytes, s, sch);
  }
  return launch_main_n<CAL, REC, MODE, X3, 2>(maps, p, smem_bytes, s, sch);
}

// One calibration without a surrogate placement (the exponentials).
template <int CAL>
static cudaError_t launch_main_exp(const Maps& maps, const Params& p, int smem_bytes, cudaStream_t s, const Sched& sch) {
  return p.x3 ? launch_main_t<CAL, REC_LERP, 0, true>(maps, p, smem_bytes, s, sch)
              : launch_main_t<CAL, REC_LERP, 0, false>(maps, p, smem_bytes, s, sch);
}
// One calibration with a grid: LERP, or Nearest with the launch's product selection.
template <int CAL>
static cudaError_t launch_main_grid(const Maps& maps, const Params& p, int smem_bytes, cudaStream_t s, const Sched& sch) {
  if (p.recon == REC_LERP)
    return p.x3 ? launch_main_t<CAL, REC_LERP, 0, true>(maps, p, smem_bytes, s, sch)
                : launch_main_t<CAL, REC_LERP, 0, false>(maps, p, smem_bytes, s, sch);
  if (p.pv_sel == PV_MAIN)
    return p.x3 ? launch_main_t<CAL, REC_NEAREST, 0, true>(maps, p, smem_bytes, s, sch)
                : launch_main_t<CAL, REC_NEAREST, 0, false>(maps, p, smem_bytes, s, sch);
  if (p.pv_sel == PV_MAIN_LERP) return launch_main_t<CAL, REC_NEAREST, 1, false>(maps, p, smem_bytes, s, sch);
  return launch_main_t<CAL, REC_NEAREST, 2, true>(maps, p, smem_bytes, s, sch);
}

}  // namespace kint
