// dK/dV kernel of the backward (App. B), as a template: included by the
// translation unit of the plain kernels and by the one of the kernels that also
// accumulate the per-row score-gradient sums (RS), so the two compile in parallel.
#pragma once
#include "kint_pair.cuh"

namespace kint {

// Thread roles: sixteen compute warps (thread t owns key kb*128 + t%128 and the 16 query columns
// 16 (t/128) .. + 15 of each 64-query tile), the MMA warp, the producer warp and two idle
// warps (dK alone: a second MMA and a second producer warp, kint_pair.cuh).  The fifth
// warpgroup gives registers to the compute warpgroups: launched at 96 per thread, it keeps 64
// and they take 104.
constexpr int NCG_KV = 4, NCOMP_KV = 128 * NCG_KV, NTHR_KV = NCOMP_KV + 128;
constexpr int MMA_WARP_KV = NCOMP_KV / 32, PRODUCER_WARP_KV = MMA_WARP_KV + 1;
constexpr int REG_LAUNCH_KV = 96, REG_COMP_KV = 104, REG_AUX_KV = 64;
static_assert(NCOMP_KV * REG_COMP_KV + 128 * REG_AUX_KV <= NTHR_KV * REG_LAUNCH_KV,
              "register shares exceed the launch allocation");

// ---------------------------------------------------------------------------
// dK/dV kernel element work on one 32-query chunk of one key j: the forward
// probability P_ij and dS_ij = gamma_ij Delta_ij plus, at the arg-max / arg-min
// key of row i, c_M / n_max and c_m / n_min (Eq. full).  Row constants come
// from the RowRec array of the tile in shared memory (broadcast loads).
// ---------------------------------------------------------------------------
// DV / DK: which of P and dS the launch feeds to a product; the other is not formed (its record
// words and table entries are not read either: the shared-memory loads are this chunk's
// largest cost).
template <int CAL, int REC, bool FULLG, bool PROJ, bool MASKED, bool TIES, bool DV, bool DK, int W>
__device__ __forceinline__ void kv_chunk(const float (&sv)[W], const float (&gv)[W], float (&pa)[W],
                                         float (&da)[W], int j, int i0, int T, uint32_t recs, uint32_t tabs,
                                         uint32_t fwtab, uint32_t tstride, float Kf, float fwm_inv_h,
                                         float scale, float hl, float b0l) {
#pragma unroll
  for (int ii = 0; ii < W; ++ii) {
    const uint32_t ra = recs + ii * 64u;  // RowRec of query row i0 + ii
    const float4 r0 = lds_f4(ra);          // c0, k1, invWf, ga
    float4 r1 = make_float4(0.f, 0.f, 0.f, 0.f), r2 = r1;
    if constexpr (DK) r1 = lds_f4(ra + 16);                         // gb, cMn, amax, flags
    else if constexpr (CAL == CAL_MINMAX) r1.w = lds_f32(ra + 28);  // flags
    if constexpr (DK && CAL == CAL_MINMAX) r2 = lds_f4(ra + 32);    // inv_h, cmn, amin, -
    float gam = 0.f;
    if constexpr (DK) gam = __fmaf_rn(gv[ii], r0.w, r1.x);
    float pv = 0.f, ds = 0.f;
    if constexpr (CAL == CAL_SOFTMAX) {
      pv = ex2_approx(__fmaf_rn(sv[ii], r0.y, r0.x)) * r0.z;
      ds = pv * gam;
    } else if constexpr (CAL == CAL_EXP8) {
      // forward P from the E4M3-rounded weight; dS from the exponential itself
      const float we = ex2_approx(__fmaf_rn(sv[ii], r0.y, r0.x));
      if constexpr (DV) pv = e4m3_rn(we) * r0.z;
      ds = gam * we;
    } else if constexpr (CAL == CAL_EXPB) {
      // record holds -M, scale: z = acc * scale - M; the bfloat16 chain rule
      float zb;
      const float w = bf16_exp_weight(__fadd_rn(__fmul_rn(sv[ii], r0.y), r0.x), zb);
      pv = w * r0.z;
      ds = bf16_rn(__fmul_rn(bf16_rn(gam), w));
    } else if constexpr (fwm_like(CAL) && REC == REC_NEAREST) {
      // record holds 2k1, 2c0; Kf = 2K; fwtab: the half-bin table of (w^N, Delta_r / h)
      const float v = __fmaf_rn(sv[ii], r0.y, r0.x);
      const uint32_t qb = fwm_half_bits(v, Kf);
      float2 e = make_float2(0.f, 0.f);
      if constexpr (DV && DK) e = lds_f2(fwtab + qb * 8u);
      else if constexpr (DV) e.x = lds_f32(fwtab + qb * 8u);
      else e.y = lds_f32(fwtab + qb * 8u + 4u);
      if constexpr (CAL == CAL_FWMR) {
        // resolved: below the window, (w^N, Delta_r / h) of the continued grid (u = v / 2 exactly)
        const BelowPair bp = resolved_below(__fmul_rn(v, 0.5f), hl, b0l);
        const float2 eb = make_float2(bp.t >= 0.5f ? bp.e1 : bp.e0, __fmul_rn(__fsub_rn(bp.e1, bp.e0), fwm_inv_h));
        e = v < 0.0f ? eb : e;
      }
      pv = e.x * r0.z;
      ds = gam * e.y;
    } else {
      const float u = __fmaf_rn(sv[ii], r0.y, r0.x);
      float t, rf;
      uint32_t rb;
      decode_u(u, Kf, t, rb, rf);
      float2 e = lds_f2(fwm_like(CAL) ? fwtab + rb * 8u : tabs + ii * tstride + rb * 8u);
      if constexpr (CAL == CAL_FWMR) {
        const BelowPair bp = resolved_below(u, hl, b0l);
        const bool below = u < 0.0f;
        t = below ? bp.t : t;
        e = below ? make_float2(bp.e0, bp.e1) : e;
      }
      const float de = __fsub_rn(e.y, e.x);
      const float wl = __fmaf_rn(t, de, e.x);
      const float wn = (t >= 0.5f) ? e.y : e.x;
      float w = (REC == REC_NEAREST) ? wn : wl;
      ds = gam * (de * (CAL == CAL_MINMAX ? r2.x : fwm_inv_h));
      if constexpr (CAL == CAL_FWM) {
        const bool tail = u < 0.0f;
        w = tail ? 0.f : w;
        ds = tail ? 0.f : ds;
      }
      if constexpr (CAL == CAL_MINMAX) {
        const bool ng = (__float_as_int(r1.w) & REC_NOGRID) != 0;
        w = ng ? 1.f : w;
        ds = ng ? 0.f : ds;
      }
      pv = w * r0.z;
    }
    if constexpr (DK && FULLG && CAL != CAL_SOFTMAX) {
      ds += (j == __float_as_int(r1.z)) ? r1.y : 0.f;
      if constexpr (CAL == CAL_MINMAX) ds += (j == __float_as_int(r2.z)) ? r2.y : 0.f;
    } else if constexpr (DK && PROJ && CAL != CAL_SOFTMAX) {
      ds = __fsub_rn(ds, r1.y);  // detached, P1 projection: minus the row mean
    }
    if constexpr (MASKED) {
      const int iq = i0 + ii;
      const bool ok = iq >= j && iq < T;
      pv = ok ? pv : 0.f;
      ds = ok ? ds : 0.f;
    }
    if constexpr (DK && FULLG && TIES && CAL != CAL_SOFTMAX) {
      // rows with tied extrema (flagged per 64-row query tile by the dQ kernel): the tie set
      // is found by equality on the recomputed scores (rare, kept off the common path)
      const int fl = __float_as_int(r1.w);
      const int iq = i0 + ii;
      const bool okr = (!MASKED || (iq >= j && iq < T)) && (fl & (REC_TIEMAX | REC_TIEMIN)) && !(fl & REC_NOGRID);
      if (okr) {
        const float2 ext = lds_f2(ra + 48);  // M, m
        const float sc = __fmul_rn(sv[ii], scale);
        if ((fl & REC_TIEMAX) && sc == ext.x) ds += r1.y;
        if (CAL == CAL_MINMAX && (fl & REC_TIEMIN) && sc == ext.y) ds += r2.y;
      }
    }
    if constexpr (DV) pa[ii] = pv;
    if constexpr (DK) da[ii] = ds;
  }
}

// Per-row score-gradient sums (a diagnostic side output of the backward): the calling
// warp holds dS for 16 query rows (v[c], row r0 + c) at 32 keys (one per lane).  A
// butterfly reduce-scatter leaves the 32-key sum of row c = (lane >> 1) & 15 in lanes
// 2c and 2c + 1 (the xor-16 step keeps rows 8..15 in the upper half-warp, xor-8 rows
// +4, xor-4 rows +2, xor-2 rows +1, and xor-1 adds the pair); the even lane adds it to
// the row's global sums (fp32 atomics: the order of the additions is not fixed).
__device__ __forceinline__ void rowsum_add(const float (&v)[16], float* dsum, float* dabs, size_t r0, int nvalid) {
  const int lane = threadIdx.x & 31;
  float s[16], a[16];
#pragma unroll
  for (int c = 0; c < 16; ++c) {
    s[c] = v[c];
    a[c] = fabsf(v[c]);
  }
#pragma unroll
  for (int w = 8; w >= 1; w >>= 1) {
    const bool up = (lane & (2 * w)) != 0;
#pragma unroll
    for (int k = 0; k < w; ++k) {
      const float ss = up ? s[k] : s[k + w], sa = up ? a[k] : a[k + w];
      const float ks = up ? s[k + w] : s[k], ka = up ? a[k + w] : a[k];
      s[k] = ks + __shfl_xor_sync(0xffffffffu, ss, 2 * w);
      a[k] = ka + __shfl_xor_sync(0xffffffffu, sa, 2 * w);
    }
  }
  s[0] += __shfl_xor_sync(0xffffffffu, s[0], 1);
  a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
  const int c = (lane >> 1) & 15;
  if ((lane & 1) == 0 && c < nvalid) {
    if (dsum) atomicAdd(dsum + r0 + c, s[0]);
    if (dabs) atomicAdd(dabs + r0 + c, a[0]);
  }
}

// MMA warp of k_bwd_dkdv: the products of the query tile in stage s (landed) into score buffer b.
__device__ __forceinline__ void kv_issue_s(const Params& p, const uint8_t* st, int b, uint32_t cKa, uint32_t cSG,
                                           int qtile) {
  const int D = p.d;
  const uint32_t cS = cSG + 128 * b;
  if (p.x3) {
    mma_tmem_smem(cS, cKa + D, st, BT, D, false);
    mma_tmem_smem(cS, cKa, st + qtile, BT, D, true);
    mma_tmem_smem(cS, cKa, st, BT, D, true);
  } else {
    mma_tmem_smem(cS, cKa, st, BT, D, false);
  }
}
__device__ __forceinline__ void kv_issue_g(const Params& p, const uint8_t* st, int b, uint32_t cVa, uint32_t cSG,
                                           int qtile, int odO) {
  const int D = p.d;
  const uint32_t cG = cSG + 128 * b + 64;
  if (p.x3) {
    mma_tmem_smem(cG, cVa + D, st + odO, BT, D, false);
    mma_tmem_smem(cG, cVa, st + odO + qtile, BT, D, true);
    mma_tmem_smem(cG, cVa, st + odO, BT, D, true);
  } else {
    mma_tmem_smem(cG, cVa, st + odO, BT, D, false);
  }
}
// Both (S^T_b = K Q^T and, with V, g^T_b = V dO^T) once the tile in stage stg has landed.
__device__ __forceinline__ bool kv_issue_sg(const Params& p, RingPos stg, int b, uint64_t* bar_full,
                                            uint64_t* bar_sfull, const uint8_t* st0, uint32_t cKa, uint32_t cVa,
                                            uint32_t cSG, int qtile, bool needV, int odO) {
  if (!mbar_wait_warp(&bar_full[stg.i], stg.ph, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA)) return false;
  tc_fence_after();
  const uint8_t* st = st0 + stg.i * p.sm_stage_bytes;
  kv_issue_s(p, st, b, cKa, cSG, qtile);
  if (needV) kv_issue_g(p, st, b, cVa, cSG, qtile, odO);
  mma_commit(&bar_sfull[b]);
  return true;
}

// Producer warp of k_bwd_dkdv: TMA-stores the dV / dK tiles of its k-th item, which the
// compute warps staged at `tile` (dV, then dK), and returns once they have been read out.
template <class Order>
__device__ __forceinline__ bool store_staged_dkdv(const Maps& maps, const Params& p, const Order& sch, uint64_t* bar_ostg, int k,
                                                  const uint8_t* tile, bool doDV, bool doDK) {
  if (!mbar_wait_warp(bar_ostg, k & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_SYNC)) return false;
  const int item = sched_item(sch, k), kb = item / p.BH, bh = item % p.BH;
  if (doDV) store_rows_tile_boxed(tile, &maps.dv, p.d, 64, kb * 128, bh, false);
  if (doDK) store_rows_tile_boxed(tile + 128 * p.d * 4, &maps.dk, p.d, 64, kb * 128, bh, false);
  tma_store_wait_read();
  return true;
}

// ---------------------------------------------------------------------------
// k_bwd_dkdv.  TMEM: K [0, dp), V [dp, 2dp) (dK launches),
// then per buffer b: S^T_b (64 columns) and g^T_b (64 columns) from `base`,
// dV, dK.  P^T overwrites S^T_b and dS^T overwrites g^T_b (3xTF32: the single
// product's hi part goes to S^T_b, its lo part to g^T_b).
// smem stage: the tiles the launch reads of Q | dO | Q^T | dO^T (hi[, lo]): Q, and dO and Q^T
// for dK, dO^T for dV; the 64 RowRecs of the tile, and (MinMax) their grid pair tables;
// FWM's shared table at sm_table.  (With all four in every stage a one-product launch at
// d = 128 or under 3xTF32 had one stage and nothing overlapped.)
// dK alone (d = 128, 3xTF32) runs the product pipeline of kint_pair.cuh instead of the stage
// ring: K in TMEM, V as an operand in smem, Q, dO and Q^T in rings of their own.
// What bounds it: the issue of the products by one warp, then the shared-memory loads of the
// row records.
// Measured on GB300 against eight compute warps and stages of all four tiles: B=4 H=16 T=2048
// d=128 FWM Weight-STE dV 340 -> 170 us, dK 403 -> 231; H=16 T=16384 d=128 MinMax K=16 LERP
// 5097 -> 2104, 5878 -> 2984; 3xTF32 B=8 H=12 T=1024 168 -> 93, 203 -> 127; MinMax B=4 H=12
// T=1024 d=64 (both products) 73.6 -> 71.6, and 63.4 with d, the precision and the staging path fixed
// at compile time for the launch of both products.  (dK in the stage ring with 32-query tiles: 313,
// 3785 and 170.)
// ---------------------------------------------------------------------------
template <int CAL, int REC, bool FULLG, bool PROJ, bool RS, int SEL>
__global__ void __launch_bounds__(NTHR_KV, 1) k_bwd_dkdv(const __grid_constant__ Maps maps, const Params p,
                                                         const __grid_constant__ ItemOrder<SEL == DKV_DK> sch) {
  uint8_t* sm = smem_base();
  if (p.gate != nullptr) {
    // launched on one side of a device-side decision: when the single-pass backward ran
    // instead, leave before any set-up (no barrier, no tensor memory)
    pdl_wait();
    if (gated_off(p)) return;
  }
  // both products: TF32 at d = 64; one: d = 128 or 3xTF32
  constexpr bool STAGED = SEL == DKV_BOTH;  // K, V rows and the outputs pass through smem by TMA
  const bool x3 = !STAGED && p.x3;
  const int D = STAGED ? 64 : p.d, Kq = p.Kint, parts = x3 ? 2 : 1, NS = p.nstage, nbuf = p.nbuf;
  constexpr bool doDV = SEL != DKV_DK, doDK = SEL != DKV_DV, needV = doDK;
  constexpr bool PAIR = SEL == DKV_DK;  // the product pipeline of kint_pair.cuh
  const int qtile = BT * D * 4;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm + p.sm_bars);
  uint64_t* bar_full = bars;
  uint64_t* bar_empty = bars + NS;
  uint64_t* bar_sfull = bars + 2 * NS;
  uint64_t* bar_pready = bars + 2 * NS + 2;
  uint64_t* bar_done = bars + 2 * NS + 4;
  uint64_t* bar_ops = bars + 2 * NS + 5;  // K / V rows stored in TMEM by every compute warp
  uint64_t* bar_stg = bars + 2 * NS + 6;   // K / V tiles staged in smem by TMA
  uint64_t* bar_ostg = bars + 2 * NS + 7;  // an item's dV / dK tiles staged in the K / V area
  // a stage's transposed tiles (Q^T, dO^T) complete on their own barrier, so the products
  // S^T, g^T wait only for the first half of the stage's bytes
  uint64_t* bar_fullT = bars + 2 * NS + 8;  // [NS]
  // the first half of a stage (Q, dO, row records) is free once the compute warps are done
  // with the tile (S^T, g^T completed before they started); the transposed half once the
  // products dV, dK that read it complete (bar_empty)
  uint64_t* bar_emptyA = bars + 3 * NS + 8;  // [NS]
  uint64_t* bar_drain = bars + 4 * NS + 8;   // the MMA warp's clean-up commit
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + (PAIR ? PAIR_NBARS : 4 * NS + 9));
  const PairBars B = pair_bars(bars);
  const int tid = threadIdx.x, warp = warp_id_uniform();
  const int dp = D * parts;
  const int cK = 0, cV = dp, base = PAIR ? 128 : needV ? 2 * dp : dp;
  const int cdV = base + 128 * (PAIR ? 2 : nbuf), cdK = cdV + (doDV ? D : 0);
  // 3xTF32 (one product per launch): the two cross terms accumulate apart from hi x hi.
  // The tensor core rounds each accumulation step toward zero, so a dK / dV row summed
  // over a whole causal column (up to T / 8 x 3 steps) drifts by about one unit in the
  // last place per step; keeping the cross terms out of the main accumulator cuts its
  // steps by three, and the two sums meet in fp32 in the epilogue.
  const int cdC = cdK + (doDK ? D : 0);
  const int nqt = (p.T + BT - 1) / BT;
  const int oQ = 0, odO = parts * qtile, oQT = (needV ? 2 : 1) * parts * qtile,
            odOT = oQT + (doDK ? parts * qtile : 0);
  const int oRec = odOT + (doDV ? parts * qtile : 0), oTab = oRec + BT * 64;
  const uint32_t tstride = (uint32_t)p.Kp * 8u;
  constexpr int W = 16;            // query columns per thread per tile

  if (PAIR && tid == 0) {
    pair_init(B, NCOMP_KV / 32);
    fence_mbar_init();
  }
  if (!PAIR && tid == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(&bar_full[s], 1);
      mbar_init(&bar_fullT[s], 1);
      mbar_init(&bar_empty[s], 1);
      mbar_init(&bar_emptyA[s], NCOMP_KV / 32);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&bar_sfull[b], 1);
      mbar_init(&bar_pready[b], NCOMP_KV / 32);
    }
    mbar_init(bar_done, 1);
    mbar_init(bar_ops, NCOMP_KV / 32);
    mbar_init(bar_stg, 1);
    mbar_init(bar_ostg, NCOMP_KV / 32);
    mbar_init(bar_drain, 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(tslot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_trigger();
  pdl_wait();  // everything below may read what the previous kernel wrote
  // All 512 columns are allocated, so the allocation starts at lane 0, column 0; a
  // compile-time base keeps the TMEM addresses of the issue paths in uniform registers.
  if (threadIdx.x == 0 && *tslot != 0u) dev_flag(p.status, DEV_ERR_BOUNDS);
  constexpr uint32_t tmem = 0;

  // Work items are (128-key block kb, head) pairs, longest first (kb = 0 meets every
  // query tile); a CTA takes the items sched_item(sch, 0), sched_item(sch, 1), ...  Tile counters
  // (stage ring, score buffers) run on across items.
  if (warp >= NCOMP_KV / 32) {
  setmaxnreg_dec<REG_AUX_KV>();
  if constexpr (PAIR) {
    auto get = [&](int n) {
      const int item = sched_item(sch, n), kb = item / p.BH;
      return PairItem{item % p.BH, kb * 128, kb * 128, nqt - kb * 128 / BT, item < p.nitems};
    };
    const PairMaps m{&maps.k, &maps.k_lo, &maps.v, &maps.v_lo, &maps.q, &maps.q_lo, &maps.dout, &maps.dout_lo,
                     &maps.qt, &maps.qt_lo};
    if (warp == PRODUCER_WARP_KV) {
      pair_producer<true>(p, m, B, sm, get, [&](const PairItem& it, int q0, uint8_t* dst, uint64_t* bar) {
        const int nrows = min(BT, p.T - q0);
        const size_t r0 = (size_t)it.bh * p.T + q0;
        mbar_arrive_expect_tx(bar, nrows * 64 + (CAL == CAL_MINMAX ? nrows * (int)tstride : 0));
        bulk_load(dst, reinterpret_cast<const RowRec*>(p.rec) + r0, nrows * 64, bar);
        if (CAL == CAL_MINMAX) bulk_load(dst + BT * 64, p.rtab + r0 * p.Kp * 2, nrows * tstride, bar);
      });
    } else if (warp == PRODUCER_WARP_KV + 1) {
      pair_producer_t(p, m, B, sm, get);
    } else if (warp == MMA_WARP_KV) {
      pair_mma_sg(p, B, sm, get);
    } else {
      pair_mma_acc(p, B, sm, get, [&](uint32_t cS, uint32_t cG, const uint8_t* qt, bool first) {
        if (x3) {
          mma_tmem_smem(cdK, cS, qt, D, BT, !first);          // hi x hi
          mma_tmem_smem(cdC, cS, qt + qtile, D, BT, !first);  // hi x lo
          mma_tmem_smem(cdC, cG, qt, D, BT, true);            // lo x hi
        } else {
          mma_tmem_smem(cdK, cG, qt, D, BT, !first);
        }
      });
    }
  } else if (warp == PRODUCER_WARP_KV) {
    int gt = 0, n = 0;
    RingPos ld;  // stage of the next tile loaded
    RingPos nf, nT;  // ring positions after the last first-half and transposed-half loads issued
    int cf = 0, cT = 0;  // how many of each were issued
    bool ok = true;
    // K / V of this CTA's k-th item into the staging area (TF32 at d = 64)
    int staged = 0;  // staging loads issued
    auto stage_ops = [&](int k) {
      const int it_ = sched_item(sch, k), kb_ = it_ / p.BH, bh_ = it_ % p.BH;
      mbar_arrive_expect_tx(bar_stg, (needV ? 2 : 1) * 128 * D * 4);
      load_rows_tile_boxed(sm + p.sm_a, &maps.k, bar_stg, D, 128, BT, 0, kb_ * 128, bh_);
      if (needV) load_rows_tile_boxed(sm + p.sm_a + 128 * D * 4, &maps.v, bar_stg, D, 128, BT, 0, kb_ * 128, bh_);
      staged = k + 1;
    };
    if (STAGED && sched_item(sch, 0) < p.nitems) stage_ops(0);
    for (int item = sched_item(sch, n); item < p.nitems && ok; item = sched_item(sch, ++n)) {
      const int kb = item / p.BH, bh = item % p.BH;
      const int qt0 = (kb * 128) / BT, nit = nqt - qt0;
      for (int it = 0; it < nit; ++it, ++gt, ld.next(NS)) {
        const int s = ld.i, q0 = (qt0 + it) * BT;
        if (gt >= NS && !mbar_wait_warp(&bar_emptyA[s], ld.ph ^ 1u, p.wait_ns, p.status, DEV_ERR_TIMEOUT_SYNC)) {
          ok = false;
          break;
        }
        uint8_t* dst = sm + p.sm_stage0 + s * p.sm_stage_bytes;
        // first the operands of S^T, g^T and the row records, then the transposed tiles
        uint64_t* b = &bar_full[s];
        const int nrows = min(BT, p.T - q0);
        uint32_t bytes = (1 + (needV ? 1 : 0)) * parts * qtile + nrows * 64;
        if (CAL == CAL_MINMAX) bytes += nrows * tstride;
        mbar_arrive_expect_tx(b, bytes);
        load_rows_tile(dst + oQ, &maps.q, b, D, BT, 0, q0, bh);
        if (x3) load_rows_tile(dst + oQ + qtile, &maps.q_lo, b, D, BT, 0, q0, bh);
        if (needV) {
          load_rows_tile(dst + odO, &maps.dout, b, D, BT, 0, q0, bh);
          if (x3) load_rows_tile(dst + odO + qtile, &maps.dout_lo, b, D, BT, 0, q0, bh);
        }
        const size_t r0 = (size_t)bh * p.T + q0;
        bulk_load(dst + oRec, reinterpret_cast<const RowRec*>(p.rec) + r0, nrows * 64, b);
        if (CAL == CAL_MINMAX) bulk_load(dst + oTab, p.rtab + r0 * p.Kp * 2, nrows * tstride, b);
        nf.next(NS);
        ++cf;
        if (gt >= NS && !mbar_wait_warp(&bar_empty[s], ld.ph ^ 1u, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA)) {
          ok = false;
          break;
        }
        uint64_t* bt = &bar_fullT[s];
        mbar_arrive_expect_tx(bt, ((doDK ? 1 : 0) + (doDV ? 1 : 0)) * parts * qtile);
        if (doDK) {
          load_rows_tile(dst + oQT, &maps.qt, bt, BT, D, q0, 0, bh);
          if (x3) load_rows_tile(dst + oQT + qtile, &maps.qt_lo, bt, BT, D, q0, 0, bh);
        }
        if (doDV) {
          load_rows_tile(dst + odOT, &maps.dot, bt, BT, D, q0, 0, bh);
          if (x3) load_rows_tile(dst + odOT + qtile, &maps.dot_lo, bt, BT, D, q0, 0, bh);
        }
        nT.next(NS);
        ++cT;
        // The next item's K / V, as soon as the stage ring holds this item's first tiles: it needs
        // this item's K / V copied out into TMEM and the previous item's dV / dK tiles, staged in
        // the same area since, stored; both happen at the end of the previous item, so the load
        // has this whole item to land.
        if (STAGED && it == min(nit, NS) - 1 && sched_item(sch, n + 1) < p.nitems) {
          if (!mbar_wait_warp(bar_ops, n & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_SYNC) ||
              (n >= 1 && !store_staged_dkdv(maps, p, sch, bar_ostg, n - 1, sm + p.sm_a, doDV, doDK))) {
            ok = false;
            break;
          }
          stage_ops(n + 1);
        }
      }
    }
    // the last-but-one item's tiles (the last item's are stored by the compute warps)
    if (STAGED && ok && n >= 2) store_staged_dkdv(maps, p, sch, bar_ostg, n - 2, sm + p.sm_a, doDV, doDK);
    tma_store_wait_all();
    // clean-up: the last tiles issued have landed
    drain_ring(bar_full, nf, cf, NS, p.wait_ns, p.status);
    drain_ring(bar_fullT, nT, cT, NS, p.wait_ns, p.status);
    if (staged > 0) mbar_wait_warp(bar_stg, (staged - 1) & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA);
  } else if (warp == MMA_WARP_KV) {
    const uint8_t* st0 = sm + p.sm_stage0;
    const uint32_t cKa = tmem + cK, cVa = tmem + cV, cSG = tmem + base;
    int n = 0;
    RingPos is, ib, cs, cb;  // stage / buffer of the next S^T, g^T product and of the tile being finished
    bool ok = true;
    for (int item = sched_item(sch, n); item < p.nitems && ok; item = sched_item(sch, ++n)) {
      const int kb = item / p.BH, nit = nqt - (kb * 128) / BT;
      // K / V of the item in TMEM (the compute warps copy them only after the previous
      // item's last S, g were read)
      ok = mbar_wait_warp(bar_ops, n & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_SYNC);
      if (ok) tc_fence_after();
      ok = ok && kv_issue_sg(p, is, ib.i, bar_full, bar_sfull, st0, cKa, cVa, cSG, qtile, needV, odO);
      is.next(NS);
      ib.next(nbuf);
      for (int it = 0; it < nit && ok; ++it, cs.next(NS), cb.next(nbuf)) {
        const int b = cb.i, s = cs.i;
        if (nbuf == 2 && it + 1 < nit) {
          ok = kv_issue_sg(p, is, ib.i, bar_full, bar_sfull, st0, cKa, cVa, cSG, qtile, needV, odO);
          is.next(NS);
          ib.next(nbuf);
        }
        if (!ok) break;
        if (!mbar_wait_warp(&bar_pready[b], cb.ph, p.wait_ns, p.status, DEV_ERR_TIMEOUT_SYNC) ||
            !mbar_wait_warp(&bar_fullT[s], cs.ph, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint8_t* st = sm + p.sm_stage0 + s * p.sm_stage_bytes;
        const uint32_t cS = tmem + base + 128 * b, cG = cS + 64;
        const bool acc = it > 0;
        if (x3) {
          const uint32_t cacc = tmem + (doDV ? cdV : cdK);
          const uint8_t* bt = st + (doDV ? odOT : oQT);
          mma_tmem_smem(cacc, cS, bt, D, BT, acc);                   // hi x hi
          mma_tmem_smem(tmem + cdC, cS, bt + qtile, D, BT, acc);     // hi x lo
          mma_tmem_smem(tmem + cdC, cG, bt, D, BT, true);            // lo x hi
        } else {
          if (doDV) mma_tmem_smem(tmem + cdV, cS, st + odOT, D, BT, acc);
          if (doDK) mma_tmem_smem(tmem + cdK, cG, st + oQT, D, BT, acc);
        }
        mma_commit(&bar_empty[s]);
        if (nbuf == 1 && it + 1 < nit) {
          ok = kv_issue_sg(p, is, ib.i, bar_full, bar_sfull, st0, cKa, cVa, cSG, qtile, needV, odO);
          is.next(NS);
          ib.next(nbuf);
        }
      }
      mma_commit(bar_done);
    }
    drain_mma(bar_drain, p.wait_ns, p.status);  // clean-up: no product still writes TMEM
  }
  } else {
    setmaxnreg_inc<REG_COMP_KV>();
    const int row = tid & 127, cg = tid >> 7;
    // K / V rows of the n-th item into TMEM (each thread a share of its key's columns: with V two
    // column groups take K and two take V), handed to the MMA warp through bar_ops: TF32 at
    // d = 64 from the tiles the producer staged in smem, otherwise from global rows.  The
    // next item's rows go in as soon as the current item's last S^T, g^T have been read, so
    // its first products run under the current item's epilogue.
    auto ops_to_tmem = [&](int n) {
      if constexpr (PAIR) {
        pair_ops_to_tmem(p, B, sm, n, row, cg * (D / NCG_KV), D / NCG_KV);
        return;
      }
      const int item = sched_item(sch, n), kb = item / p.BH, bh = item % p.BH, j = kb * 128 + row;
      const bool isV = needV && cg >= 2;
      const int nc = needV ? D / 2 : D / NCG_KV, c0 = (needV ? cg & 1 : cg) * nc;
      const bool ok = !STAGED || mbar_wait(bar_stg, n & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA);
      if (ok) {
        const int lim = j < p.T ? (bh + 1) * p.T : 0;
#pragma unroll 1
        for (int c = c0; c < c0 + nc; c += 16) {
          if (STAGED)
            staged16_to_tmem(tmem, isV ? cV : cK, sm + p.sm_a + (isV ? 128 * D * 4 : 0), row, c);
          else
            row_to_tmem_part<16>(tmem, isV ? cV : cK, isV ? p.V : p.K, bh * p.T + j, lim, D, c, x3);
        }
      }
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if ((tid & 31) == 0) mbar_arrive(bar_ops);
    };
    if (sched_item(sch, 0) < p.nitems) ops_to_tmem(0);
    // FWM Nearest: the half-bin table (entry q at sm_table + 8 (q + 2)) and the doubled
    // position; FWM LERP: the pair table, entry r at sm_table + 8 r (0x4B000000 * 8 =
    // 0x58000000 mod 2^32)
    constexpr bool half = fwm_like(CAL) && REC == REC_NEAREST;
    if constexpr (fwm_like(CAL)) {
      if (half && tid < 2 * Kq + 1 + kHalfTail)
        *reinterpret_cast<float2*>(sm + p.sm_table + tid * 8) = fwm_half_entry(p, tid - kHalfTail);
      if (!half && tid < Kq)
        *reinterpret_cast<float2*>(sm + p.sm_table + tid * 8) = make_float2(p.fwm_e[tid], p.fwm_e[tid + 1]);
    }
    const float Kf = (float)(half ? 2 * Kq : Kq);
    const uint32_t fwtab = smem_u32(sm + p.sm_table) + (half ? 8u * kHalfTail : 0u) - 0x58000000u;
    group_sync(BAR_COMPUTE, NCOMP_KV);  // the FWM table
    bool failed = false;
    int n = 0;
    RingPos cs, cb;  // stage (dK alone: slot of the record ring) and score buffer of the current tile
    const int ncs = PAIR ? 2 : NS, ncb = PAIR ? 2 : nbuf;
    for (int item = sched_item(sch, n); item < p.nitems && !failed; item = sched_item(sch, ++n)) {
      const int kb = item / p.BH, bh = item % p.BH;
      const int qt0 = (kb * 128) / BT, nit = nqt - qt0;
      const int j = kb * 128 + row;
      // the tie flags are per 64 query rows
      constexpr bool ties = doDK && FULLG && CAL != CAL_SOFTMAX;
      const int* tflags = p.tileflags + (size_t)bh * p.nqt + qt0 * BT / 64;
      int tie_next = ties ? __ldg(tflags) : 0;
      for (int it = 0; it < nit; ++it, cs.next(ncs), cb.next(ncb)) {
        // the next tile's tie flag, loaded one tile ahead
        const int tie_here = tie_next;
        if (ties && it + 1 < nit) tie_next = __ldg(tflags + (it + 1) * BT / 64);
        const int b = cb.i, s = cs.i;
        const int q0 = (qt0 + it) * BT;
        const bool ok1 = mbar_wait(PAIR ? &B.sfull[b] : &bar_sfull[b], cb.ph, p.wait_ns, p.status, DEV_ERR_TIMEOUT_MMA);
        // the stage's row records arrived with its tiles (bar_full), before the products were issued
        const bool ok2 = ok1 && mbar_wait(PAIR ? &B.fullR[s] : &bar_full[s], cs.ph, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA);
        if (!ok2) {
          failed = true;
          break;
        }
        tc_fence_after();
        const uint8_t* st = PAIR ? sm + p.sm_rec + s * p.rec_bytes : sm + p.sm_stage0 + s * p.sm_stage_bytes + oRec;
        const int c0 = cg * W, i0h = q0 + c0;
        const uint32_t recs = smem_u32(st) + c0 * 64;
        const uint32_t tabs = smem_u32(st + BT * 64) + c0 * tstride - 0x58000000u;
        const int cS = base + 128 * b + c0, cG = cS + 64;
        float sv[W], gv[W], pa[W], da[W];
        tmem_ldw<W>(lane_addr(tmem, cS), sv);
        if (needV) {
          tmem_ldw<W>(lane_addr(tmem, cG), gv);
        } else {
#pragma unroll
          for (int q = 0; q < W; ++q) gv[q] = 0.f;
        }
        tmem_ld_wait();
        // this warp's keys against its queries: all pairs masked, some, or none
        const int j0w = kb * 128 + (warp & 3) * 32;
        if (i0h + W <= j0w) {
#pragma unroll
          for (int q = 0; q < W; ++q) pa[q] = da[q] = 0.f;
        } else {
          const bool masked = i0h < j0w + 31 || i0h + W > p.T;
          if (doDK && FULLG && CAL != CAL_SOFTMAX && tie_here)
            kv_chunk<CAL, REC, FULLG, PROJ, true, true, doDV, doDK, W>(sv, gv, pa, da, j, i0h, p.T, recs, tabs, fwtab, tstride, Kf,
                                                     p.fwm_inv_h, p.scale, p.fwm_hl, p.fwm_b0l);
          else if (masked)
            kv_chunk<CAL, REC, FULLG, PROJ, true, false, doDV, doDK, W>(sv, gv, pa, da, j, i0h, p.T, recs, tabs, fwtab, tstride,
                                                      Kf, p.fwm_inv_h, p.scale, p.fwm_hl, p.fwm_b0l);
          else
            kv_chunk<CAL, REC, FULLG, PROJ, false, false, doDV, doDK, W>(sv, gv, pa, da, j, i0h, p.T, recs, tabs, fwtab, tstride,
                                                       Kf, p.fwm_inv_h, p.scale, p.fwm_hl, p.fwm_b0l);
          // optional side outputs: per-query-row sums of dS and |dS| over this warp's 32 keys
          if constexpr (RS) {
            if (doDK) rowsum_add(da, p.dsum_out, p.dabs_out, (size_t)bh * p.T + i0h, min(W, p.T - i0h));
          }
        }
        if (x3) {
#pragma unroll
          for (int q = 0; q < W; ++q) {
            const float x = doDV ? pa[q] : da[q];
            const float hh = tf32_rna(x);
            pa[q] = hh;
            da[q] = __fsub_rn(x, hh);
          }
          tmem_stw<W>(lane_addr(tmem, cS), pa);
          tmem_stw<W>(lane_addr(tmem, cG), da);
        } else {
          if (doDV) tmem_stw<W>(lane_addr(tmem, cS), pa);
          if (doDK) tmem_stw<W>(lane_addr(tmem, cG), da);
        }
        __syncwarp();
        if ((tid & 31) == 0) mbar_arrive(PAIR ? &B.emptyR[s] : &bar_emptyA[s]);  // the stage's records are read
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if ((tid & 31) == 0) mbar_arrive(PAIR ? &B.pready[b] : &bar_pready[b]);
      }
      // the next item's K / V (this item's S^T, g^T have all been read: the last tile's were)
      if (!failed && sched_item(sch, n + 1) < p.nitems) ops_to_tmem(n + 1);
      const bool dok = !failed && mbar_wait(PAIR ? B.done : bar_done, n & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_MMA);
      failed = group_any(BAR_COMPUTE, NCOMP_KV, !dok);
      if (!failed) {
        tc_fence_after();
        // dV, dK rows into swizzled tiles for TMA stores: in the K / V staging area (free now
        // that the next item's K / V are in TMEM; the producer stores them before it stages
        // the item after next), or, for the last item, in the idle stage ring (stored here).
        // Without the staging area (3xTF32, d = 128, one-product launches) straight to
        // global memory.
        const bool last = sched_item(sch, n + 1) >= p.nitems;
        uint8_t* stg = last ? sm + p.sm_stage0 : sm + p.sm_a;
        for (int pass = 0; pass < 2; ++pass) {
          if (pass == 0 ? !doDV : !doDK) continue;
          const int col = pass == 0 ? cdV : cdK;
          const float mul = pass == 0 ? 1.0f : p.scale;
          float* out = (pass == 0 ? p.dV : p.dK) + ((size_t)bh * p.T + j) * D;
          for (int c = cg * (D / NCG_KV); c < (cg + 1) * (D / NCG_KV); c += 16) {
            float v[16];
            tmem_ld16(lane_addr(tmem, col + c), v);
            if (x3) {
              float w[16];
              tmem_ld16(lane_addr(tmem, cdC + c), w);
              tmem_ld_wait();
#pragma unroll
              for (int q = 0; q < 16; ++q) v[q] += w[q];
            }
            tmem_ld_wait();
#pragma unroll
            for (int q = 0; q < 16; ++q) v[q] *= mul;
            if (STAGED) {
              row16_to_staged(stg + pass * 128 * D * 4, row, c, v);
            } else if (j < p.T) {
              float4* dst = reinterpret_cast<float4*>(out + c);
#pragma unroll
              for (int q = 0; q < 4; ++q) dst[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            }
          }
        }
        if (STAGED) {
          fence_async_smem();
          if (last) {
            group_sync(BAR_COMPUTE, NCOMP_KV);
            if (warp == 0 && doDV) store_rows_tile_boxed(stg, &maps.dv, D, 64, kb * 128, bh, false);
            if (warp == 1 && doDK) store_rows_tile_boxed(stg + 128 * D * 4, &maps.dk, D, 64, kb * 128, bh, false);
          } else {
            __syncwarp();
            if ((tid & 31) == 0) mbar_arrive(bar_ostg);
          }
        }
      }
    }
    if (warp < 2) tma_store_wait_all();
    tc_fence_before();
  }
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, 512);
}

// Every backward mode of one calibration and reconstruction; softmax ignores the mode, and a dV
// launch does not depend on it.
template <int CAL, int REC, bool RS, int SEL>
cudaError_t launch_dkdv_modes(dim3 grid, const Maps& maps, const Params& p, int smem_bytes, cudaStream_t s,
                              const ItemOrder<SEL == DKV_DK>& sch) {
  if constexpr (CAL == CAL_SOFTMAX || SEL == DKV_DV) {
    return launch3(k_bwd_dkdv<CAL, REC, false, false, RS, SEL>, grid, maps, p, smem_bytes, s, sch, NTHR_KV);
  } else {
    const bool proj = p.grad == GRAD_DETACH_PROJ, full = p.grad != GRAD_DETACH && !proj;
    return full ? launch3(k_bwd_dkdv<CAL, REC, true, false, RS, SEL>, grid, maps, p, smem_bytes, s, sch, NTHR_KV)
           : proj ? launch3(k_bwd_dkdv<CAL, REC, false, true, RS, SEL>, grid, maps, p, smem_bytes, s, sch, NTHR_KV)
                  : launch3(k_bwd_dkdv<CAL, REC, false, false, RS, SEL>, grid, maps, p, smem_bytes, s, sch, NTHR_KV);
  }
}

// The dK/dV launch of p's configuration.  RS: the instantiation that also accumulates the
// per-row sums of dS and |dS| (p.dsum_out, p.dabs_out); SEL: its products (DkvSel).
template <bool RS, int SEL>
cudaError_t launch_bwd_dkdv_t(const Maps& maps, const Params& p, int smem_bytes, cudaStream_t s, const ItemOrder<SEL == DKV_DK>& sch) {
  const dim3 grid((unsigned)p.ngrid);
  const bool near = p.recon == REC_NEAREST;
  switch (p.calib) {
    case CAL_SOFTMAX: return launch_dkdv_modes<CAL_SOFTMAX, REC_LERP, RS, SEL>(grid, maps, p, smem_bytes, s, sch);
    case CAL_EXP8: return launch_dkdv_modes<CAL_EXP8, REC_LERP, RS, SEL>(grid, maps, p, smem_bytes, s, sch);
    case CAL_EXPB: return launch_dkdv_modes<CAL_EXPB, REC_LERP, RS, SEL>(grid, maps, p, smem_bytes, s, sch);
    case CAL_MINMAX:
      return near ? launch_dkdv_modes<CAL_MINMAX, REC_NEAREST, RS, SEL>(grid, maps, p, smem_bytes, s, sch)
                  : launch_dkdv_modes<CAL_MINMAX, REC_LERP, RS, SEL>(grid, maps, p, smem_bytes, s, sch);
    case CAL_FWMR:
      return near ? launch_dkdv_modes<CAL_FWMR, REC_NEAREST, RS, SEL>(grid, maps, p, smem_bytes, s, sch)
                  : launch_dkdv_modes<CAL_FWMR, REC_LERP, RS, SEL>(grid, maps, p, smem_bytes, s, sch);
    default:
      return near ? launch_dkdv_modes<CAL_FWM, REC_NEAREST, RS, SEL>(grid, maps, p, smem_bytes, s, sch)
                  : launch_dkdv_modes<CAL_FWM, REC_LERP, RS, SEL>(grid, maps, p, smem_bytes, s, sch);
  }
}
extern template cudaError_t launch_bwd_dkdv_t<false, DKV_BOTH>(const Maps&, const Params&, int, cudaStream_t, const SnakeOrder&);
extern template cudaError_t launch_bwd_dkdv_t<false, DKV_DV>(const Maps&, const Params&, int, cudaStream_t, const SnakeOrder&);
extern template cudaError_t launch_bwd_dkdv_t<false, DKV_DK>(const Maps&, const Params&, int, cudaStream_t, const Sched&);
extern template cudaError_t launch_bwd_dkdv_t<true, DKV_BOTH>(const Maps&, const Params&, int, cudaStream_t, const SnakeOrder&);
extern template cudaError_t launch_bwd_dkdv_t<true, DKV_DK>(const Maps&, const Params&, int, cudaStream_t, const Sched&);

}  // namespace kint
