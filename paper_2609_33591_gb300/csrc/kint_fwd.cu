// Forward of K-interval attention on sm_103a: operand preparation and pass 1 (row
// extrema); pass 2 (grid reconstruction, normalization, P V) is in kint_fwd_main.cuh.
//
// Two passes are needed because the grid of a row depends on its final
// extrema (Sec. 3: MinMax spans [m, M]; FWM is anchored at M), so partial
// results cannot be rescaled online the way a softmax running maximum can.
#include <cfloat>
#include "kint_dev.cuh"
#include "kint_launch.h"

namespace kint {

// Row record of the single-pass backward for row rw (position t of head bh) from its row
// max M, forward normalizer Wf, the W* of gamma Ws, tie count nm and <g>_{P*} = dg;
// returns whether this row's tied keys overflow the tie list.
__device__ __forceinline__ bool prep_row_record(const RecJob& R, size_t rw, int bh, int t, float M, float Wf, float Ws,
                                                int nm, float dg) {
  float4 f;
  f.z = R.softmax ? 1.0f : 1.0f / Ws;  // gamma = g * f.z + f.w
  f.w = R.softmax ? -dg : -dg * f.z;
  f.y = 1.0f / Wf;
  if (R.c0_kind == 0) {
    f.x = -M * kLog2e;
  } else if (R.c0_kind == 1) {
    const float c0 = __fmul_rn(__fsub_rn(R.tau, M), R.inv_h);
    f.x = R.half ? 2.0f * c0 : c0;
  } else {
    f.x = -M;
  }
  R.frec[rw] = f;
  R.rsum[rw] = 0.0f;
  // the calibration-sum outputs stay 0 in the modes whose extremum pass does not write them
  if (R.cM_out) R.cM_out[rw] = 0.0f;
  if (R.cm_out) R.cm_out[rw] = 0.0f;
  if (nm <= 1) return false;
  // a row with tied maxima: its 64-row query tile takes the single pass's tie search
  R.tileflags[(size_t)bh * R.nqt + t / 64] = 1;
  return atomicAdd(R.tie_total, nm) + nm > R.tie_cap;
}

// ---------------------------------------------------------------------------
// Operand preparation (HBM-bound).  tcgen05.mma kind::tf32 reads both operands
// K-major, so every second-stage product (P V, dS K, P^T dO, dS^T Q) reads a
// transposed copy X^T [BH][d][Tp].  3xTF32 also needs tf32 hi/lo splits.  A job
// with Y also forms the row dot products dot[t] = X_t . Y_t (the backward's
// <g>_{P*} = dO_i . O*_i, App. B) from the rows it already holds.
// One launch serves up to four tensors.  The work units (job, head, 32-row block)
// are spread over a grid of sixteen CTAs per SM that loop over them, so the launch
// has no partial last wave; a unit moves all d columns in 64-column steps through a
// padded 32 x 65 shared tile (128 threads, four float4 loads and stores each).
// ---------------------------------------------------------------------------
template <bool SPLIT>
__global__ void __launch_bounds__(128) k_prep(const __grid_constant__ PrepJobs jobs, int T, int Tp, int d,
                                              int BH) {
  __shared__ float hs[32][65];
  __shared__ float ls[SPLIT ? 32 : 1][65];
  __shared__ float dots[32];
  const int tid = threadIdx.x;
  const int r = tid >> 4, c4 = tid & 15;  // load phase: rows r + 8 q, columns 4 c4 .. 4 c4 + 3
  const int k = tid >> 3, tq = tid & 7;   // store phase: output rows k + 16 q, keys 4 tq .. 4 tq + 3
  const int ntb = Tp / 32, per_job = BH * ntb, units = jobs.n * per_job;
  pdl_wait();
  for (int u = blockIdx.x; u < units; u += gridDim.x) {
    const PrepJob& J = jobs.j[u / per_job];
    const int bh = (u % per_job) / ntb, t0 = (u % ntb) * 32;
    const size_t nat = (size_t)bh * T * d, tr = (size_t)bh * d * Tp;
    const bool dotj = J.Y != nullptr;
    const RecJob& R = jobs.rec;
    const bool recj = dotj && R.frec != nullptr;
    // single-pass set-up: this unit's row statistics load under the transposes, and its dQ
    // rows start at zero (the single pass adds its partial sums to them)
    float rM = 0.f, rW = 1.f, rWs = 1.f;
    int rnm = 0;
    if (recj) {
      const int t = t0 + tid;
      if (tid < 32 && t < T) {
        const size_t rw = (size_t)bh * T + t;
        rM = R.row_max[rw];
        rW = R.W[rw];
        rWs = R.Ws[rw];
        rnm = R.n_max[rw];
      }
      const int nr = min(32, T - t0);
      float4* dq = reinterpret_cast<float4*>(R.dQ + nat + (size_t)t0 * d);
      for (int k4 = tid; k4 < nr * d / 4; k4 += 128) dq[k4] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float dacc[4] = {0.f, 0.f, 0.f, 0.f};
    for (int k0 = 0; k0 < d; k0 += 64) {
      float4 x[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int t = t0 + r + 8 * q;
        x[q] = t < T ? __ldg(reinterpret_cast<const float4*>(J.X + nat + (size_t)t * d + k0 + 4 * c4))
                     : make_float4(0.f, 0.f, 0.f, 0.f);
      }
      if (dotj) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int t = t0 + r + 8 * q;
          if (t < T) {
            const float4 y = __ldg(reinterpret_cast<const float4*>(J.Y + nat + (size_t)t * d + k0 + 4 * c4));
            dacc[q] = __fmaf_rn(x[q].x, y.x, dacc[q]);
            dacc[q] = __fmaf_rn(x[q].y, y.y, dacc[q]);
            dacc[q] = __fmaf_rn(x[q].z, y.z, dacc[q]);
            dacc[q] = __fmaf_rn(x[q].w, y.w, dacc[q]);
          }
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int rr = r + 8 * q, t = t0 + rr;
        float4 v = x[q];
        if constexpr (SPLIT) {
          float4 h, l;
          h.x = tf32_rna(v.x); l.x = __fsub_rn(v.x, h.x);
          h.y = tf32_rna(v.y); l.y = __fsub_rn(v.y, h.y);
          h.z = tf32_rna(v.z); l.z = __fsub_rn(v.z, h.z);
          h.w = tf32_rna(v.w); l.w = __fsub_rn(v.w, h.w);
          if (t < T && J.nat_hi) {
            const size_t off = nat + (size_t)t * d + k0 + 4 * c4;
            *reinterpret_cast<float4*>(J.nat_hi + off) = h;
            *reinterpret_cast<float4*>(J.nat_lo + off) = l;
          }
          v = h;
          ls[rr][4 * c4] = l.x; ls[rr][4 * c4 + 1] = l.y; ls[rr][4 * c4 + 2] = l.z; ls[rr][4 * c4 + 3] = l.w;
        }
        hs[rr][4 * c4] = v.x; hs[rr][4 * c4 + 1] = v.y; hs[rr][4 * c4 + 2] = v.z; hs[rr][4 * c4 + 3] = v.w;
      }
      __syncthreads();
      if (J.tr_hi) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int kk = k + 16 * q, t = t0 + 4 * tq;
          const size_t off = tr + (size_t)(k0 + kk) * Tp + t;
          *reinterpret_cast<float4*>(J.tr_hi + off) =
              make_float4(hs[4 * tq][kk], hs[4 * tq + 1][kk], hs[4 * tq + 2][kk], hs[4 * tq + 3][kk]);
          if constexpr (SPLIT) {
            if (J.tr_lo)
              *reinterpret_cast<float4*>(J.tr_lo + off) =
                  make_float4(ls[4 * tq][kk], ls[4 * tq + 1][kk], ls[4 * tq + 2][kk], ls[4 * tq + 3][kk]);
          }
        }
      }
      __syncthreads();
    }
    if (dotj) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float v = dacc[q];
#pragma unroll
        for (int o = 8; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        const int t = t0 + r + 8 * q;
        if (c4 == 0 && t < T) {
          J.dot[(size_t)bh * T + t] = v;
          dots[r + 8 * q] = v;
        }
      }
      if (recj) {
        __syncthreads();  // dots[] (the next unit writes it only after the syncs of its own loop)
        const int t = t0 + tid;
        if (tid < 32 && t < T &&
            prep_row_record(R, (size_t)bh * T + t, bh, t, rM, rW, rWs, rnm, dots[tid]))
          atomicOr(R.tie_any, 1);
      }
    }
  }
}

cudaError_t launch_prep(const PrepJobs& jobs, int BH, int T, int Tp, int d, bool split, int nsm, cudaStream_t s) {
  if (jobs.n <= 0) return cudaSuccess;
  const int units = jobs.n * BH * (Tp / 32);
  // sixteen 128-thread CTAs per SM (the most that are resident): a unit's loads, transpose
  // and stores run one after the other, so the SM hides their latency with other CTAs' units
  dim3 grid((unsigned)(units < 16 * nsm ? units : 16 * nsm)), block(128);
  return launch_pdl(split ? k_prep<true> : k_prep<false>, grid, block, 0, s, jobs, T, Tp, d, BH);
}

// ---------------------------------------------------------------------------
// Pass 1: row extrema (App. A: M = max_j s_j, m = min_j s_j over valid keys,
// lowest index among ties and the tie counts of Table "Edge cases").
// CTA = one 128-row query block of one head.  Compute thread t owns query row
// qb*128 + t%128 (TMEM lane t%128) and the column half t/128 of every 128-key
// score tile S = Q K^T.  The MMA warp computes S into two TMEM buffers
// (columns [0,128) and [128,256)), so the product of tile kb+1 runs while tile
// kb is reduced; the producer warp streams K tiles through a TMA ring.
// ---------------------------------------------------------------------------

// One 16-key chunk against a row's running extremum.  The chunk's maximum comes from a tree; a
// lane whose chunk beats its running maximum keeps a copy of the chunk (one select per key),
// and only the row's end looks for the equal keys in the last copy: some lane of a warp
// improves in most chunks, and finding the equal keys there took about five instructions per
// key against the select's one (pass 1 at B=8 H=12 T=1024 d=64: 31.6 -> 27.4 us).  A chunk that
// only ties with the running maximum (rare) counts its equal keys at once.  Masked keys
// (j > i) are -inf.  The minimum side runs on negated scores.  RAW: the scale is a
// power of two (d = 64: 2^-3), so the dot products are compared unscaled (exact scaling: only
// scores below 2^-123 in magnitude, subnormal after scaling, could merge), and the extremum is
// scaled once when the row is stored.
constexpr int SCW = 16;
struct RunMax {
  float M = -FLT_MAX;  // running maximum
  int j = -1;          // first key of the kept chunk
  int extra = 0;       // keys of later chunks equal to it
  float best[SCW];     // the kept chunk
  __device__ __forceinline__ void chunk(const float (&v)[SCW], int j0) {
    float t[SCW / 2];
#pragma unroll
    for (int q = 0; q < SCW / 2; ++q) t[q] = fmaxf(v[q], v[q + SCW / 2]);
#pragma unroll
    for (int w = SCW / 4; w >= 1; w >>= 1)
#pragma unroll
      for (int q = 0; q < w; ++q) t[q] = fmaxf(t[q], t[q + w]);
    const bool up = t[0] > M, tie = t[0] == M;
    if (__any_sync(0xffffffffu, up)) {
#pragma unroll
      for (int q = 0; q < SCW; ++q) best[q] = up ? v[q] : best[q];
      M = up ? t[0] : M;
      j = up ? j0 : j;
      extra = up ? 0 : extra;
    }
    if (__any_sync(0xffffffffu, tie)) {
      int c = 0;
#pragma unroll
      for (int q = 0; q < SCW; ++q) c += v[q] == M ? 1 : 0;
      if (tie) extra += c;
    }
  }
  // lowest index (0 where no chunk exceeded -FLT_MAX) and number of the keys equal to M
  __device__ __forceinline__ void finish(int& arg, int& n) const {
    uint32_t mk = 0;
#pragma unroll
    for (int q = 0; q < SCW; ++q) mk |= best[q] == M ? (1u << q) : 0u;
    arg = j < 0 ? 0 : j + __ffs(mk) - 1;
    n = extra + (j < 0 ? 0 : __popc(mk));
  }
};

// LW keys of a thread's row from key j0: masking, scaling, and the extrema.
template <bool MASK, bool MIN, bool RAW, int LW>
__device__ __forceinline__ void stats_chunk(float (&v)[LW], int j0, int i, float scale, RunMax& hi, RunMax& lo) {
  if constexpr (!RAW) {
#pragma unroll
    for (int jj = 0; jj < LW; ++jj) v[jj] = __fmul_rn(v[jj], scale);
  }
#pragma unroll
  for (int h = 0; h < LW; h += SCW) {
    float x[SCW];
#pragma unroll
    for (int q = 0; q < SCW; ++q) x[q] = MASK && j0 + h + q > i ? -INFINITY : v[h + q];
    hi.chunk(x, j0 + h);
    if constexpr (MIN) {
#pragma unroll
      for (int q = 0; q < SCW; ++q) x[q] = MASK && j0 + h + q > i ? -INFINITY : -v[h + q];
      lo.chunk(x, j0 + h);
    }
  }
}

// The extrema of a row's two column halves: value, lowest index, count (the half at `o` second).
__device__ __forceinline__ void merge_max(float& M, int& a, int& n, float Mo, int ao, int no) {
  if (Mo > M || (Mo == M && no > 0 && ao < a)) a = (Mo > M || n == 0) ? ao : min(a, ao);
  if (Mo > M) {
    n = no;
    M = Mo;
  } else if (Mo == M) {
    n += no;
  }
}

static dim3 launch_grid(const Params& p) { return dim3((unsigned)p.ngrid); }

template <bool MIN, bool RAW>
__global__ void __launch_bounds__(NTHR, RAW ? 2 : 1) k_fwd_stats(const __grid_constant__ Maps maps, const Params p,
                                                         const __grid_constant__ Sched sch) {
  uint8_t* sm = smem_base();
  const int D = p.d, tile = D * 512, parts = p.x3 ? 2 : 1, NS = p.nstage;
  uint8_t* sQ = sm + p.sm_a;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm + p.sm_bars);
  uint64_t* bar_q = bars;
  uint64_t* bar_full = bars + 1;
  uint64_t* bar_empty = bars + 1 + NS;
  uint64_t* bar_s = bars + 1 + 2 * NS;      // [2] S_b computed
  uint64_t* bar_sfree = bars + 3 + 2 * NS;  // [2] S_b read by every compute warp
  uint64_t* bar_qfree = bars + 5 + 2 * NS;  // the item's last product complete: Q may be reloaded
  uint64_t* bar_never = bars + 6 + 2 * NS;  // nothing arrives (test hook of the bounded waits)
  uint64_t* bar_drain = bars + 7 + 2 * NS;  // the MMA warp's clean-up commit
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + 8 + 2 * NS);
  float* xch = reinterpret_cast<float*>(sm + p.sm_rows);  // [6][128]
  const int tid = threadIdx.x, warp = warp_id_uniform();

  if (tid == 0) {
    mbar_init(bar_q, 1);
    for (int s = 0; s < NS; ++s) {
      mbar_init(&bar_full[s], 1);
      mbar_init(&bar_empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&bar_s[b], 1);
      mbar_init(&bar_sfree[b], NCOMP / 32);
    }
    mbar_init(bar_qfree, 1);
    mbar_init(bar_never, 1);
    mbar_init(bar_drain, 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(tslot, 256);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_trigger();
  pdl_wait();  // everything below may read what the previous kernel wrote
  const uint32_t tmem = *tslot;
  const bool skip = expire_first_wait(p, bar_never);

  // Work items as in pass 2: (query block, head), longest first, strided over the grid.
  if (skip) {
    // (the test hook's wait ran out before anything was issued)
  } else if (warp == PRODUCER_WARP) {
    int g = 0, n = 0;
    RingPos ld;  // stage of the next K tile loaded
    bool ok = true;
    for (int item = sched_item(sch, n); item < p.nitems && ok; item = sched_item(sch, ++n)) {
      const int qb = p.nqb - 1 - item / p.BH, bh = item % p.BH, nkb = qb + 1;
      if (n > 0 && !mbar_wait_warp(bar_qfree, (n - 1) & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_SYNC)) break;
      mbar_arrive_expect_tx(bar_q, parts * tile);
      load_rows_tile(sQ, &maps.q, bar_q, D, 128, 0, qb * 128, bh);
      if (p.x3) load_rows_tile(sQ + tile, &maps.q_lo, bar_q, D, 128, 0, qb * 128, bh);
      for (int kb = 0; kb < nkb; ++kb, ++g, ld.next(NS)) {
        const int s = ld.i;
        if (g >= NS && !mbar_wait_warp(&bar_empty[s], ld.ph ^ 1u, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA)) {
          ok = false;
          break;
        }
        uint8_t* dst = sm + p.sm_stage0 + s * p.sm_stage_bytes;
        mbar_arrive_expect_tx(&bar_full[s], parts * tile);
        load_rows_tile_boxed(dst, &maps.k, &bar_full[s], D, 128, 64, 0, kb * 128, bh);
        if (p.x3) load_rows_tile_boxed(dst + tile, &maps.k_lo, &bar_full[s], D, 128, 64, 0, kb * 128, bh);
      }
    }
    // clean-up: the last K tiles and Q tile issued have landed
    drain_ring(bar_full, ld, g, NS, p.wait_ns, p.status);
    if (n > 0) mbar_wait_warp(bar_q, (n - 1) & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA);
  } else if (warp == MMA_WARP) {
    int g = 0, n = 0;
    RingPos cs;  // stage of the current K tile
    bool ok = true;
    for (int item = sched_item(sch, n); item < p.nitems && ok; item = sched_item(sch, ++n)) {
      const int qb = p.nqb - 1 - item / p.BH, nkb = qb + 1;
      ok = mbar_wait_warp(bar_q, n & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA);
      for (int kb = 0; kb < nkb && ok; ++kb, cs.next(NS)) {
        const int gk = g + kb, s = cs.i, b = gk & 1;
        // S_b was last read two tiles ago
        if (gk >= 2 && !mbar_wait_warp(&bar_sfree[b], ((gk >> 1) - 1) & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_SYNC)) {
          ok = false;
          break;
        }
        if (!mbar_wait_warp(&bar_full[s], cs.ph, p.wait_ns, p.status, DEV_ERR_TIMEOUT_TMA)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint8_t* sk = sm + p.sm_stage0 + s * p.sm_stage_bytes;
        const uint32_t dcol = tmem + b * 128;
        if (p.x3) {
          mma_smem_smem(dcol, sQ + tile, sk, 128, D, false);  // Q_lo K_hi
          mma_smem_smem(dcol, sQ, sk + tile, 128, D, true);   // Q_hi K_lo
          mma_smem_smem(dcol, sQ, sk, 128, D, true);          // Q_hi K_hi
        } else {
          mma_smem_smem(dcol, sQ, sk, 128, D, false);
        }
        mma_commit(&bar_s[b]);
        mma_commit(&bar_empty[s]);
        if (kb + 1 == nkb) mma_commit(bar_qfree);
      }
      g += nkb;
    }
    drain_mma(bar_drain, p.wait_ns, p.status);  // clean-up: no product still writes TMEM
  } else {
    const int row = tid & 127, cg = tid >> 7;
    int g = 0, n = 0;
    bool failed = false;
    for (int item = sched_item(sch, n); item < p.nitems && !failed; item = sched_item(sch, ++n)) {
      const int qb = p.nqb - 1 - item / p.BH, bh = item % p.BH, nkb = qb + 1;
      const int i = qb * 128 + row;
      RunMax hi, lo;  // (lo: of the negated scores)
      for (int kb = 0; kb < nkb; ++kb) {
        const int gk = g + kb, b = gk & 1;
        if (!mbar_wait(&bar_s[b], (gk >> 1) & 1, p.wait_ns, p.status, DEV_ERR_TIMEOUT_MMA)) {
          failed = true;
          break;
        }
        tc_fence_after();
        const bool diag = kb == qb;
        constexpr int LW = MIN && RAW ? 16 : 32;  // (two CTAs per SM: two kept chunks leave few registers)
#pragma unroll 1
        for (int c = cg * 64; c < cg * 64 + 64; c += LW) {
          float v[LW];
          tmem_ldw<LW>(lane_addr(tmem, b * 128 + c), v);
          tmem_ld_wait();
          const int j0 = kb * 128 + c;
          if (diag)
            stats_chunk<true, MIN, RAW>(v, j0, i, p.scale, hi, lo);
          else
            stats_chunk<false, MIN, RAW>(v, j0, i, p.scale, hi, lo);
        }
        tc_fence_before();
        __syncwarp();
        if ((tid & 31) == 0) mbar_arrive(&bar_sfree[b]);
      }
      g += nkb;
      failed = group_any(BAR_COMPUTE, NCOMP, failed);
      if (failed) break;
      // combine the two column halves of each row
      float M = hi.M, m = -FLT_MAX;
      int amax, nmax, amin = 0, nmin = 0;
      hi.finish(amax, nmax);
      if constexpr (MIN) {
        m = lo.M;
        lo.finish(amin, nmin);
      }
      if (cg == 1) {
        xch[0 * 128 + row] = M;
        xch[1 * 128 + row] = m;
        xch[2 * 128 + row] = __int_as_float(amax);
        xch[3 * 128 + row] = __int_as_float(amin);
        xch[4 * 128 + row] = __int_as_float(nmax);
        xch[5 * 128 + row] = __int_as_float(nmin);
      }
      group_sync(BAR_COMPUTE, NCOMP);
      if (cg == 0 && i < p.T) {
        const float M1 = xch[row], m1 = xch[128 + row];
        const int amax1 = __float_as_int(xch[256 + row]), amin1 = __float_as_int(xch[384 + row]);
        const int nmax1 = __float_as_int(xch[512 + row]), nmin1 = __float_as_int(xch[640 + row]);
        merge_max(M, amax, nmax, M1, amax1, nmax1);
        if (MIN) {
          merge_max(m, amin, nmin, m1, amin1, nmin1);
          m = -m;
        } else {  // not computed: +inf, index -1, count 0
          m = INFINITY;
          amin = -1;
          nmin = 0;
        }
        if constexpr (RAW) {
          M = __fmul_rn(M, p.scale);
          m = __fmul_rn(m, p.scale);  // (+inf stays +inf when the minimum is not computed)
        }
        const size_t rw = (size_t)bh * p.T + i;
        p.row_max[rw] = M;
        p.row_min[rw] = m;
        p.arg_max[rw] = amax;
        p.arg_min[rw] = amin;
        p.n_max[rw] = nmax;
        p.n_min[rw] = nmin;
      }
      group_sync(BAR_COMPUTE, NCOMP);  // the exchange words are read before the next item writes them
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, 256);
}

cudaError_t launch_fwd_stats(const Maps& maps, const Params& p, int smem_bytes, cudaStream_t s, const Sched& sch) {
  // d = 64: scale 1/8, a power of two (RAW)
  auto kern = p.calib == CAL_MINMAX ? (p.d == 64 ? k_fwd_stats<true, true> : k_fwd_stats<true, false>)
                                    : (p.d == 64 ? k_fwd_stats<false, true> : k_fwd_stats<false, false>);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, launch_grid(p), dim3(NTHR), smem_bytes, s, maps, p, sch);
}

}  // namespace kint
