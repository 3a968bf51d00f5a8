// Local pass (Eq. 2) of more work items than SMs, head size 128: the tile arithmetic of attn_fwd_kernel (attn_fwd.cu, which
// has the layout of its warps and of tensor memory) in CTAs that process items until none is left.
//
// An item is a group of 256 query rows of one head.  The launch has one CTA per item, and a CTA whose last key blocks are on
// their way takes over one that has not started (cluster launch control).  So the next item's Q, K and V arrive, and its
// first scores are computed, under the end of the present one.  A CTA per item spends 8300 clk of each on its start, first
// loads and exit, of 107000 at W = 4096 and fewer for short sequences.  What that takes beside attn_fwd_kernel: results leave
// through a buffer of their own instead of the Q tiles, stored by a warp that does nothing else, and barriers whose
// phases run on over the items.
// Measured, local launch, a CTA per item -> this kernel: 32K tokens (28 heads) 1439 -> 1398 us, 16K packed in documents of 2700
// (32 heads) 454 -> 404, 4001 tokens (28 heads) 119 -> 113.  Over windows, call with S_save of 32K tokens (32/8 heads): W = 0
// 303 -> 170 us, 128 345 -> 248, 512 472 -> 375, 1000 679 -> 616, 4096 1963 -> 1890 (run to run 30); documents of 100 tokens
// 441 -> 273; 4001 tokens (28/4) W = 0 49 -> 37, 4096 125 -> 118.  Without S_save the gains are the same or larger.
// Launches of fewer items, and with D = 64 (where it gained nothing: 16K tokens 372 -> 382), stay with a CTA per item.
#include "l2a_common.cuh"
#include "sm100_prims.cuh"

namespace l2a {

namespace {

constexpr int D = 128;
constexpr int kNumTiles = 2;
constexpr int kStages = 2;
constexpr int kSoftmaxWarps = 8;
constexpr int kTmaWarp = kSoftmaxWarps, kMmaWarp = kSoftmaxWarps + 1, kStoreWarp = kSoftmaxWarps + 3;
constexpr int kThreads = (kSoftmaxWarps + 4) * 32;   // 384, of 168 registers each
constexpr int kSoftmaxRegs = 200, kOtherRegs = 104;  // (208 / 88 and 192 / 120 are 1 % slower, 216 / 72 is the same)
static_assert(kSoftmaxWarps * kSoftmaxRegs + 4 * kOtherRegs <= (kSoftmaxWarps + 4) * 168, "register shares exceed the launch allocation");
constexpr float kRescaleThreshold = 8.0f;            // log2 units

constexpr int kTileBytes = 128 * D * 2;
constexpr int kBoxBytes = 128 * 128;                 // one TMA box: 128 rows x 64 bf16 (128 B)
constexpr int kKOff = kNumTiles * kTileBytes;
constexpr int kVOff = kKOff + kStages * kTileBytes;
constexpr int kStageOff = kVOff + kStages * kTileBytes;     // an output tile on its way to global memory
constexpr int kBarOff = kStageOff + kTileBytes;
constexpr int kSmemTotal = kBarOff + 512 + 1024 /* alignment slack */;

struct TileRange {
  int active;            // tile has at least one row
  int min_pos, max_lo;   // position of the first row; largest "first visible key position" (the last row's)
  int lo, hi;            // first / last key block
};
struct Item {
  int exists;            // 0: no work is left
  int h, b, row0;
  int jlo, jhi;          // key blocks of the two tiles
  TileRange tr[kNumTiles];
};

struct Barriers {
  uint64_t claim_result[2];       // answer of the cluster launch control
  uint64_t q_full[kNumTiles], q_empty[kNumTiles];
  uint64_t k_full[kStages], k_empty[kStages];
  uint64_t v_full[kStages], v_empty[kStages];
  uint64_t s_full[kNumTiles];
  uint64_t p_half[kNumTiles], p_full[kNumTiles];   // P of the first 64 keys of a block / of all
  uint64_t o_final[kNumTiles];
  // The tiles take turns on one output buffer.  The store warp gives a tile its turn when the rows staged before have left,
  // so that each side waits for every phase of its barrier: a wait for every second phase of a common barrier returns at
  // once, by the parity of the phase before, when the barrier is two phases behind.
  uint64_t turn[kNumTiles];       // the buffer is the tile's
  uint64_t staged[kNumTiles];     // the tile's output rows are in it
  uint64_t claim;
  uint64_t item_full, item_empty; // `next` holds the next item / every role has it
  Item next;
  uint32_t tmem_base;
  int abort_flag;
};
static_assert(sizeof(Barriers) <= 512, "barrier block");

// Work of CTA `index`: largest row index first (longest tiles first), heads fastest for K/V reuse in L2.
__device__ __forceinline__ void make_item(const FwdArgs& a, int index, Item& w) {
  const int rest = index / a.Hq;
  w.exists = 1;
  w.h = index % a.Hq;
  w.b = rest % a.B;
  w.row0 = (a.pair_end - 1 - rest / a.B) * kRowsPerCta;
  w.jlo = 0x7fffffff;
  w.jhi = -1;
#pragma unroll
  for (int t = 0; t < kNumTiles; ++t) {
    TileRange& tr = w.tr[t];
    const int first = w.row0 + t * kTileM, last = min(first + kTileM, a.Lq) - 1;
    tr.active = first < a.Lq;
    tr.min_pos = tr.max_lo = 0;
    tr.lo = 1;
    tr.hi = 0;
    if (tr.active) {
      const int max_pos = last + a.q_pos_offset;
      tr.min_pos = first + a.q_pos_offset;
      int lo_pos = tr.min_pos - a.window;
      tr.max_lo = max_pos - a.window;
      if (a.seq_bounds != nullptr) {
        // packed sequences: no key before the start of the row's own sequence (starts ascend with the rows)
        lo_pos = max(lo_pos, a.seq_bounds[2 * first]);
        tr.max_lo = max(tr.max_lo, a.seq_bounds[2 * last]);
      }
      // A tile takes at least one block, all of it masked if a table names a start behind the tile: every role counts on the
      // barriers' phases of an active tile.
      tr.hi = max_pos / kTileN;
      tr.lo = min(lo_pos > 0 ? lo_pos / kTileN : 0, tr.hi);
      w.jlo = min(w.jlo, tr.lo);
      w.jhi = max(w.jhi, tr.hi);
    }
  }
}

__global__ void __launch_bounds__(kThreads, 1)
attn_fwd_local_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapK,
                      const __grid_constant__ CUtensorMap mapV, const __grid_constant__ CUtensorMap mapOut,
                      const __grid_constant__ CUtensorMap mapOut2, const FwdArgs a) {
  constexpr int kKSteps = D / 16;      // MMA k-steps of Q*K^T
  constexpr int kOCol0 = 2 * kTileN;   // first TMEM column of the O accumulators
  dependency_wait();
  dependents_release();                // the global pass may fill SMs as this one drains
  Item w;
  make_item(a, blockIdx.x, w);

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sQ = smem;
  uint8_t* sK = smem + kKOff;
  uint8_t* sV = smem + kVOff;
  uint8_t* sStage = smem + kStageOff;
  Barriers* bar = reinterpret_cast<Barriers*>(smem + kBarOff);
  volatile int* abort_flag = &bar->abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (tid == 0) {
    for (int t = 0; t < kNumTiles; ++t) {
      mbar_init(&bar->q_full[t], 1);
      mbar_init(&bar->q_empty[t], 1);
      mbar_init(&bar->s_full[t], 1);
      mbar_init(&bar->p_half[t], kTileM);
      mbar_init(&bar->p_full[t], kTileM);
      mbar_init(&bar->o_final[t], 1);
      mbar_init(&bar->turn[t], 1);
      mbar_init(&bar->staged[t], kTileM);
    }
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&bar->k_full[s], 1);
      mbar_init(&bar->k_empty[s], 1);
      mbar_init(&bar->v_full[s], 1);
      mbar_init(&bar->v_empty[s], 1);
    }
    mbar_init(&bar->claim, 1);
    mbar_init(&bar->item_full, 1);
    mbar_init(&bar->item_empty, kSoftmaxWarps + 2);     // the soft-max warps, the MMA issuer, the store warp
    bar->abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == kMmaWarp) {
    tmem_alloc(&bar->tmem_base, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bar->tmem_base;
  if (tmem != 0) {
    // all 512 columns were requested, so the allocation must start at column 0; the MMA warp relies on it to
    // keep its TMEM operand addresses compile-time constants
    __syncthreads();
    if (warp == kMmaWarp) tmem_dealloc(tmem, 512);
    if (tid == 0) atomicExch(a.status, 3);
    return;
  }

  if (warp == kTmaWarp) {
    // =========================================================================== TMA producer
    setmaxnreg_dec<kOtherRegs>();
    if (lane == 0) {
      tma_prefetch_desc(&mapQ);
      tma_prefetch_desc(&mapK);
      tma_prefetch_desc(&mapV);
    }
    const int G = a.Hq / a.Hkv;
    uint32_t it = 0, n_q1 = 0;                    // K/V blocks and second Q tiles loaded so far (tile 0 always has rows)
    for (uint32_t n_items = 0;; ++n_items) {
      bool ok = true;
      if (lane == 0) {
        const int hc = w.h * (D / 64), gc = w.h / G * (D / 64);
#pragma unroll
        for (int t = 0; t < kNumTiles; ++t) {
          if (!ok || !w.tr[t].active) continue;
          ok = mbar_wait(&bar->q_empty[t], ((t ? n_q1 : n_items) & 1) ^ 1, abort_flag);
          if (!ok) continue;
          mbar_expect_tx(&bar->q_full[t], kTileBytes);
          tma_load_4d(sQ + t * kTileBytes, &mapQ, &bar->q_full[t], 0, w.row0 + t * kTileM, hc, w.b);
          if (t) ++n_q1;
        }
        for (int j = w.jlo; ok && j <= w.jhi; ++j, ++it) {
          const int s = it % kStages;
          const uint32_t ph = (it / kStages) & 1;
          if (!mbar_wait(&bar->k_empty[s], ph ^ 1, abort_flag)) { ok = false; break; }
          mbar_expect_tx(&bar->k_full[s], kTileBytes);
          tma_load_4d(sK + s * kTileBytes, &mapK, &bar->k_full[s], 0, j * kTileN, gc, w.b);
          if (!mbar_wait(&bar->v_empty[s], ph ^ 1, abort_flag)) { ok = false; break; }
          mbar_expect_tx(&bar->v_full[s], kTileBytes);
          tma_load_4d(sV + s * kTileBytes, &mapV, &bar->v_full[s], 0, j * kTileN, gc, w.b);
        }
      }
      if (!__shfl_sync(0xffffffffu, ok, 0)) break;
      // the last blocks are on their way: the next item, taken over from a CTA that has not started
      if (lane == 0) {
        mbar_expect_tx(&bar->claim, 16);
        claim_cta(bar->claim_result, &bar->claim);
      }
      if (!mbar_wait_warp(&bar->claim, n_items & 1, abort_flag)) break;
      const int index = claimed_cta(bar->claim_result);
      fence_async_smem();          // the answer has been read before the next one is written
      if (index >= 0) make_item(a, index, w);
      else w.exists = 0;
      if (!mbar_wait_warp(&bar->item_empty, (n_items & 1) ^ 1, abort_flag)) break;
      if (lane == 0) {
        bar->next = w;
        mbar_arrive(&bar->item_full);
      }
      __syncwarp();
      if (index < 0) break;
    }
  } else if (warp == kMmaWarp) {
    // =========================================================================== MMA issuer
    setmaxnreg_dec<kOtherRegs>();
    if (elect_one()) {             // (one elected thread runs the loop: see tc_commit)
      constexpr uint32_t tmem = 0;   // checked above: TMEM operand addresses are immediates in this loop
      static_assert(kStages == 2 && kNumTiles == 2, "descriptor selects below assume two stages and two tiles");
      constexpr uint32_t idesc_qk = idesc_bf16_f32(kTileM, kTileN, 0, 0);
      constexpr uint32_t idesc_pv = idesc_bf16_f32(kTileM, D, 0, 1);
      const uint64_t dq0 = smem_desc_sw128(smem_u32(sQ), 16, 1024);
      const uint64_t dq1 = smem_desc_sw128(smem_u32(sQ + kTileBytes), 16, 1024);
      const uint64_t dk0 = smem_desc_sw128(smem_u32(sK), 16, 1024);
      const uint64_t dk1 = smem_desc_sw128(smem_u32(sK + kTileBytes), 16, 1024);
      const uint64_t dv0 = smem_desc_sw128(smem_u32(sV), kBoxBytes, 1024);
      const uint64_t dv1 = smem_desc_sw128(smem_u32(sV + kTileBytes), kBoxBytes, 1024);
      int jlo = w.jlo, jhi = w.jhi;
      int lo0 = w.tr[0].lo, hi0 = w.tr[0].hi, lo1 = w.tr[1].lo, hi1 = w.tr[1].hi;  // an inactive tile has lo > hi
      uint32_t p_cnt0 = 0, p_cnt1 = 0, q_cnt1 = 0, it = 0;       // running over the items
      bool ok = true;

      auto issue_qk = [&](int t, int s, bool last) {
        const uint64_t qd = t ? dq1 : dq0, kd = s ? dk1 : dk0;
#pragma unroll
        for (int kk = 0; kk < kKSteps; ++kk) {
          const uint32_t c = ((kk >> 2) * kBoxBytes + (kk & 3) * 32) >> 4;
          mma_ss(tmem + t * kTileN, qd + c, kd + c, idesc_qk, kk > 0);
        }
        tc_commit(&bar->s_full[t]);
        if (last) tc_commit(&bar->q_empty[t]);
      };
      auto issue_pv = [&](int t, int s, int half, uint32_t acc) {   // P*V of 64 keys
        const uint64_t vd = s ? dv1 : dv0;
        const uint32_t d = tmem + kOCol0 + t * D, p = tmem + t * kTileN + half * 64;
#pragma unroll
        for (int kk = 0; kk < kTileN / 32; ++kk)
          mma_ts(d, p + kk * 8, vd + (((half * 4 + kk) * 2048) >> 4), idesc_pv, kk > 0 ? 1u : acc);
      };
      auto in_range = [&](int t, int j) { return t ? (j >= lo1 && j <= hi1) : (j >= lo0 && j <= hi0); };

      for (uint32_t n_items = 0;; ++n_items) {
        // first key block: Q*K^T for both tiles
        const int s0 = it & 1;
        if (!mbar_spin(&bar->k_full[s0], (it >> 1) & 1, abort_flag)) ok = false;
#pragma unroll
        for (int t = 0; t < kNumTiles; ++t) {
          if (ok && in_range(t, jlo)) {
            if (!mbar_spin(&bar->q_full[t], (t ? q_cnt1 : n_items) & 1, abort_flag)) { ok = false; }
            else { tc_fence_after(); issue_qk(t, s0, jlo == (t ? hi1 : hi0)); }
          }
        }
        if (ok) tc_commit(&bar->k_empty[s0]);
        for (int j = jlo; ok && j <= jhi; ++j, ++it) {
          const int s = it & 1, sn = s ^ 1;
          const uint32_t ph = (it >> 1) & 1;
          const uint32_t phn = ((it + 1) >> 1) & 1;
          // both operand blocks of this step are waited for ahead of the probabilities: they arrive long before, and
          // a wait between P*V and the next Q*K^T, even one already satisfied, is part of a tile's serial chain
          if (!mbar_spin(&bar->v_full[s], ph, abort_flag)) { ok = false; break; }
          if (j + 1 <= jhi && !mbar_spin(&bar->k_full[sn], phn, abort_flag)) { ok = false; break; }
#pragma unroll
          for (int t = 0; t < kNumTiles; ++t) {
            if (ok && in_range(t, j)) {
              uint32_t& pc = t ? p_cnt1 : p_cnt0;
              if (mbar_spin(&bar->p_half[t], pc & 1, abort_flag)) {
                tc_fence_after();
                issue_pv(t, s, 0, j > (t ? lo1 : lo0) ? 1u : 0u);
              } else {
                ok = false;
              }
              if (ok && mbar_spin(&bar->p_full[t], pc & 1, abort_flag)) {
                ++pc;
                tc_fence_after();
                issue_pv(t, s, 1, 1u);
                if (j == (t ? hi1 : hi0)) tc_commit(&bar->o_final[t]);
              } else {
                ok = false;
              }
            }
            if (ok && j + 1 <= jhi && in_range(t, j + 1)) {
              if (j + 1 == (t ? lo1 : lo0) && !mbar_spin(&bar->q_full[t], (t ? q_cnt1 : n_items) & 1, abort_flag)) ok = false;
              if (ok) issue_qk(t, sn, j + 1 == (t ? hi1 : hi0));
            }
          }
          if (!ok) break;
          // V block j is released once both tiles' P*V have drained; K block j+1 once both Q*K^T have
          tc_commit(&bar->v_empty[s]);
          if (j + 1 <= jhi) tc_commit(&bar->k_empty[sn]);
        }
        q_cnt1 += lo1 <= hi1;
        if (!ok || !mbar_spin(&bar->item_full, n_items & 1, abort_flag)) break;
        const bool more = bar->next.exists != 0;
        jlo = bar->next.jlo; jhi = bar->next.jhi;
        lo0 = bar->next.tr[0].lo; hi0 = bar->next.tr[0].hi; lo1 = bar->next.tr[1].lo; hi1 = bar->next.tr[1].hi;
        mbar_arrive(&bar->item_empty);
        if (!more) break;
      }
    }
    __syncwarp();
  } else if (warp == kStoreWarp) {
    // =========================================================================== output tiles
    setmaxnreg_dec<kOtherRegs>();
    if (lane == 0) {
      int row0 = w.row0, hc = w.h * (D / 64), b = w.b, active1 = w.tr[1].active;
      uint32_t n1 = 0;
      bool ok = true;
      mbar_arrive(&bar->turn[0]);
      for (uint32_t n_items = 0;; ++n_items) {
        for (int t = 0; t < 1 + active1; ++t) {
          ok = mbar_wait(&bar->staged[t], (t ? n1 : n_items) & 1, abort_flag);
          if (!ok) break;
          tma_store_4d(&mapOut, sStage, 0, row0 + t * kTileM, hc, b);
          if (a.out2) tma_store_4d(&mapOut2, sStage, 0, row0 + t * kTileM, hc, b);
          tma_store_commit();
          tma_store_wait_read();
          mbar_arrive(&bar->turn[t < active1 ? 1 : 0]);     // tile 0 of the next item, if the tile was the item's last
        }
        n1 += active1;
        if (!ok || !mbar_wait(&bar->item_full, n_items & 1, abort_flag)) break;
        const bool more = bar->next.exists != 0;
        row0 = bar->next.row0; hc = bar->next.h * (D / 64); b = bar->next.b; active1 = bar->next.tr[1].active;
        mbar_arrive(&bar->item_empty);
        if (!more) break;
      }
    }
    __syncwarp();
  } else if (warp > kMmaWarp) {
    setmaxnreg_dec<kOtherRegs>();     // idle warp of the fourth warpgroup
  } else {
    // =========================================================================== soft-max warpgroups
    setmaxnreg_inc<kSoftmaxRegs>();
    const int t = warp >> 2;                 // tile of this warpgroup
    const int r = (warp & 3) * 32 + lane;    // row inside the tile == TMEM lane
    const uint32_t lane_base = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const uint32_t s_addr = tmem + lane_base + t * kTileN;        // this row's 128 score columns
    const uint32_t o_addr = tmem + lane_base + kOCol0 + t * D;    // its D accumulator columns
    TileRange my = t ? w.tr[1] : w.tr[0];
    int row0 = w.row0, h = w.h, b = w.b;
    uint32_t n_s = 0, n_o = 0;     // blocks and results of this tile so far
    bool ok = true;
    for (uint32_t n_items = 0;; ++n_items) {
      if (my.active) {
        float m_use = -INFINITY;   // reference maximum, exp2 domain
        float l = 0.f;             // row sum
        const int row = row0 + t * kTileM + r;
        const bool valid = row < a.Lq;
        const int pos = valid ? row + a.q_pos_offset : -1;            // largest visible key position
        int pos_lo = valid ? pos - a.window : 0x7fffffff;             // smallest visible key position
        if (valid && a.seq_bounds != nullptr) pos_lo = max(pos_lo, a.seq_bounds[2 * row]);

        for (int j = my.lo; j <= my.hi; ++j, ++n_s) {
          // warp-uniform outcome: the TMEM loads/stores below are warp-collective
          if (!__all_sync(0xffffffffu, mbar_wait(&bar->s_full[t], n_s & 1, abort_flag))) { ok = false; break; }
          tc_fence_after();
          const int k0 = j * kTileN;
          const bool partial = (k0 + kTileN - 1 > my.min_pos) || (k0 < my.max_lo);
          uint32_t v[4][32];       // the row's scores of this key block
#pragma unroll
          for (int c = 0; c < 4; ++c) tmem_ld32(s_addr + c * 32, v[c]);
          tmem_ld_wait();
          if (partial) {
            // edge block (causal diagonal, left window edge, ragged rows): one bit per column; masked scores become -inf
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const uint32_t visible = bit_range(pos_lo - k0 - c * 32, pos + 1 - k0 - c * 32);
#pragma unroll
              for (int e = 0; e < 32; ++e) v[c][e] = (visible >> e) & 1u ? v[c][e] : 0xff800000u;
            }
          }
          float mx0 = -INFINITY, mx1 = -INFINITY, mx2 = -INFINITY, mx3 = -INFINITY;
#pragma unroll
          for (int e = 0; e < 32; e += 2) {
            mx0 = fmax3(mx0, __uint_as_float(v[0][e]), __uint_as_float(v[0][e + 1]));
            mx1 = fmax3(mx1, __uint_as_float(v[1][e]), __uint_as_float(v[1][e + 1]));
            mx2 = fmax3(mx2, __uint_as_float(v[2][e]), __uint_as_float(v[2][e + 1]));
            mx3 = fmax3(mx3, __uint_as_float(v[3][e]), __uint_as_float(v[3][e + 1]));
          }
          const float m_new = fmaxf(m_use, fmaxf(fmaxf(mx0, mx1), fmaxf(mx2, mx3)) * a.scale_log2);

          // correction: rescale the running sum and the TMEM accumulator only when the maximum moved a lot
          const bool first = j == my.lo;
          const bool need = first ? false : (m_new - m_use > kRescaleThreshold);
          if (first) m_use = m_new;
          if (__any_sync(0xffffffffu, need)) {
            const float alpha = need ? fast_exp2(m_use - m_new) : 1.0f;
            l *= alpha;
#pragma unroll 1
            for (int c = 0; c < D / 32; ++c) {
              uint32_t o[32];
              tmem_ld32(o_addr + c * 32, o);
              tmem_ld_wait();
#pragma unroll
              for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
              tmem_st32(o_addr + c * 32, o);
            }
            if (need) m_use = m_new;
          }
          const float neg_m = (m_use == -INFINITY) ? 0.f : -m_use;
          // probabilities, a quarter of the exponentials on the FMA pipe; the bf16 P of keys 64h .. 64h+63 overwrites score
          // columns 64h .. 64h+31, and its first half is handed over while the second is computed
          // (the same order of additions as attn_fwd_kernel: the rows of a sequence are the same bits in a call of any size)
          float2 sum2 = make_float2(0.f, 0.f);
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            uint32_t pk[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              const float2 x = __ffma2_rn(make_float2(__uint_as_float(v[c][2 * e]), __uint_as_float(v[c][2 * e + 1])),
                                          make_float2(a.scale_log2, a.scale_log2), make_float2(neg_m, neg_m));
              const float2 p = e % 4 == 3 ? exp2_fma2(x) : make_float2(fast_exp2(x.x), fast_exp2(x.y));
              sum2 = __fadd2_rn(sum2, p);
              pk[e] = pack_bf16(p.x, p.y);
            }
            tmem_st16(s_addr + (c >> 1) * 64 + (c & 1) * 16, pk);
            if (c == 1) {
              tmem_st_wait();
              tc_fence_before();
              mbar_arrive(&bar->p_half[t]);
            }
          }
          l += sum2.x + sum2.y;
          tmem_st_wait();
          tc_fence_before();
          mbar_arrive(&bar->p_full[t]);
        }

        if (ok) ok = __all_sync(0xffffffffu, mbar_wait(&bar->o_final[t], n_o & 1, abort_flag));
        tc_fence_after();
        // ---- epilogue: O / l through the buffer that the tiles use in turn, log-sum-exp
        if (ok) {
          const float inv_l = (l > 0.f) ? 1.0f / l : 0.f;
          if (valid && a.lse != nullptr)
            a.lse[((int64_t)b * a.Hq + h) * a.Lq + row] = (m_use + log2f(l)) * 0.6931471805599453f;
          ok = __all_sync(0xffffffffu, mbar_wait(&bar->turn[t], n_o & 1, abort_flag));
#pragma unroll 1
          for (int c = 0; ok && c < D / 32; ++c) {
            uint32_t o[32];
            tmem_ld32(o_addr + c * 32, o);
            tmem_ld_wait();
            const uint32_t dst = smem_u32(sStage) + (c >> 1) * kBoxBytes + r * 128;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              uint32_t u[4];
#pragma unroll
              for (int k = 0; k < 4; ++k)
                u[k] = pack_bf16(__uint_as_float(o[8 * q + 2 * k]) * inv_l, __uint_as_float(o[8 * q + 2 * k + 1]) * inv_l);
              asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst + ((((c & 1) * 4 + q) ^ (r & 7)) << 4)),
                           "r"(u[0]), "r"(u[1]), "r"(u[2]), "r"(u[3]) : "memory");
            }
          }
          if (ok) {
            fence_async_smem();
            mbar_arrive(&bar->staged[t]);
          }
        }
        ++n_o;
      }
      // the next item; its first scores are computed while this one's results leave
      if (!ok || !__all_sync(0xffffffffu, mbar_wait(&bar->item_full, n_items & 1, abort_flag))) break;
      const bool more = bar->next.exists != 0;
      my = bar->next.tr[t];
      row0 = bar->next.row0; h = bar->next.h; b = bar->next.b;
      __syncwarp();
      if (lane == 0) mbar_arrive(&bar->item_empty);
      if (!more) break;
    }
  }

  // ---- teardown
  tc_fence_before();
  __syncthreads();
  if (bar->abort_flag) {
    // a bounded wait ran out: give copies still in flight time to land before shared memory is released
    const uint64_t t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
    if (tid == 0) atomicExch(a.status, 1);
    __syncthreads();
  }
  if (warp == kMmaWarp) tmem_dealloc(tmem, 512);
}

}  // namespace

cudaError_t launch_attn_fwd_local(const FwdArgs& a, int64_t items, const CUtensorMap& mapQ, const CUtensorMap& mapK,
                                  const CUtensorMap& mapV, const CUtensorMap& mapOut, const CUtensorMap& mapOut2,
                                  cudaStream_t stream) {
  static PerDeviceOnce once;
  const cudaError_t e = once.run([] {
    return cudaFuncSetAttribute(attn_fwd_local_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemTotal);
  });
  if (e != cudaSuccess) return e;
  return launch_dependent(attn_fwd_local_kernel, dim3((unsigned)items), kThreads, kSmemTotal, stream, a.overlap != 0, mapQ, mapK,
                          mapV, mapOut, mapOut2, a);
}

}  // namespace l2a
