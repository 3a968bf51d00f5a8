// Forward attention kernel for sm_100a: one kernel, two modes.
//
//   local  mode (Eq. 2, sliding-window mask of Section 2): query rows are sequence rows; key blocks
//          wholly outside the band [p - W, p] are never loaded.
//   global mode (Eq. 4; Algorithm 1): query rows are the compacted routed rows (Q_c), the G query heads of a KV group
//          packed into them (row c * G + i is head i of compact index c), so that the padding of the last group and the
//          positions a group spans are those of one head in G; the causal
//          mask uses the true position Q_idx of each compact index; the key loop of a tile stops at
//          the block holding its largest position; the epilogue scatters the result to O by
//          position and combines it with the local output already there (Eq. 5), and also stores
//          the compact output O_c and log-sum-exp L_c.
//
//          The soft-max warps gather the routed rows of Q of their tile themselves, while barriers and tensor memory are set up
//          (instead of a kernel ahead of the local pass that writes Q_c, 2 to 16 us).
// Packed heads against a launch over the rows of each head, global pass: 64K tokens (28/4 heads, 8 % routed) 2333 -> 2057 us,
// 64K in 24 documents (32/8, 20 %) 726 -> 607, 2 x 4096 tokens 104 -> 72; whole call of 2000 new tokens on 34K keys 421 -> 401.
//
// Structure (per CTA: two 128-row query tiles of one head or KV group, sharing the K/V stream):
//   warps 0-7       : soft-max + correction + epilogue.  Warpgroup t (4 warps) owns tile t; one thread per query
//                     row (= TMEM lane) holds the row's 128 scores of a key block in registers, so the row maximum
//                     and the row sum need no exchange between threads.
//   warp 8          : TMA producer (Q once; K and V blocks through 2-stage rings)
//   warp 9          : tcgen05 MMA issuer and TMEM owner
//   TMEM (512 cols) : S0 | S1 | O0 | O1 (fp32); the bf16 probabilities P overwrite the first half
//                     of their own S columns and are consumed from TMEM as the A operand of P*V.
// While one tile's soft-max runs on the CUDA cores, the tensor core works on the other tile.
// The online soft-max follows Algorithm 1 (running max m, running sum l, rescaled accumulator),
// in the exp2 domain, with the rescale skipped while the maximum grows by less than 2^8.
#include <algorithm>

#include "l2a_common.cuh"
#include "sm100_prims.cuh"

namespace l2a {

namespace {

constexpr int kNumTiles = 2;
constexpr int kStages = 2;
constexpr int kSoftmaxWarps = 8;
constexpr int kTmaWarp = kSoftmaxWarps, kMmaWarp = kSoftmaxWarps + 1;
// Twelve warps start with 168 registers each (warps are allocated four at a time, so ten would cost the same); the
// warpgroup of the TMA, MMA and two idle warps hands most of its share to the soft-max warps.
constexpr int kFwdThreads = (kSoftmaxWarps + 4) * 32;   // 384
constexpr int kSoftmaxRegs = 216, kOtherRegs = 72;
static_assert(kSoftmaxWarps * kSoftmaxRegs + 4 * kOtherRegs <= (kSoftmaxWarps + 4) * 168, "register shares exceed the launch allocation");
constexpr float kRescaleThreshold = 8.0f;  // log2 units

template <int D>
struct FwdSmem {
  static constexpr int kQTileBytes = kTileM * D * 2;
  static constexpr int kKVTileBytes = kTileN * D * 2;
  static constexpr int kBoxBytes = 128 * 128;  // one TMA box: 128 rows x 64 bf16 (128 B)
  static constexpr int kQOff = 0;
  static constexpr int kKOff = kQOff + kNumTiles * kQTileBytes;
  static constexpr int kVOff = kKOff + kStages * kKVTileBytes;
  static constexpr int kBarOff = kVOff + kStages * kKVTileBytes;
  static constexpr int kTotal = kBarOff + 256 + 1024 /* alignment slack */;
};

struct Barriers {
  uint64_t q_full[kNumTiles];
  uint64_t k_full[kStages], k_empty[kStages];
  uint64_t v_full[kStages], v_empty[kStages];
  uint64_t s_full[kNumTiles];
  uint64_t p_half[kNumTiles], p_full[kNumTiles];   // P of the first 64 keys of a block / of all
  uint64_t o_final[kNumTiles];
  uint64_t staged[kNumTiles];     // the tile's output rows are in shared memory
  uint32_t tmem_base;
  int abort_flag;
};

struct TileRange {
  int active;    // tile has at least one valid row
  int min_pos, max_pos;
  int max_lo;    // largest "first visible key position" among the rows (the last row's)
  int lo, hi;    // first / last key block
};

// Key blocks of the last group of a launch over compact rows, if the last row is routed
__host__ __device__ inline int longest_group(const FwdArgs& a) {
  const int keys = a.Lq + a.q_pos_offset - (a.shared_window ? a.window + 1 : 0);
  return keys > kTileN ? (keys + kTileN - 1) / kTileN : 1;
}

// Key-range splits of a launch over compact rows; every warp of a CTA calls it as a whole.  Each lane weighs one number of
// parts, in key blocks' time (1.55 us for two tiles): an item's start, end and the gap to the next one cost kItemCost, the
// combination kCombineCost and its data kPartCost a part.  Groups of about equal length (a chunk of new tokens) run in waves;
// those of a whole prefill, whose lengths fall from the longest to nothing, fill the SMs, longest first, up to half a part.  Nothing
// is gained by ending ahead of a local pass of fewer items than SMs.
struct KeySplit {
  int64_t groups;     // that exist (a batch entry of fewer routed rows has fewer)
  int parts, blocks;  // most parts of a group, key blocks of a part
};
// Clock traces of the items of 4001 tokens: set-up 2.9 us, first scores 3.2, 1.54 a block, the end 0.5, the rows of a part 1.5,
// to the next item 3.6.  Whole call, key ranges undivided below 32 key blocks and combined by the group's last CTA / this: 4001
// tokens (28/4 heads) 177 / 170 us, 100 new tokens on 60K keys 223 / 122, 500 (32/8, shared window) on 30K 193 / 140, 2000 on 33K
// 428 / 393.  (Twice as many parts: 4001 tokens 213: their rows, 133 KB a part, take longer than the blocks they save.)
// With the SMs of a small local pass taken as busy until it ends, against all SMs as free: 100 new tokens on 60K keys 123.5 -> 88, 500
// on 30K 138 -> 110, 64 on 40K 111 -> 78; of 1000 tokens and more the same.  From kSplitGroups groups on nothing was gained by parts.
// The same for a prefill, and a last wave behind a local pass that fills the SMs counted half (they come free one after the other):
// over 634 calls of 32 to 940 blocks and 1 to 127 groups the plan is on average 3.7 % off the best number of parts instead of 5.2 %,
// and 33 instead of 57 of them are more than 2.5 % slower than with at most eight parts of 16 blocks or more (20000 tokens, one head,
// window 4096: 102 -> 78 us, 81 with those).
constexpr float kItemCost = 7.f, kCombineCost = 3.f, kPartCost = 0.04f;
__device__ __forceinline__ KeySplit key_split(const FwdArgs& a) {
  const int lane = threadIdx.x & 31;
  int most = 0;
  for (int i = lane; i < a.B; i += 32) most = max(most, a.n_routed[i]);
  most = __reduce_max_sync(0xffffffffu, most);
  KeySplit k;
  k.groups = compact_groups(most, a.Hq / a.Hkv) * a.Hkv * a.B;
  k.parts = 1;
  const int longest = longest_group(a), shortest = max(0, longest - (a.Lq + kTileN - 1) / kTileN);
  if (a.part != nullptr && k.groups > 0 && k.groups < kSplitGroups && longest >= kMinSplitBlocks) {
    const int p = lane + 1, items = (int)k.groups * p;      // (kMaxKeySplit = 32 candidates, one a lane)
    const float part = (longest + p - 1) / p, sms = kSplitSms;
    float cost;
    if (2 * shortest >= longest) {
      // Waves of equal items, on the SMs that the local pass leaves and on its own from its end on: from the time at which the
      // SMs could have done them without waves up to a wave's end on either side.
      const float c = part + kItemCost, inv = __fdividef(1.f, c);
      if (a.local_items == 0) {
        const float waves = items * (1.f / kSplitSms);
        cost = fmaxf(1.f, 0.5f * (waves + ceilf(waves))) * c;
      } else {
        const float busy = (float)a.local_items, until = a.local_blocks + kItemCost;
        const float even = (items * c + busy * until) * (1.f / kSplitSms);
        const float k = ceilf(even * inv - 1e-3f), n = fmaxf(1.f, ceilf((even - until) * inv - 1e-3f));
        float t0 = k * c, t1 = until + n * c;
        if ((sms - busy) * k + busy * floorf(fmaxf(t0 - until, 0.f) * inv + 1e-3f) < items) t0 += c;
        if ((sms - busy) * floorf(t1 * inv + 1e-3f) + busy * n < items) t1 += c;
        cost = fmaxf(fminf(t0, t1), until);
      }
    } else {
      cost = fmaxf(part + kItemCost, (items * kItemCost + k.groups * 0.5f * (longest + shortest)) / sms + 0.5f * part);
      if (a.local_items > 0) cost = fmaxf(cost, a.local_blocks + kItemCost);
    }
    if (p > 1) cost += kCombineCost + kPartCost * items;
    const bool possible = items <= kSplitItems && p <= longest;
    const uint32_t key = possible ? ((uint32_t)fminf(cost * 16.f, 1e8f) << 5) + lane : 0xffffffffu;
    const uint32_t best = __reduce_min_sync(0xffffffffu, key);
    if (best != 0xffffffffu) k.parts = (int)(best & 31u) + 1;
  }
  k.blocks = (longest + k.parts - 1) / k.parts;
  return k;
}

// Row sum of row r of a slot
template <int D>
__device__ __forceinline__ void put_row_sum(const FwdArgs& a, int item, int r, float l) {
  a.part[(size_t)item * (kRowsPerCta * (D + 2)) + (r / kTileM) * (kTileM * (D + 2)) + kTileM * (D + 1) + r % kTileM] = l;
}

template <int D>
__global__ void __launch_bounds__(kFwdThreads, 1)
attn_fwd_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapK,
                const __grid_constant__ CUtensorMap mapV, const __grid_constant__ CUtensorMap mapOut,
                const __grid_constant__ CUtensorMap mapOut2, const FwdArgs a) {
  using SM = FwdSmem<D>;
  constexpr int kKSteps = D / 16;      // MMA k-steps of Q*K^T
  constexpr int kOCol0 = 2 * kTileN;   // first TMEM column of the O accumulators

  // ---- work item: heaviest first (largest row index first), heads fastest for K/V reuse in L2
  const bool compact = a.global_mode && !a.all_rows;           // rows are (compact index into q_idx, head of the group)
  const int G = a.Hq / a.Hkv;
  int item = blockIdx.x, split = 0, n_split = 1, pi;
  // (2: what is read up to the combination was complete before the local pass, a plain launch, started)
  if (a.overlap != 2) dependency_wait();
  // the global pass may fill SMs as the local one drains, the combination as the global one does
  if (!a.global_mode || a.part != nullptr) dependents_release();
  KeySplit ks;
  if (compact) {
    // the launch covers every row that could be routed; the groups that exist come first
    ks = key_split(a);
    if (item >= ks.groups * ks.parts) { dependency_wait(); return; }
    split = item % ks.parts;
    item /= ks.parts;
  }
  const int group = item;
  const int n_heads = compact ? a.Hkv : a.Hq;
  const int hi = item % n_heads;                               // KV head, or head of the rows
  const int rest = item / n_heads;
  const int b = rest % a.B;
  const int g = compact ? hi : hi / G;
  const int pack = compact ? G : 1;                            // rows of one token
  const int n_rows = compact ? a.n_routed[b] * G : a.Lq;       // valid rows of this batch entry
  pi = (compact ? (n_rows + kRowsPerCta - 1) / kRowsPerCta : a.pair_end) - 1 - rest / a.B;
  const int row0 = pi * kRowsPerCta;
  if (pi < 0 || row0 >= n_rows) { dependency_wait(); return; }

  const int32_t* q_idx_b = a.q_idx + (int64_t)b * a.Lq;
  const int w_eff = a.global_mode ? 0x3fffffff : a.window;
  // shared-window mode: a row at position p attends to the keys 0 .. p - W - 1 only (the window p - W .. p is the
  // local pass's share and enters in the epilogue)
  const bool shared = a.global_mode && a.shared_window;
  const int vis_shift = shared ? a.window + 1 : 0;
  if (a.global_mode && (a.row_begin > 0 || a.row_end < a.Lq)) {
    // launches restricted to a row range take the groups whose last row falls into it: every group exactly once
    const int c_last = min(row0 + kRowsPerCta, n_rows) - 1;
    const int t_last = compact ? q_idx_b[c_last / pack] : c_last;
    if (t_last < a.row_begin || t_last >= a.row_end) { dependency_wait(); return; }
  }

  TileRange tr[kNumTiles];
  int jlo = 0x7fffffff, jhi = -1;
#pragma unroll
  for (int t = 0; t < kNumTiles; ++t) {
    const int first = row0 + t * kTileM;
    int last = first + kTileM - 1;
    if (last > n_rows - 1) last = n_rows - 1;
    tr[t].active = first < n_rows;
    if (tr[t].active) {
      const int first_seq = compact ? q_idx_b[first / pack] : first, last_seq = compact ? q_idx_b[last / pack] : last;
      tr[t].min_pos = first_seq + a.q_pos_offset;
      tr[t].max_pos = last_seq + a.q_pos_offset;
      int lo_pos = tr[t].min_pos - w_eff;
      tr[t].max_lo = tr[t].max_pos - w_eff;
      if (a.seq_bounds != nullptr) {
        // packed sequences: no key before the start of the row's own sequence (starts ascend with the rows)
        lo_pos = max(lo_pos, a.seq_bounds[2 * first_seq]);
        tr[t].max_lo = max(tr[t].max_lo, a.seq_bounds[2 * last_seq]);
      }
      const int hi_pos = tr[t].max_pos - vis_shift;   // last key position any row of the tile attends to
      if (hi_pos >= 0 && hi_pos >= lo_pos) {
        tr[t].lo = lo_pos > 0 ? lo_pos / kTileN : 0;
        tr[t].hi = hi_pos / kTileN;
        jlo = min(jlo, tr[t].lo);
        jhi = max(jhi, tr[t].hi);
      } else {
        tr[t].lo = 1; tr[t].hi = 0;   // shared-window mode: every key of these rows lies inside the window
      }
    } else {
      tr[t].min_pos = tr[t].max_pos = tr[t].max_lo = 0;
      tr[t].lo = 1; tr[t].hi = 0;
    }
  }

  // this item's part of the group's key blocks
  if (compact && a.part != nullptr) {
    if (ks.parts > 1 && jhi - jlo + 1 >= kMinSplitGroup) n_split = min(ks.parts, (jhi - jlo + ks.blocks) / ks.blocks);
    if (split >= n_split) { dependency_wait(); return; }
    // the plan for fwd_combine_kernel, undivided groups included: slots of a group, parts in use
    if (split == 0 && threadIdx.x == 0 && group < kSplitGroups) a.group_parts[group] = (ks.parts << 16) | n_split;
  }
  if (n_split > 1) {
    const int n = jhi - jlo + 1, first = jlo;
    jlo = first + n * split / n_split;
    jhi = first + n * (split + 1) / n_split - 1;
#pragma unroll
    for (int t = 0; t < kNumTiles; ++t) {
      tr[t].lo = max(tr[t].lo, jlo);
      tr[t].hi = min(tr[t].hi, jhi);
    }
  }

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sQ = smem + SM::kQOff;
  uint8_t* sK = smem + SM::kKOff;
  uint8_t* sV = smem + SM::kVOff;
  Barriers* bar = reinterpret_cast<Barriers*>(smem + SM::kBarOff);
  volatile int* abort_flag = &bar->abort_flag;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (compact && warp < kSoftmaxWarps) {
    // Algorithm 1, step 1: each soft-max warp brings its 32 rows of Q, 16-byte pieces, into the layout a TMA copy would leave
    constexpr int kPieces = D / 8, kRowsPerStep = 32 / kPieces;
    const int row = row0 + warp * 32 + lane, c = row / pack;
    const int t = row < n_rows ? q_idx_b[c] : -1;
    // (debug build: an index outside of Q is reported and its row read as zeros)
    const bool inside = row < n_rows && dbg_in_range(t >= 0 && t < a.Lq, a.status);
    const bf16* src = inside ? a.q + b * a.q_st.b + t * a.q_st.t + (int64_t)(g * G + row - c * pack) * D : nullptr;
    const int piece = lane % kPieces;
    uint4 x[kPieces];
#pragma unroll
    for (int k = 0; k < kPieces; ++k) {
      const bf16* p = reinterpret_cast<const bf16*>(
          __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(src), k * kRowsPerStep + lane / kPieces));
      x[k] = p != nullptr ? __ldcg(reinterpret_cast<const uint4*>(p) + piece) : make_uint4(0, 0, 0, 0);
    }
    const uint32_t dst = smem_u32(sQ + (warp >> 2) * SM::kQTileBytes) + (piece >> 3) * SM::kBoxBytes;
#pragma unroll
    for (int k = 0; k < kPieces; ++k) {
      const int rr = (warp & 3) * 32 + k * kRowsPerStep + lane / kPieces;
      asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst + rr * 128 + (((piece & 7) ^ (rr & 7)) << 4)),
                   "r"(x[k].x), "r"(x[k].y), "r"(x[k].z), "r"(x[k].w) : "memory");
    }
    fence_async_smem();
  }
  if (tid == kTmaWarp * 32) {
    for (int t = 0; t < kNumTiles; ++t) {
      mbar_init(&bar->q_full[t], compact ? kTileM : 1);
      mbar_init(&bar->s_full[t], 1);
      mbar_init(&bar->p_half[t], kTileM);
      mbar_init(&bar->p_full[t], kTileM);
      mbar_init(&bar->o_final[t], 1);
      mbar_init(&bar->staged[t], kTileM);
    }
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&bar->k_full[s], 1);
      mbar_init(&bar->k_empty[s], 1);
      mbar_init(&bar->v_full[s], 1);
      mbar_init(&bar->v_empty[s], 1);
    }
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
    dependency_wait();
    // all 512 columns were requested, so the allocation must start at column 0; the MMA warp relies on it to
    // keep its TMEM operand addresses compile-time constants
    __syncthreads();
    if (warp == kMmaWarp) tmem_dealloc(tmem, 512);
    if (n_split > 1 && tid < kRowsPerCta) put_row_sum<D>(a, blockIdx.x, tid, -1.f);
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
      for (int t = 0; t < kNumTiles; ++t) {
        if (compact || !tr[t].active || tr[t].lo > tr[t].hi) continue;      // (compact rows: the soft-max warps gather them)
        mbar_expect_tx(&bar->q_full[t], SM::kQTileBytes);
        tma_load_4d(sQ + t * SM::kQTileBytes, &mapQ, &bar->q_full[t], 0, row0 + t * kTileM, hi * (D / 64), b);
      }
      for (int j = jlo; j <= jhi; ++j) {
        const int it = j - jlo, s = it % kStages;
        const uint32_t ph = (it / kStages) & 1;
        if (!mbar_wait(&bar->k_empty[s], ph ^ 1, abort_flag)) break;
        mbar_expect_tx(&bar->k_full[s], SM::kKVTileBytes);
        tma_load_4d(sK + s * SM::kKVTileBytes, &mapK, &bar->k_full[s], 0, j * kTileN, g * (D / 64), b);
        if (!mbar_wait(&bar->v_empty[s], ph ^ 1, abort_flag)) break;
        mbar_expect_tx(&bar->v_full[s], SM::kKVTileBytes);
        tma_load_4d(sV + s * SM::kKVTileBytes, &mapV, &bar->v_full[s], 0, j * kTileN, g * (D / 64), b);
      }
    }
    __syncwarp();
  } else if (warp == kMmaWarp) {
    // =========================================================================== MMA issuer
    setmaxnreg_dec<kOtherRegs>();
    // One elected thread runs this loop (see tc_commit): operand descriptors are built once per tile / stage and advanced
    // by compile-time constants, so that issuing stays well under the 64 clocks one 128x128x16 MMA takes.
    if (elect_one()) {
      constexpr uint32_t tmem = 0;   // checked above: TMEM operand addresses are immediates in this loop
      static_assert(kStages == 2 && kNumTiles == 2, "descriptor selects below assume two stages and two tiles");
      constexpr uint32_t idesc_qk = idesc_bf16_f32(kTileM, kTileN, 0, 0);
      constexpr uint32_t idesc_pv = idesc_bf16_f32(kTileM, D, 0, 1);
      const uint64_t dq0 = smem_desc_sw128(smem_u32(sQ), 16, 1024);
      const uint64_t dq1 = smem_desc_sw128(smem_u32(sQ + SM::kQTileBytes), 16, 1024);
      const uint64_t dk0 = smem_desc_sw128(smem_u32(sK), 16, 1024);
      const uint64_t dk1 = smem_desc_sw128(smem_u32(sK + SM::kKVTileBytes), 16, 1024);
      const uint64_t dv0 = smem_desc_sw128(smem_u32(sV), SM::kBoxBytes, 1024);
      const uint64_t dv1 = smem_desc_sw128(smem_u32(sV + SM::kKVTileBytes), SM::kBoxBytes, 1024);
      const int lo0 = tr[0].lo, hi0 = tr[0].hi, lo1 = tr[1].lo, hi1 = tr[1].hi;  // an inactive tile has lo > hi
      uint32_t p_cnt0 = 0, p_cnt1 = 0;
      bool ok = true;

      auto issue_qk = [&](int t, int s) {
        const uint64_t qd = t ? dq1 : dq0, kd = s ? dk1 : dk0;
        const uint32_t d = tmem + t * kTileN;
#pragma unroll
        for (int kk = 0; kk < kKSteps; ++kk) {
          const uint32_t c = ((kk >> 2) * SM::kBoxBytes + (kk & 3) * 32) >> 4;
          mma_ss(d, qd + c, kd + c, idesc_qk, kk > 0);
        }
        tc_commit(&bar->s_full[t]);
      };
      auto issue_pv = [&](int t, int s, int half, uint32_t acc) {   // P*V of 64 keys
        const uint64_t vd = s ? dv1 : dv0;
        const uint32_t d = tmem + kOCol0 + t * D, p = tmem + t * kTileN + half * 64;
#pragma unroll
        for (int kk = 0; kk < kTileN / 32; ++kk)
          mma_ts(d, p + kk * 8, vd + (((half * 4 + kk) * 2048) >> 4), idesc_pv, kk > 0 ? 1u : acc);
      };
      auto in_range = [&](int t, int j) { return t ? (j >= lo1 && j <= hi1) : (j >= lo0 && j <= hi0); };

      if (jhi < jlo) ok = false;   // no key block at all (shared-window mode): nothing to issue, nobody waits
      // first key block: Q*K^T for both tiles
      if (ok && !mbar_spin(&bar->k_full[0], 0, abort_flag)) ok = false;
#pragma unroll
      for (int t = 0; t < kNumTiles; ++t) {
        if (ok && in_range(t, jlo)) {
          if (!mbar_spin(&bar->q_full[t], 0, abort_flag)) { ok = false; }
          else { tc_fence_after(); issue_qk(t, 0); }
        }
      }
      if (ok) tc_commit(&bar->k_empty[0]);

      for (int j = jlo; ok && j <= jhi; ++j) {
        const int it = j - jlo, s = it & 1, sn = s ^ 1;
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
            if (j + 1 == (t ? lo1 : lo0) && !mbar_spin(&bar->q_full[t], 0, abort_flag)) ok = false;
            if (ok) issue_qk(t, sn);
          }
        }
        if (!ok) break;
        // V block j is released once both tiles' P*V have drained; K block j+1 once both Q*K^T have
        tc_commit(&bar->v_empty[s]);
        if (j + 1 <= jhi) tc_commit(&bar->k_empty[sn]);
      }
    }
    __syncwarp();
  } else if (warp > kMmaWarp) {
    setmaxnreg_dec<kOtherRegs>();     // idle warps of the fourth warpgroup
  } else {
    // =========================================================================== soft-max warpgroups
    setmaxnreg_inc<kSoftmaxRegs>();
    const int t = warp >> 2;                 // tile of this warpgroup
    const int r = (warp & 3) * 32 + lane;    // row inside the tile == TMEM lane
    const uint32_t lane_base = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const uint32_t s_addr = tmem + lane_base + t * kTileN;        // this row's 128 score columns
    const uint32_t o_addr = tmem + lane_base + kOCol0 + t * D;    // its D accumulator columns
    const TileRange my = t ? tr[1] : tr[0];
    float m_use = -INFINITY;   // reference maximum, exp2 domain
    float l = 0.f;             // row sum
    bool ok = true;
    const int n_my = my.active ? my.hi - my.lo + 1 : 0;
    if (my.active) {
      const int row = row0 + t * kTileM + r;           // sequence row (local) or compact row (global)
      const bool valid = row < n_rows;
      const int seq_row = valid ? (compact ? q_idx_b[row / pack] : row) : -1;
      const int pos = valid ? seq_row + a.q_pos_offset - vis_shift : -1;   // largest visible key position
      int pos_lo = valid ? (pos - w_eff) : 0x7fffffff;                     // smallest visible key position
      if (valid && a.seq_bounds != nullptr) pos_lo = max(pos_lo, a.seq_bounds[2 * seq_row]);

      if (compact && n_my > 0) mbar_arrive(&bar->q_full[t]);       // gathered ahead of the set-up

      for (int i = 0; i < n_my; ++i) {
        const int j = my.lo + i;
        // warp-uniform outcome: the TMEM loads/stores below are warp-collective
        if (!__all_sync(0xffffffffu, mbar_wait(&bar->s_full[t], i & 1, abort_flag))) { ok = false; break; }
        tc_fence_after();
        const int k0 = j * kTileN;
        const bool partial = (k0 + kTileN - 1 > my.min_pos - vis_shift) || (k0 < my.max_lo);
        uint32_t v[4][32];       // the row's scores of this key block
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_ld32(s_addr + c * 32, v[c]);
        tmem_ld_wait();
        if (partial) {
          // edge block (causal diagonal, left window edge, ragged rows): the row's visible keys are one range, hence one
          // bit per column; masked scores become -inf, whose exponential is an exact zero below.  (Two comparisons of
          // key positions per score instead cost 1100 to 2000 clk a block, next to 1800 for all of an interior one.)
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
        const float mx = fmaxf(fmaxf(mx0, mx1), fmaxf(mx2, mx3));
        const float m_new = fmaxf(m_use, mx * a.scale_log2);

        // correction: rescale the running sum and the TMEM accumulator only when the maximum moved a lot
        const bool need = (i == 0) ? false : (m_new - m_use > kRescaleThreshold);
        if (i == 0) m_use = m_new;
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
        const float m_eff = (m_use == -INFINITY) ? 0.f : m_use;
        const float neg_m = -m_eff;
        // probabilities; the bf16 P of keys 64h .. 64h+63 overwrites score columns 64h .. 64h+31.  A quarter of the
        // exponentials runs on the FMA pipe: ex2 takes 8 clk a warp, 1024 of the 1430 clk this took with all on the
        // special-function unit, and it is part of the tile's serial chain S -> P -> P*V -> next S (1200 clk now; three
        // eighths and more are slower again).  The first half of P is handed over while the second is computed.
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

      if (ok && n_my > 0) ok = __all_sync(0xffffffffu, mbar_wait(&bar->o_final[t], 0, abort_flag));
      tc_fence_after();
    }
    if (n_split > 1 && my.active) {
      // Split key range: the rows go to this item's slot unnormalised, 16-byte pieces 128 rows apart; fwd_combine_kernel
      // combines the slots of the group.  A negative sum marks a wait that ran out.
      float* slot = a.part + (size_t)blockIdx.x * (kRowsPerCta * (D + 2)) + t * kTileM * (D + 2);
#pragma unroll 1
      for (int c = 0; ok && n_my > 0 && c < D / 32; ++c) {
        uint32_t o[32];
        tmem_ld32(o_addr + c * 32, o);
        tmem_ld_wait();
#pragma unroll
        for (int x = 0; x < 8; ++x)
          *reinterpret_cast<uint4*>(slot + ((c * 8 + x) * kTileM + r) * 4) =
              make_uint4(o[4 * x], o[4 * x + 1], o[4 * x + 2], o[4 * x + 3]);
      }
      slot[kTileM * D + r] = m_use;
      put_row_sum<D>(a, blockIdx.x, t * kTileM + r, !ok ? -1.f : n_my > 0 ? l : 0.f);
    }
    if (my.active && n_split == 1) {
      // ---- epilogue: O / l, log-sum-exp, store (local) or scatter + combine (global)
      if (a.global_mode) dependency_wait();      // out2 and lse_loc are the local pass's results
      const int tile_row = row0 + t * kTileM + r;
      const bool valid = tile_row < n_rows;
      const int row = compact ? tile_row / pack : tile_row;      // sequence row, or compact index
      const int h = compact ? g * G + (tile_row - row * pack) : hi;
      const int seq_row = valid ? (compact ? q_idx_b[row] : row) : -1;
      if (ok) {
        float inv_l = (l > 0.f) ? 1.0f / l : 0.f;
        float lse2 = m_use + log2f(l);   // log-sum-exp in the exp2 domain
        float c_loc = 0.f;               // shared-window mode: weight of the local result s_t in a_t
        if (shared && valid) {
          // a_t = (e^{lse_out} o_out + e^{lse_loc} s_t) / (e^{lse_out} + e^{lse_loc}): the softmax over the whole
          // prefix, split into the keys before the window (this kernel) and the window (the local pass)
          const float lse_out2 = (l > 0.f) ? lse2 : -INFINITY;
          const float lse_loc2 = a.lse_loc[((int64_t)b * a.Hq + h) * a.Lq + seq_row] * 1.4426950408889634f;
          const float mm = fmaxf(lse_out2, lse_loc2);
          const float w_out = fast_exp2(lse_out2 - mm), w_loc = fast_exp2(lse_loc2 - mm);
          const float inv = 1.0f / (w_out + w_loc);
          inv_l *= w_out * inv;
          c_loc = w_loc * inv;
          lse2 = mm + log2f(w_out + w_loc);
        }
        if (valid && a.lse != nullptr) {
          const float lse = lse2 * 0.6931471805599453f;
          a.lse[((int64_t)b * a.Hq + h) * a.Lq + row] = lse;
        }
        if (!a.global_mode) {
          // A tile of consecutive rows leaves through its Q buffer (free once its last product is done) with one TMA store
          // per destination.  A store per thread and row, 32 lines an instruction, took 4900 clk a tile, of 108000 for
          // all of a CTA at W = 4096; rows gathered from shared memory by plain stores took as long.
#pragma unroll 1
          for (int c = 0; c < D / 32; ++c) {
            uint32_t o[32];
            tmem_ld32(o_addr + c * 32, o);
            tmem_ld_wait();
            const uint32_t dst = smem_u32(sQ + t * SM::kQTileBytes) + (c >> 1) * SM::kBoxBytes + r * 128;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              uint32_t w[4];
#pragma unroll
              for (int k = 0; k < 4; ++k)
                w[k] = pack_bf16(__uint_as_float(o[8 * q + 2 * k]) * inv_l, __uint_as_float(o[8 * q + 2 * k + 1]) * inv_l);
              asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst + ((((c & 1) * 4 + q) ^ (r & 7)) << 4)),
                           "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]) : "memory");
            }
          }
          fence_async_smem();
          mbar_arrive(&bar->staged[t]);
          if (r == 0 && mbar_wait(&bar->staged[t], 0, abort_flag)) {
            tma_store_4d(&mapOut, sQ + t * SM::kQTileBytes, 0, row0 + t * kTileM, hi * (D / 64), b);
            if (a.out2) tma_store_4d(&mapOut2, sQ + t * SM::kQTileBytes, 0, row0 + t * kTileM, hi * (D / 64), b);
            tma_store_commit();
            tma_store_wait_read();
          }
        } else {
          bf16* dst1 = nullptr;   // row-indexed destination (s rows, or compact a rows)
          bf16* dst2 = nullptr;   // position-indexed destination
          if (valid && dbg_in_range(row >= 0 && row < a.Lq && seq_row >= 0 && seq_row < a.Lq, a.status)) {
            if (a.out) dst1 = a.out + b * a.out_st.b + row * a.out_st.t + (int64_t)h * D;
            if (a.out2 && (a.combine_mask == nullptr || a.combine_mask[(int64_t)b * a.Lq + seq_row]))
              dst2 = a.out2 + b * a.out2_st.b + seq_row * a.out2_st.t + (int64_t)h * D;
          }
          const bool accumulate = a.global_mode && a.accumulate_into_out2;
#pragma unroll 1
          for (int c = 0; c < D / 32; ++c) {
            uint32_t o[32];
            if (n_my > 0) {
              tmem_ld32(o_addr + c * 32, o);
              tmem_ld_wait();
            } else {
#pragma unroll
              for (int e = 0; e < 32; ++e) o[e] = 0u;    // no key before the window: the accumulator was never written
            }
            float f[32];
#pragma unroll
            for (int e = 0; e < 32; ++e) f[e] = __uint_as_float(o[e]) * inv_l;
            if (shared && dst2) {
              const uint4* s4 = reinterpret_cast<const uint4*>(dst2 + c * 32);   // s_t, written by the local pass
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const uint4 old = s4[q];
                const uint32_t ow[4] = {old.x, old.y, old.z, old.w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                  f[8 * q + 2 * k] = fmaf(c_loc, __uint_as_float(ow[k] << 16), f[8 * q + 2 * k]);
                  f[8 * q + 2 * k + 1] = fmaf(c_loc, __uint_as_float(ow[k] & 0xffff0000u), f[8 * q + 2 * k + 1]);
                }
              }
            }
            if (dst1) {
              uint4* d4 = reinterpret_cast<uint4*>(dst1 + c * 32);
#pragma unroll
              for (int q = 0; q < 4; ++q)
                d4[q] = make_uint4(pack_bf16(f[8 * q], f[8 * q + 1]), pack_bf16(f[8 * q + 2], f[8 * q + 3]),
                                   pack_bf16(f[8 * q + 4], f[8 * q + 5]), pack_bf16(f[8 * q + 6], f[8 * q + 7]));
            }
            if (dst2) {
              uint4* d4 = reinterpret_cast<uint4*>(dst2 + c * 32);
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                if (accumulate) {
                  const uint4 old = d4[q];
                  const uint32_t ow[4] = {old.x, old.y, old.z, old.w};
#pragma unroll
                  for (int k = 0; k < 4; ++k) {
                    f[8 * q + 2 * k] += __uint_as_float(ow[k] << 16);
                    f[8 * q + 2 * k + 1] += __uint_as_float(ow[k] & 0xffff0000u);
                  }
                }
                d4[q] = make_uint4(pack_bf16(f[8 * q], f[8 * q + 1]), pack_bf16(f[8 * q + 2], f[8 * q + 3]),
                                   pack_bf16(f[8 * q + 4], f[8 * q + 5]), pack_bf16(f[8 * q + 6], f[8 * q + 7]));
              }
            }
          }
        }
      }
    }
  }

  // ---- teardown
  tc_fence_before();
  dependency_wait();       // this grid must not count as finished before the one it overlaps with
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

// Combines the parts of the groups whose key range was split, and does with their rows what the epilogue above does with
// those of an undivided group.  A CTA takes 32 rows, a thread D / 8 columns of one: the parts of a group are read by eight CTAs
// instead of the one that finished last (latency bound).  The plan comes from the workspace, where attn_fwd_kernel left it: a second
// evaluation of key_split, compiled into another kernel, could round a cost differently and look for the parts in other slots.
template <int D>
__global__ void __launch_bounds__(256) fwd_combine_kernel(const FwdArgs a) {
  constexpr int kCols = D / 8, kSlot = kRowsPerCta * (D + 2);
  dependency_wait();
  const int group = blockIdx.x >> 3, plan = a.group_parts[group];      // (of no meaning where no such group was in the launch)
  const int n_split = plan & 0xffff, n_slots = plan >> 16;
  if (n_split <= 1) return;
  const int G = a.Hq / a.Hkv, g = group % a.Hkv, b = group / a.Hkv % a.B, n_rows = a.n_routed[b] * G;
  const int pi = (n_rows + kRowsPerCta - 1) / kRowsPerCta - 1 - group / a.Hkv / a.B, row0 = pi * kRowsPerCta;
  if (pi < 0) return;                  // no such group
  const int32_t* q_idx_b = a.q_idx + (int64_t)b * a.Lq;
  if (a.row_begin > 0 || a.row_end < a.Lq) {       // (as in attn_fwd_kernel, which then has written the group's word)
    const int t_last = q_idx_b[(min(row0 + kRowsPerCta, n_rows) - 1) / G];
    if (t_last < a.row_begin || t_last >= a.row_end) return;
  }
  const int r = (blockIdx.x & 7) * 32 + (threadIdx.x & 31), col = (threadIdx.x >> 5) * kCols;
  const int tile_row = row0 + r;
  if (tile_row >= n_rows) return;
  const int row = tile_row / G, h = g * G + (tile_row - row * G), seq_row = q_idx_b[row];
  if (!dbg_in_range(row < a.Lq && seq_row >= 0 && seq_row < a.Lq, a.status)) return;
  const float* parts = a.part + (size_t)group * n_slots * kSlot + (r / kTileM) * (kTileM * (D + 2)) + r % kTileM;
  bf16* dst2 = a.out2 + b * a.out2_st.b + seq_row * a.out2_st.t + (int64_t)h * D + col;
  uint4 old[kCols / 8];                // s_t
#pragma unroll
  for (int q = 0; q < kCols / 8; ++q)
    old[q] = a.accumulate_into_out2 || a.shared_window ? reinterpret_cast<const uint4*>(dst2)[q] : make_uint4(0, 0, 0, 0);
  // The loads of several parts in flight by arrays, not by the unrolling of a loop, which the compiler need not use for that: behind
  // the last part of 28 / of five / of eleven parts the kernel ends after 11.0 / 12.9 / 8.5 us, unrolled four times after 17.1 / 18.4 /
  // 10.6; with eight parts in flight instead of four the same.
  constexpr int kAhead = 4;
  float m = -INFINITY, least = 0.f, l = 0.f;
  for (int s0 = 0; s0 < n_split; s0 += 2 * kAhead) {
    float ls[2 * kAhead], ms[2 * kAhead];
#pragma unroll
    for (int u = 0; u < 2 * kAhead; ++u) {
      const float* p = parts + min(s0 + u, n_split - 1) * kSlot;
      ls[u] = p[kTileM * (D + 1)];
      ms[u] = p[kTileM * D];
    }
#pragma unroll
    for (int u = 0; u < 2 * kAhead; ++u) {
      least = fminf(least, ls[u]);
      if (ls[u] != 0.f) m = fmaxf(m, ms[u]);
    }
  }
  if (least < 0.f) return;             // a wait ran out in a part: nothing of the group is stored
  float f[kCols];
#pragma unroll
  for (int e = 0; e < kCols; ++e) f[e] = 0.f;
  const float* p0 = parts - r % kTileM + (col / 4 * kTileM + r % kTileM) * 4;
  for (int s0 = 0; s0 < n_split; s0 += kAhead) {
    float ls[kAhead], ms[kAhead];
    float4 v[kAhead][kCols / 4];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const int s = min(s0 + u, n_split - 1);
      ls[u] = s0 + u < n_split ? parts[s * kSlot + kTileM * (D + 1)] : 0.f;
      ms[u] = parts[s * kSlot + kTileM * D];
#pragma unroll
      for (int x = 0; x < kCols / 4; ++x) v[u][x] = *reinterpret_cast<const float4*>(p0 + s * kSlot + x * (4 * kTileM));
    }
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const bool any = ls[u] != 0.f;     // else no key of that part is visible to the row, and perhaps nothing was written
      const float w = any ? fast_exp2(ms[u] - m) : 0.f;
      l = fmaf(ls[u], w, l);
#pragma unroll
      for (int x = 0; x < kCols / 4; ++x) {
        f[4 * x] = any ? fmaf(w, v[u][x].x, f[4 * x]) : f[4 * x];
        f[4 * x + 1] = any ? fmaf(w, v[u][x].y, f[4 * x + 1]) : f[4 * x + 1];
        f[4 * x + 2] = any ? fmaf(w, v[u][x].z, f[4 * x + 2]) : f[4 * x + 2];
        f[4 * x + 3] = any ? fmaf(w, v[u][x].w, f[4 * x + 3]) : f[4 * x + 3];
      }
    }
  }
  float inv_l = l > 0.f ? 1.0f / l : 0.f, lse2 = m + log2f(l), c_loc = 0.f;
  if (a.shared_window) {             // (as in attn_fwd_kernel)
    const float lse_out2 = l > 0.f ? lse2 : -INFINITY;
    const float lse_loc2 = a.lse_loc[((int64_t)b * a.Hq + h) * a.Lq + seq_row] * 1.4426950408889634f;
    const float mm = fmaxf(lse_out2, lse_loc2);
    const float w_out = fast_exp2(lse_out2 - mm), w_loc = fast_exp2(lse_loc2 - mm);
    const float inv = 1.0f / (w_out + w_loc);
    inv_l *= w_out * inv;
    c_loc = w_loc * inv;
    lse2 = mm + log2f(w_out + w_loc);
  }
  if (col == 0 && a.lse != nullptr) a.lse[((int64_t)b * a.Hq + h) * a.Lq + row] = lse2 * 0.6931471805599453f;
  bf16* dst1 = a.out ? a.out + b * a.out_st.b + row * a.out_st.t + (int64_t)h * D + col : nullptr;
#pragma unroll
  for (int q = 0; q < kCols / 8; ++q) {
    const uint32_t ow[4] = {old[q].x, old[q].y, old[q].z, old[q].w};
    uint32_t u[4], v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float s0 = __uint_as_float(ow[k] << 16), s1 = __uint_as_float(ow[k] & 0xffff0000u);       // s_t
      float f0 = f[8 * q + 2 * k] * inv_l, f1 = f[8 * q + 2 * k + 1] * inv_l;
      if (a.shared_window) { f0 = fmaf(c_loc, s0, f0); f1 = fmaf(c_loc, s1, f1); }
      u[k] = pack_bf16(f0, f1);
      v[k] = a.accumulate_into_out2 ? pack_bf16(f0 + s0, f1 + s1) : u[k];
    }
    if (dst1) reinterpret_cast<uint4*>(dst1)[q] = make_uint4(u[0], u[1], u[2], u[3]);
    reinterpret_cast<uint4*>(dst2)[q] = make_uint4(v[0], v[1], v[2], v[3]);
  }
}

template <int D>
cudaError_t launch_fwd(const FwdArgs& a, int64_t grid, const CUtensorMap& mapQ, const CUtensorMap& mapK, const CUtensorMap& mapV,
                       const CUtensorMap& mapOut, const CUtensorMap& mapOut2, int64_t groups, cudaStream_t stream) {
  static PerDeviceOnce once;
  cudaError_t e = once.run([] {
    return cudaFuncSetAttribute(attn_fwd_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, FwdSmem<D>::kTotal);
  });
  if (e != cudaSuccess) return e;
  e = launch_dependent(attn_fwd_kernel<D>, dim3((unsigned)grid), kFwdThreads, FwdSmem<D>::kTotal, stream, a.overlap != 0, mapQ,
                       mapK, mapV, mapOut, mapOut2, a);
  if (e != cudaSuccess || a.part == nullptr || longest_group(a) < kMinSplitBlocks) return e;     // nothing is split
  return launch_dependent(fwd_combine_kernel<D>, dim3((unsigned)(8 * std::min<int64_t>(groups, kSplitGroups))), 256, 0, stream,
                          a.overlap != 0, a);
}

}  // namespace

cudaError_t launch_attn_fwd(const FwdArgs& a, const CUtensorMap& mapQ, const CUtensorMap& mapK,
                            const CUtensorMap& mapV, const CUtensorMap& mapOut, const CUtensorMap& mapOut2,
                            cudaStream_t stream) {
  if (a.pair_end <= a.pair_begin) return cudaSuccess;
  int64_t grid = (int64_t)(a.pair_end - a.pair_begin) * a.Hq * a.B;
  if (a.global_mode && !a.all_rows) grid = compact_groups(a.Lq, a.Hq / a.Hkv) * a.Hkv * a.B;
  const int64_t groups = grid;
  if (a.part != nullptr) grid = std::max(grid, std::min<int64_t>(grid * kMaxKeySplit, kSplitItems));
  // Local launches of more items than SMs take CTAs that process one item after the other, at any window: attn_fwd_local.cu
  // has both sides from W = 0 to 4096.  Global ones do not: with the same loop 32K tokens took 1267 instead of 1256 us, 4001
  // tokens 66 instead of 62, 2000 tokens on 34K keys 328 instead of 303.
  const DeviceInfo* dev = device_info();
  if (dev == nullptr) return cudaErrorUnknown;
  if (!a.global_mode && a.D == 128 && grid > dev->sms)
    return launch_attn_fwd_local(a, grid, mapQ, mapK, mapV, mapOut, mapOut2, stream);
  return a.D == 128 ? launch_fwd<128>(a, grid, mapQ, mapK, mapV, mapOut, mapOut2, groups, stream)
                    : launch_fwd<64>(a, grid, mapQ, mapK, mapV, mapOut, mapOut2, groups, stream);
}

}  // namespace l2a
