// Backward of the layer for sm_100a.
//
// The paper states only that the backward computes gradients for active queries and reuses L_c and
// Q_idx (Section 3.2); the arithmetic is the vector-Jacobian product of the forward with the routing
// mask fixed.  For each attention X in {local, global}, with P = exp(scale*q.k - lse_X):
//     Delta_i = dO_i . out_X,i      dP_ij = dO_i . v_j      dS_ij = P_ij (dP_ij - Delta_i)
//     dV_j += P_ij dO_i             dK_j += scale dS_ij q_i  dQ_i += scale dS_ij k_j
// where "global" rows are the routed rows only.
//
// Kernels
//   bwd_delta_kernel : Delta_loc (all rows), Delta_glb (compact rows), optional dgate.  HBM bound.
//   dq_zero_kernel   : clears the fp32 dQ accumulators (where they are small CTAs of bwd_delta_kernel do).
//   bwd_kernel       : key/value-stationary, five GEMMs per (query tile, key block) pair.  One CTA owns a block of
//                      128 keys of one KV head and walks every query tile that can see it -- local band tiles of
//                      the G query heads, then the compact routed tiles from the first one at or after the block.
//                      dK, dV accumulate in TMEM (no atomics, one bf16 store); the scores are built transposed (keys
//                      on TMEM lanes) so that P^T feeds dV straight from TMEM; dQ(i) = dS(i) K is a fresh tile per
//                      item that dedicated read-out warps add into fp32 accumulators in global memory.
//   dq_merge_kernel  : dQ = scale * (local accumulator + routed rows' global accumulator), rounded to bf16 once.
#include "l2a_common.cuh"
#include "sm100_prims.cuh"

namespace l2a {

namespace {

constexpr int kBoxBytes = 128 * 128;
constexpr float kLog2e = 1.4426950408889634f;

// ------------------------------------------------------------------------------------------------
// Delta / dgate preprocess.  The grid is one resident wave; the warps take the tokens round-robin, so that at any
// moment the whole grid reads one contiguous stretch of each tensor (a contiguous range per warp, i.e. thousands of
// separate streams, ran at 0.7 of this speed).  A token's Hq*D values are read with 16-byte loads: D/8 lanes per
// head, 32/(D/8) heads per pass, four passes in flight: with the rows of two groups of passes in registers two CTAs fit an
// SM (held to three or four they spill: 70 / 71 us instead of 59 beside a concurrent clearing, 2 x 4096 tokens).  The kernel
// reads nothing that the gather ahead of it writes, so it waits for that at its end only.  From the gather to the end of the
// clearing: 2 x 4096 tokens (28/4 heads) 90 -> 75 us, 16K tokens 121 -> 114, 64K packed (32/8) 546 -> 516; with a gradient of
// its own for the local output, whose rows are those asked for ahead and not dO's, 92 -> 81, 140 -> 128 and (64K) 581 -> 545; of
// the global part alone 50 -> 29, 68 -> 42 and 219 -> 115.  Clearing beside Delta instead of behind it (one gradient): 69, 115
// and 600 (DRAM turns between reads and writes).
__device__ __forceinline__ float dot8(const uint4& x, const uint4& y) {
  const uint32_t a[4] = {x.x, x.y, x.z, x.w}, b[4] = {y.x, y.y, y.z, y.w};
  float acc = 0.f;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    acc = fmaf(__uint_as_float(a[k] << 16), __uint_as_float(b[k] << 16), acc);
    acc = fmaf(__uint_as_float(a[k] & 0xffff0000u), __uint_as_float(b[k] & 0xffff0000u), acc);
  }
  return acc;
}

// CTA `cta` of n_ctas zeroes its share of the fp32 dQ accumulators: every row tile of the local one, the compact tiles in use of
// the global one.
__device__ __forceinline__ void zero_accumulators(float* acc_loc, float* acc_glb, const int32_t* n_routed, int B, int Hq, int Hkv,
                                                  int L, int tile_floats, int cta, int n_ctas) {
  const int n_tiles = (L + kTileM - 1) / kTileM, n_ctiles = compact_tiles(L, Hq / Hkv);
  const int per = B * Hq * n_tiles;
  for (int item = cta; item < per + B * Hkv * n_ctiles; item += n_ctas) {
    const int which = item >= per, rem = which ? item - per : item;
    float* base = which ? acc_glb : acc_loc;
    if (base == nullptr) continue;
    if (which && rem % n_ctiles >= compact_tiles(n_routed[rem / (n_ctiles * Hkv)], Hq / Hkv)) continue;
    float4* p = reinterpret_cast<float4*>(base + (int64_t)rem * tile_floats);
    for (int k = threadIdx.x; k < tile_floats / 4; k += blockDim.x) p[k] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

// What the CTAs behind the first n_delta do: the accumulators are cleared by the Delta kernel itself where they are small.
struct ZeroArgs {
  int n_delta;
  float *acc_loc, *acc_glb;
  const int32_t* n_routed;
  int Hkv;
};

template <int D>
__global__ void __launch_bounds__(256, 2) bwd_delta_kernel(const bf16* __restrict__ dO, const bf16* __restrict__ dO_loc,
                                                        const bf16* __restrict__ S,
                                                        const bf16* __restrict__ A_c,
                                                        const uint8_t* __restrict__ d_mask,
                                                        const int32_t* __restrict__ prefix, float* __restrict__ delta_loc,
                                                        float* __restrict__ delta_glb, float* __restrict__ dgate, int B,
                                                        int L, int Hq, int a_by_row, int64_t do_bs, int64_t do_ts,
                                                        const float* __restrict__ lse_loc,
                                                        const float* __restrict__ lse_glb, float* __restrict__ lse_eff,
                                                        const ZeroArgs z) {
  constexpr int kLanesPerHead = D / 8;                 // 16-byte chunks per head row
  constexpr int kHeadsPerPass = 32 / kLanesPerHead;
  const int lane = threadIdx.x & 31;
  const int64_t n_tokens = (int64_t)B * L;
  const int64_t n_warps = (int64_t)z.n_delta * (blockDim.x >> 5);
  const int64_t gw = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (S == nullptr) dO_loc = dO;                       // local part skipped: its gradient is not read
  const bool split = dO_loc != dO;                     // separate gradient for the local output
  dependents_release();       // (reads nothing that the kernels ahead of it in the call write: it waits at its end)
  if ((int)blockIdx.x >= z.n_delta) {
    zero_accumulators(z.acc_loc, z.acc_glb, z.n_routed, B, Hq, z.Hkv, L, kTileM * D, blockIdx.x - z.n_delta,
                      gridDim.x - z.n_delta);
    dependency_wait();
    return;
  }
  const int sub = lane / kLanesPerHead;                // head inside the pass
  const int n_pass = (Hq + kHeadsPerPass - 1) / kHeadsPerPass;
  const bool global = d_mask != nullptr;               // NULL: the global part is skipped
  bool next_routed = global && gw < n_tokens && d_mask[gw] != 0;
  int next_c = global && gw < n_tokens ? prefix[gw / L * (L + 1) + gw % L] : 0;
  for (int64_t token = gw; token < n_tokens; token += n_warps) {
    const int b = (int)(token / L), t = (int)(token % L);
    const bool routed = next_routed;
    const int c = next_c;
    if (global && token + n_warps < n_tokens) {        // the next token's routing, ahead of this one's rows
      const int64_t n = token + n_warps;
      next_routed = d_mask[n] != 0;
      next_c = prefix[n / L * (L + 1) + n % L];
    }
    // a_by_row: the global output was computed for every token and A is indexed by row (forced-global iterations)
    const bool with_a = routed || a_by_row;
    if (S == nullptr && !with_a) {                     // local part skipped, and no global part of this token
      if (dgate != nullptr && lane == 0) dgate[token] = 0.f;
      continue;
    }
    const int64_t row = token * Hq * D;                          // S: dense
    const int64_t orow = b * do_bs + t * do_ts;                  // dO, dO_loc: the strides of O
    const int64_t crow = ((int64_t)b * L + (a_by_row ? t : c)) * Hq * D;
    const uint4* po = reinterpret_cast<const uint4*>(dO + orow) + lane;
    const uint4* pl = reinterpret_cast<const uint4*>(dO_loc + orow) + lane;
    const uint4* ps = reinterpret_cast<const uint4*>(S + row) + lane;
    const uint4* pa = reinterpret_cast<const uint4*>(A_c + crow) + lane;
    float gate = 0.f;
    // shared-window statistics: the two log-sum-exps of head (32 j + lane), fetched ahead of the passes that need them
    float pre_loc[2] = {0.f, 0.f}, pre_glb[2] = {0.f, 0.f};
    if (lse_eff != nullptr) {
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int h = 32 * j + lane;
        if (h < Hq) {
          pre_loc[j] = __ldg(&lse_loc[((int64_t)b * Hq + h) * L + t]);
          if (routed) pre_glb[j] = __ldg(&lse_glb[((int64_t)b * Hq + h) * L + c]);
        }
      }
    }
    // The rows of one group of passes are asked for before those of the group ahead are reduced: the shuffles of a group
    // otherwise stand between its loads and the next group's.
    constexpr int kGroup = 2;
    struct Rows { uint4 l[kGroup], s[kGroup], a[kGroup]; } cur, nxt;      // dO_loc, S, A
    auto fetch = [&](int p0, Rows& x) {
#pragma unroll
      for (int i = 0; i < kGroup; ++i) {
        const int p = p0 + i;
        if (p < n_pass && p * kHeadsPerPass + sub < Hq) {
          x.l[i] = __ldg(pl + p * 32);
          if (S != nullptr) x.s[i] = __ldg(ps + p * 32);
          if (with_a) x.a[i] = __ldg(pa + p * 32);
        }
      }
    };
    fetch(0, cur);
    for (int p0 = 0; p0 < n_pass; p0 += kGroup) {
      fetch(p0 + kGroup, nxt);
#pragma unroll
      for (int i = 0; i < kGroup; ++i) {
        const int h = (p0 + i) * kHeadsPerPass + sub;
        float dl = 0.f, dg = 0.f;
        if (p0 + i < n_pass && h < Hq) {
          if (S != nullptr) dl = dot8(cur.l[i], cur.s[i]);      // NULL: local part skipped
          if (with_a) dg = dot8(split ? __ldg(po + (p0 + i) * 32) : cur.l[i], cur.a[i]);
        }
#pragma unroll
        for (int off = kLanesPerHead / 2; off > 0; off >>= 1) {
          dl += __shfl_xor_sync(0xffffffffu, dl, off);
          dg += __shfl_xor_sync(0xffffffffu, dg, off);
        }
        // (every lane takes part in the shuffles; heads beyond 64 fall back to loads in place)
        float pre_l = __shfl_sync(0xffffffffu, (h & 32) ? pre_loc[1] : pre_loc[0], h & 31);
        float pre_g = __shfl_sync(0xffffffffu, (h & 32) ? pre_glb[1] : pre_glb[0], h & 31);
        if (p0 + i < n_pass && h < Hq && (lane % kLanesPerHead) == 0) {
          const int64_t it = ((int64_t)b * Hq + h) * L + t, ic = ((int64_t)b * Hq + h) * L + c;
          if (lse_eff != nullptr && h >= 64) {
            pre_l = lse_loc[it];
            pre_g = routed ? lse_glb[ic] : 0.f;
          }
          float dl_out = dl;
          if (lse_eff != nullptr) {
            // Shared-window backward.  Inside the window of a routed row P_glb = beta * P_loc with
            // beta = exp(lse_loc - lse_glb), and dP is the same product dO V^T for both modules, so the two
            // contributions add up to P' (dP - Delta') with P' = (1 + beta) P_loc and
            // Delta' = (Delta_loc + beta * Delta_glb) / (1 + beta): the local items carry them with these statistics.
            float le = pre_l;
            if (routed) {
              const float beta = __expf(le - pre_g);
              dl_out = (dl + beta * dg) / (1.0f + beta);
              le -= log1pf(beta);
            }
            lse_eff[it] = le;
          }
          if (S != nullptr) delta_loc[it] = dl_out;
          if (routed) delta_glb[ic] = dg;
          gate += dg;
        }
      }
      cur = nxt;
    }
    if (dgate != nullptr) {
#pragma unroll
      for (int off = 16; off >= kLanesPerHead; off >>= 1) gate += __shfl_xor_sync(0xffffffffu, gate, off);
      if (lane == 0) dgate[token] = with_a ? gate : 0.f;
    }
  }
  dependency_wait();
}

// lse by row -> lse by compact row (forced-global iterations store the global log-sum-exp for every row)
__global__ void __launch_bounds__(256) compact_stat_kernel(const float* __restrict__ by_row, float* __restrict__ by_c,
                                                           const int32_t* __restrict__ q_idx,
                                                           const int32_t* __restrict__ n_routed, int L, int Hq) {
  const int b = blockIdx.z, h = blockIdx.y;
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  dependency_wait();
  dependents_release();
  if (c < n_routed[b]) {
    const int64_t base = ((int64_t)b * Hq + h) * L;
    by_c[base + c] = by_row[base + q_idx[(int64_t)b * L + c]];
  }
}

// ------------------------------------------------------------------------------------------------
struct BwdArgs {
  int B, Lq, Lk, Hq, Hkv, D, G;      // G = Hq / Hkv
  uint32_t g_inv;                    // ceil(2^31 / G)
  int window, q_pos_offset;
  float scale, scale_log2;
  int skip_local, skip_global;   // gradients of one module only (the other module has its own Q/K/V)
  int kb_begin, kb_count;        // key blocks [kb_begin, kb_begin + kb_count) of every KV head
  int kb_outermost;              // launch order: key blocks outermost (1) or KV heads outermost (0)
  RowStrides dq_st, dk_st, dv_st;   // strides of the gradient tensors in elements
  float* dq_acc_loc;             // fp32 dQ accumulators (layout: see bwd_kernel), by row tile
  float* dq_acc_glb;             //                 and by compact tile; NULL when that module is skipped
  int vis_shift;                 // global items see the keys 0 .. pos - vis_shift: 0, or W + 1 when the window's share of
                                 // the global gradient is carried by the local items (shared-window backward)
  const int32_t* q_idx;
  const int32_t* n_routed;
  const int32_t* prefix;
  const int32_t* seq_bounds;   // packed sequences (B == 1): per token {first token of its sequence, one past the last}
  const float* lse_loc;    // [B,Hq,Lq] by row
  const float* lse_glb;    // [B,Hq,Lq] by compact row
  const float* delta_loc;  // same indexing
  const float* delta_glb;
  bf16* dQ;
  bf16* dK;
  bf16* dV;
  int* status;
};

// ================================================================================================
// Thread roles of the tensor-core kernel below:
//   warps 0-15 : compute.  Warp w owns TMEM lanes 32*(w%4)..+31 (its thread's key, or query row of dQ) and the
//                32 score columns of quarter w/4, so that 16 warps hide each other's TMEM and MUFU latency.
//   warp 16    : TMA producer          warp 17 : tcgen05 MMA issuer, TMEM owner
//   warp 18    : stages the row statistics of each query tile          warp 19 : idle
//   warps 20-27: read every dQ(i) tile out of TMEM (one lane group and one half of the columns each) and add it into the
//                fp32 accumulators: the reductions leave an SM at about 32 bytes per clock, and a warp that issues them
//                stalls that long, so they are kept off the warps whose progress the tensor pipe waits for.  A read-out
//                warp takes its whole share (64 values per thread) into registers and releases the TMEM columns before
//                its first reduction.
// Registers: 896 threads start with 72 each (64512 in all, which is also all that setmaxnreg can redistribute: an
// increase is served from what the CTA's own warps released); the service warpgroup goes down to 40, the read-out
// warpgroups stay at 72, the compute warpgroups go up to 80 -- which they fit because scores and dP^T leave TMEM sixteen
// columns at a time.
constexpr int kComputeWarps = 16;
constexpr int kDkvThreads = 28 * 32;   // 896

__device__ __forceinline__ float bf16lo_to_f32(uint32_t packed) { return __uint_as_float(packed << 16); }
__device__ __forceinline__ float bf16hi_to_f32(uint32_t packed) { return __uint_as_float(packed & 0xffff0000u); }

struct ItemPlan {
  int loc_t0, loc_nt;   // first local query tile, number of local tiles
  int glb_t0, glb_nt;   // first compact tile, number of compact tiles (the group's heads packed into their rows)
  int total;            // items of the key block: loc_nt * G + glb_nt
};

// First tile at or after t0 that CTA `rank` of kSplit takes for head hg of the group: (tile + hg) % kSplit == rank.  By tile
// and not by position in the item list, so that more query tiles behind a sequence (padding rows) leave the sums of dK
// and dV as they are; shifted by the head, so that the shares are even.  (Compact tiles: hg = 0.)
template <int kSplit>
__device__ __forceinline__ int first_tile(int t0, int hg, int rank) {
  return kSplit == 1 ? t0 : t0 + ((rank - t0 - hg) & (kSplit - 1));
}
template <int kSplit>
__device__ __forceinline__ int share_count(const ItemPlan& p, int G, int rank) {
  if (kSplit == 1) return p.total;
  int n = (max(0, p.glb_t0 + p.glb_nt - first_tile<kSplit>(p.glb_t0, 0, rank)) + kSplit - 1) / kSplit;
  for (int hg = 0; hg < G; ++hg)
    n += (max(0, p.loc_t0 + p.loc_nt - first_tile<kSplit>(p.loc_t0, hg, rank)) + kSplit - 1) / kSplit;
  return n;
}

__device__ __forceinline__ ItemPlan make_plan(const BwdArgs& a, int b, int k0, int span = kTileN) {
  ItemPlan p;
  const int G = a.G;
  // packed sequences: no row at or after the end of the sequence that holds the block's last key sees any of its keys
  int row_end = a.Lq;
  if (a.seq_bounds != nullptr) {
    const int k_last = min(k0 + span, a.Lk) - 1;
    row_end = max(0, min(a.Lq, a.seq_bounds[2 * k_last + 1]));
  }
  // local: rows t with position in [k0, k0 + span - 1 + W]
  int tmin = k0 - a.q_pos_offset;
  const long long tmax_ll = (long long)k0 + span - 1 + a.window - a.q_pos_offset;
  int tmax = tmax_ll > row_end - 1 ? row_end - 1 : (int)tmax_ll;
  if (tmin < 0) tmin = 0;
  if (tmax < tmin || a.skip_local) { p.loc_t0 = 0; p.loc_nt = 0; }
  else { p.loc_t0 = tmin / kTileM; p.loc_nt = tmax / kTileM - p.loc_t0 + 1; }
  // global: compact rows whose last visible key (position - vis_shift) is >= k0
  const int n_c = a.skip_global ? 0 : a.n_routed[b];
  long long tmin_g = (long long)k0 - a.q_pos_offset + a.vis_shift;
  if (tmin_g < 0) tmin_g = 0;
  if (tmin_g > row_end - 1 || n_c == 0) { p.glb_t0 = 0; p.glb_nt = 0; }
  else {
    const int r_min = a.prefix[(int64_t)b * (a.Lq + 1) + (int)tmin_g] * G;
    const int r_end = (row_end < a.Lq ? min(n_c, a.prefix[(int64_t)b * (a.Lq + 1) + row_end]) : n_c) * G;
    if (r_min >= r_end) { p.glb_t0 = 0; p.glb_nt = 0; }
    else { p.glb_t0 = r_min / kTileM; p.glb_nt = (r_end - 1) / kTileM - p.glb_t0 + 1; }
  }
  p.total = p.loc_nt * G + p.glb_nt;
  return p;
}

// Walks the items of a CTA in order without divisions: the local tiles of one head after the other, then the compact tiles.
// The plan stays in shared memory and is looked at only where a head ends: the read-out warps have no registers to spare.
template <int kSplit>
struct ItemCursor {
  int hg = -1, t = 0, left = 0;      // head of the group (G: compact tiles), tile, tiles of the share left in this head
  __device__ __forceinline__ void settle(const ItemPlan& p, int G, int rank) {    // a head may hold no tile of the share
    while (left <= 0 && hg < G) {
      const bool glb = ++hg == G;
      const int t0 = glb ? p.glb_t0 : p.loc_t0, nt = glb ? p.glb_nt : p.loc_nt;
      t = first_tile<kSplit>(t0, glb ? 0 : hg, rank);
      left = kSplit == 1 ? nt : (t0 + nt - t + kSplit - 1) / kSplit;
    }
  }
  __device__ __forceinline__ void next(const ItemPlan& p, int G, int rank) {
    t += kSplit;
    if (--left <= 0) settle(p, G, rank);
  }
};

// ================================================================================================
// Five-GEMM backward kernel: the key/value-stationary kernel above plus the fifth GEMM, dQ(i) = dS(i) K, so that
// S and dP are computed once per tile pair.  dQ(i) is a fresh 128 x D accumulator per item; the read-out warps take
// it out (lane = query row) and add it into an fp32 accumulator in global memory whose layout is private to this
// file: per (batch, head, 128-row tile) one block of 128 x D floats ordered [warp 16][piece D/16][lane 32][4] (the lanes of the
// compact tiles ordered by head: head_slot), so
// that every red.global.add.v4.f32 of a warp covers 512 contiguous bytes.  Local items add into the accumulator
// indexed by row tile, global items into the one indexed by compact tile; dq_merge_kernel forms the bf16 dQ.
// All key blocks meet in those accumulators in no fixed order: dQ is not bit-reproducible from run to run
// (dK, dV are).
//   TMEM: dV [0,D) | dK [D,2D) | T [256,384): S^T(i), then P^T(i) (bf16, quarter-local) | U [384,512): dP^T(i),
//         then dS^T(i) (bf16, quarter-local), then dQ(i).
//   Shared memory: K, V resident; Q and dO in two-stage rings; dS(i) (bf16, [key][query], swizzled like a TMA
//   tile) -- the A operand of dQ = dS K (read MN-major).
//   MMA order per item i:  dV(i) | S^T(i+1) | dK(i) | dQ(i) | dP^T(i+1).  S^T(i+1) does not depend on dS(i), so it is
//   issued ahead of the wait for it: the compute warps find the next scores ready when they are done with dS(i).
//   Two loops run through the order: T: S^T -> P -> dV -> S^T and U: dP^T -> dS -> dQ -> read-out -> dP^T.  What bounds an
//   item is the traffic of shared memory (operands 2048 clk, TMA 512, dS, statistics and the reductions' data 1000 at 128
//   bytes a clock), not the tensor pipe: so dK(i) takes dS^T from U, where it lies between dP^T(i) and dQ(i), and not from
//   shared memory as before, although nothing then covers the read-out of dQ(i) that dP^T(i+1) waits for.  It also returns
//   the Q stage to the TMA warp 500 clk earlier, whose load was late under the reductions.  Backward launch of 2 x 4096
//   tokens (28/4 heads) 794 -> 758 us, of the local module at 8155 tokens 1037 -> 978; without the writes of dS it would
//   take 685, without the TMA writes 694, without the statistics 732, without any of them and the reductions 560.

// Where row `lane` of 32 packed rows lies in a piece of the compact accumulator: the rows of one head next to each other, so
// that the merge, which reads the rows of one head, finds them in whole sectors.  (In the order of the rows the merge took, with
// 32/8 heads, 1587 tokens 27 us instead of 17, 2 x 4096 tokens (28/4) 50 instead of 42.)
__device__ __forceinline__ int head_slot(int lane, int G) {
  const int q = lane % G, n = lane / G, per = 32 / G;
  return q * per + min(q, 32 - per * G) + n;
}

// The reductions of one read-out warp: piece I of its 32 x D/2 share (4 columns each) goes to a byte offset from the
// warp's base address that is a compile-time constant, so that all of them share one address register pair.
template <int kBytes>
__device__ __forceinline__ void red_add_v4(float* base, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("red.global.add.v4.f32 [%0+%5], {%1, %2, %3, %4};" ::"l"(base), "f"(__uint_as_float(a)),
               "f"(__uint_as_float(b)), "f"(__uint_as_float(c)), "f"(__uint_as_float(d)), "n"(kBytes)
               : "memory");
}
// Least distance between two reductions of a read-out warp, in SM clocks (polled: a sleep has steps of 64 ns), sixteen an item with
// D = 128, eight with D = 64.  Passes one after the other, at the board's power limit:
//   D = 128: 64K tokens / whole layer at 8155 tokens / 2 x 4096 tokens: 16 clk 22830 / 2074 us / -, 56 22430 / 2055 / -, 96 22180 /
//   2020 / -, 112 22260 / 2027 / 1289, 128 22050 / 2000 / 1277, 144 21960 / 2011 / 1273, 168 22510 / 2060 / 1299, 200 23310 / 2115 /
//   1341; on another day 112 22560 / 2055 / 1307, 128 22420 / 2035 / 1293, 136 22380 / 2038 / 1291, 144 22340 / 2034 / 1294.
//   D = 64, 16384 tokens with 4/4 / 12/2 heads: 16 clk 514 / 1480 us, 64 515 / 1483, 88 516 / 1484, 112 518 / 1498, 136 522 / 1503.
template <int D>
constexpr uint32_t kRedSpacingClk = D == 128 ? 136 : 64;
template <int D, int I>
struct ReadOutReds {
  static constexpr int kCols = D / 4;                 // columns per quarter of the accumulator layout
  static constexpr int kCol = 4 * I;                  // relative to the warp's first column
  static constexpr int kOff = ((kCol / kCols) * 4 * (8 * D) + ((kCol % kCols) / 4) * 128) * 4;
  __device__ __forceinline__ static void run(float* base, const uint32_t (&v)[D / 64][32]) {
    // spaced out: reductions issued back to back fill the queue of the memory pipe, and the compute warps' shared-memory
    // loads and stores (row statistics, dS) wait behind them; the read-out warps have most of an item's time to spare
    { const uint32_t t0 = clock(); while ((uint32_t)clock() - t0 < kRedSpacingClk<D>) { } }
    red_add_v4<kOff>(base, v[I / 8][4 * (I % 8)], v[I / 8][4 * (I % 8) + 1], v[I / 8][4 * (I % 8) + 2],
                     v[I / 8][4 * (I % 8) + 3]);
    ReadOutReds<D, I + 1>::run(base, v);
  }
};
template <int D>
struct ReadOutReds<D, D / 8> {
  __device__ __forceinline__ static void run(float*, const uint32_t (&)[D / 64][32]) {}
};

// threadIdx.x, read anew
__device__ __forceinline__ uint32_t thread_index() {
  uint32_t t;
  asm volatile("mov.u32 %0, %%tid.x;" : "=r"(t));
  return t;
}

template <int D>
struct BwdSmem {
  static constexpr int kTileBytes = 128 * D * 2;
  static constexpr int kKOff = 0;
  static constexpr int kVOff = kTileBytes;
  static constexpr int kQOff = 2 * kTileBytes;                 // 2 stages
  static constexpr int kDoOff = kQOff + 2 * kTileBytes;        // 2 stages
  static constexpr int kDsOff = kDoOff + 2 * kTileBytes;       // dS: 128 keys x 128 queries bf16
  static constexpr int kStatOff = kDsOff + 128 * 128 * 2;
  static constexpr int kStatSlot = (2 * 128 + 8) * 4;
  static constexpr int kBarOff = kStatOff + 2 * kStatSlot;
  static constexpr int kTotal = kBarOff + 256;
};
struct BwdBarriers {
  uint64_t kv_full;
  uint64_t q_full[2], q_empty[2];
  uint64_t do_full[2], do_empty[2];
  uint64_t st_full[2], st_empty[2];
  uint64_t s_full, dp_full, p_full, ds_full, ds_free, dq_full, u_free, final_bar;
  ItemPlan plan;
  int b, g, k0, n_c, count;   // batch entry, KV head, first key, routed rows, items of this CTA
  uint32_t tmem_base;
  int abort_flag;
};
static_assert(sizeof(BwdBarriers) <= 256, "barrier block");

// Which of the 32 query rows col0 .. col0 + 31 (sequence rows, or packed compact rows of a global item) attend to key kp, as a
// bit mask.  The first row is the one at the key's own position -- for a global item the first routed row whose last
// visible key is not before it, which the exclusive prefix gives -- and the last one ends the window or the sequence.
__device__ __forceinline__ uint32_t visible_columns(const BwdArgs& a, int b, int n_c, int kp, int glb, int col0) {
  int row_end = a.Lq;
  if (a.seq_bounds != nullptr) row_end = kp < a.Lq ? max(0, min(a.Lq, __ldg(&a.seq_bounds[2 * kp + 1]))) : 0;
  long long first = (long long)kp - a.q_pos_offset + (glb ? a.vis_shift : 0);
  first = first < 0 ? 0 : first > a.Lq ? a.Lq : first;
  if (glb) {
    const int32_t* prefix = a.prefix + (int64_t)b * (a.Lq + 1);
    const int c_end = row_end < a.Lq ? min(n_c, __ldg(&prefix[row_end])) : n_c;
    return bit_range(__ldg(&prefix[(int)first]) * a.G - col0, c_end * a.G - col0);
  }
  const long long last = (long long)kp + a.window - a.q_pos_offset + 1;
  return bit_range((int)first - col0, (last < row_end ? (int)last : row_end) - col0);
}

// Byte offset in the rings of row kr of quarter q in slot `slot` of its owner; the 16-byte pieces of a row lie 128 rows
// apart, so that a warp's accesses are contiguous.  kSplit - 1 slots of 4 / kSplit quarters of 128 x D / 2 floats.
template <int D, int kSplit>
__device__ __forceinline__ uint32_t dkv_slot_offset(int slot, int q, int kr) {
  return (slot * (4 / kSplit) + q % (4 / kSplit)) * (128 * (D / 2) * 4) + kr * 16;
}

template <int D, int kSplit>
__device__ __forceinline__ void send_dkv(uint32_t dst, uint32_t taddr, bool own) {
#pragma unroll
  for (int c = 0; c < D / 64; ++c) {
    uint32_t v[32];
    if (own) {
      tmem_ld32(taddr + c * 32, v);
      tmem_ld_wait();
    } else {
#pragma unroll
      for (int e = 0; e < 32; ++e) v[e] = 0u;
    }
#pragma unroll
    for (int x = 0; x < 8; ++x)
      cluster_st128(dst + (c * 8 + x) * (128 * 16), v[4 * x], v[4 * x + 1], v[4 * x + 2], v[4 * x + 3]);
  }
}

// One quarter of (dV | dK): accumulator (plus the other CTAs' shares of a cluster) to bf16.  own: this CTA had items.
template <int D, int kSplit>
__device__ __forceinline__ void store_dkv(const BwdArgs& a, const uint8_t* smem, uint32_t taddr, bool own, int b, int g,
                                          int kp, int q, int kr) {
  static_assert((kSplit - 1) * (4 / kSplit) * 128 * (D / 2) * 4 <= 4 * BwdSmem<D>::kTileBytes, "slots exceed the rings");
  const bool valid = kp < a.Lk;
  const int which = q >> 1, half = q & 1;
  const RowStrides st = which == 0 ? a.dv_st : a.dk_st;
  bf16* dst = (which == 0 ? a.dV : a.dK) + b * st.b + (valid ? kp : 0) * st.t + (int64_t)g * D + half * (D / 2);
  const float mul = which == 0 ? 1.0f : a.scale;
#pragma unroll
  for (int c = 0; c < D / 64; ++c) {
    uint32_t v[32];
    if (own) {
      tmem_ld32(taddr + c * 32, v);
      tmem_ld_wait();
    } else {
#pragma unroll
      for (int e = 0; e < 32; ++e) v[e] = 0u;
    }
#pragma unroll
    for (int s = 0; s < kSplit - 1; ++s) {
      const uint32_t src = smem_u32(smem + BwdSmem<D>::kQOff) + dkv_slot_offset<D, kSplit>(s, q, kr) + c * 8 * (128 * 16);
#pragma unroll
      for (int x = 0; x < 8; ++x) {
        const float4 f = lds128(src + x * (128 * 16));
        v[4 * x] = __float_as_uint(__uint_as_float(v[4 * x]) + f.x);
        v[4 * x + 1] = __float_as_uint(__uint_as_float(v[4 * x + 1]) + f.y);
        v[4 * x + 2] = __float_as_uint(__uint_as_float(v[4 * x + 2]) + f.z);
        v[4 * x + 3] = __float_as_uint(__uint_as_float(v[4 * x + 3]) + f.w);
      }
    }
    if (valid) {
      uint4* d4 = reinterpret_cast<uint4*>(dst + c * 32);
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        float f[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) f[e] = __uint_as_float(v[8 * x + e]) * mul;
        d4[x] = make_uint4(pack_bf16(f[0], f[1]), pack_bf16(f[2], f[3]), pack_bf16(f[4], f[5]), pack_bf16(f[6], f[7]));
      }
    }
  }
}

// kSplit > 1: the kSplit CTAs of a cluster share one key block.  Each walks its part of the items, and at the end every
// CTA sums one part of the columns of (dV | dK) over the cluster through distributed shared memory.
template <int D, int kSplit>
__global__ void __launch_bounds__(kDkvThreads, 1)
bwd_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapDO,
               const __grid_constant__ CUtensorMap mapQc, const __grid_constant__ CUtensorMap mapDOc,
               const __grid_constant__ CUtensorMap mapK, const __grid_constant__ CUtensorMap mapV, const BwdArgs a) {
  using SM = BwdSmem<D>;
  constexpr int kKSteps = D / 16;
  // Key blocks ascending: most work first.  KV heads outermost lets the CTAs that run together share query tiles in L2;
  // key blocks outermost starts the heaviest blocks of every head first, which a launch of few waves needs.
  dependency_wait();
  dependents_release();
  const int rank = kSplit > 1 ? (int)cluster_rank() : 0;
  const int work = blockIdx.x / kSplit, heads = a.B * a.Hkv;
  const int j = a.kb_begin + (a.kb_outermost ? work / heads : work % a.kb_count);
  const int rest = a.kb_outermost ? work % heads : work / a.kb_count;
  const int b = rest % a.B;
  const int g = rest / a.B;
  const int k0 = j * kTileN;
  const ItemPlan plan = make_plan(a, b, k0);
  const int count = share_count<kSplit>(plan, a.G, rank);      // this CTA's items
  const int n_c = a.skip_global ? 0 : a.n_routed[b];   // the routing arrays may be NULL when the global part is skipped

  extern __shared__ __align__(1024) uint8_t smem[];
  uint8_t* sK = smem + SM::kKOff;
  uint8_t* sV = smem + SM::kVOff;
  uint8_t* sQ = smem + SM::kQOff;
  uint8_t* sDO = smem + SM::kDoOff;
  BwdBarriers* bar = reinterpret_cast<BwdBarriers*>(smem + SM::kBarOff);
  uint8_t* sDS = smem + SM::kDsOff;          // dS (bf16, [key][query])
  volatile int* abort_flag = &bar->abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if ((smem_u32(smem) & 1023u) != 0) {   // the swizzled tiles need a 1024-byte aligned base: refuse to run otherwise
    if (tid == 0) atomicExch(a.status, 2);
    return;
  }
  if (plan.total == 0) {
    // no query can see these keys: their gradients are zero
    for (int i = tid; rank == 0 && i < kTileN * (D / 8); i += blockDim.x) {
      const int kr = i / (D / 8), c8 = i % (D / 8);
      if (k0 + kr < a.Lk) {
        const int64_t o = (int64_t)g * D + c8 * 8;
        *reinterpret_cast<uint4*>(a.dK + b * a.dk_st.b + (k0 + kr) * a.dk_st.t + o) = make_uint4(0, 0, 0, 0);
        *reinterpret_cast<uint4*>(a.dV + b * a.dv_st.b + (k0 + kr) * a.dv_st.t + o) = make_uint4(0, 0, 0, 0);
      }
    }
    return;
  }

  if (tid == 0) {
    mbar_init(&bar->kv_full, 1);
    for (int s = 0; s < 2; ++s) {
      mbar_init(&bar->q_full[s], 1); mbar_init(&bar->q_empty[s], 1);
      mbar_init(&bar->do_full[s], 1); mbar_init(&bar->do_empty[s], 1);
      mbar_init(&bar->st_full[s], 32); mbar_init(&bar->st_empty[s], kComputeWarps * 32);
    }
    mbar_init(&bar->s_full, 1);
    mbar_init(&bar->dp_full, 1);
    mbar_init(&bar->p_full, kComputeWarps * 32);     // P^T(i) is in TMEM
    mbar_init(&bar->ds_full, kComputeWarps * 32);    // dS(i) is in shared memory and in TMEM
    mbar_init(&bar->ds_free, 1);                     // dQ(i) has consumed dS(i)
    mbar_init(&bar->dq_full, 1);                     // dQ(i) is in TMEM
    mbar_init(&bar->u_free, 8 * 32);     // dQ(i) has been read out: the columns may take dP^T(i+1)
    mbar_init(&bar->final_bar, 1);
    bar->abort_flag = 0;
    bar->plan = plan;
    bar->b = b;
    bar->g = g;
    bar->k0 = k0;
    bar->n_c = n_c;
    bar->count = count;
    fence_mbar_init();
  }
  if (warp == 17) { tmem_alloc(&bar->tmem_base, 512); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bar->tmem_base;
  if (tmem != 0) {
    // all 512 columns were requested, so the allocation must start at column 0; the MMA warp relies on it to
    // keep its TMEM operand addresses compile-time constants
    __syncthreads();
    if (warp == 17) tmem_dealloc(tmem, 512);
    if (tid == 0) { atomicExch(a.status, 3); *abort_flag = 1; }
    if (kSplit > 1) {       // the cluster's other CTAs store into this one's shared memory between the two barriers
      __syncwarp();
      cluster_sync();
      if (tid == 0) share_abort<kSplit>(abort_flag);
      cluster_sync();
    }
    return;
  }

  // register shares by warpgroup: every warp of a warpgroup executes the same setmaxnreg at the top of its role
  if (warp >= 20) {
    // ------------------------------------------------------------------ dQ read-out: TMEM -> fp32 accumulators
    setmaxnreg_dec<72>();
    // lane == query row of the item's tile; this warp owns the 32 rows of its lane group and one half of the D columns,
    // read in one go: each 32 x 4 piece is then one 512-byte reduction (accumulator layout: see above)
    constexpr int kChunks = D / 32;     // 32-column TMEM loads of the whole tile; this warp takes half of them
    // The tiles of a head follow one another in the accumulator: one pointer that advances, looked up where a head ends.  64
    // of the 72 registers hold the tile, so next to nothing else lives across an item: the thread index is read anew, and
    // head and phase share a register.
    float* base = nullptr;
    int left = 0, hg2 = -2;             // tiles left in this head; 2 * head (group's compact tiles: 2 * G) + phase of dq_full
    bool item_ok = true;
    while (true) {
      if (left <= 0) {
        ItemCursor<kSplit> cur;
        cur.hg = hg2 >> 1;
        cur.settle(bar->plan, a.G, rank);
        if (cur.left <= 0) break;
        const bool glb = cur.hg == a.G;
        const int n = glb ? compact_tiles(a.Lq, a.G) : (a.Lq + kTileM - 1) / kTileM;
        const int lane = thread_index() & 31, grp = (thread_index() >> 5) & 3, half = ((thread_index() >> 5) - 20) >> 2;
        base = glb ? a.dq_acc_glb : a.dq_acc_loc;
        item_ok = dbg_in_range(cur.t >= 0 && cur.t + (cur.left - 1) * kSplit < n && cur.hg <= a.G && base != nullptr, a.status);
        // (this warp's columns start at (D / 2) * half, i.e. at quarter 2 * half of the layout)
        base += ((glb ? (int64_t)bar->b * a.Hkv + bar->g : (int64_t)bar->b * a.Hq + bar->g * a.G + cur.hg) * n + cur.t) *
                    (int64_t)(kTileM * D) + (glb ? head_slot(lane, a.G) : lane) * 4 + ((2 * half) * 4 + grp) * (8 * D);
        left = cur.left;
        hg2 = 2 * cur.hg + (hg2 & 1);
      }
      if (!__all_sync(0xffffffffu, mbar_wait(&bar->dq_full, hg2 & 1, abort_flag))) break;
      tc_fence_after();
      // the warp's whole share (32 rows x D/2 columns) goes to registers first, so that the region is released before
      // the first reduction is issued: the reductions leave the SM at about 32 bytes per clock and must not hold up
      // dP^T(i+1)
      uint32_t v[kChunks / 2][32];
      const uint32_t w = thread_index() >> 5, taddr = ((w & 3) << 21) + 384 + ((w - 20) >> 2) * (D / 2);   // (TMEM starts at 0)
#pragma unroll
      for (int cc = 0; cc < kChunks / 2; ++cc) tmem_ld32(taddr + cc * 32, v[cc]);
      tmem_ld_wait();
      tc_fence_before();
      mbar_arrive(&bar->u_free);           // everything is in registers: dP^T(i+1) may overwrite the columns
      // every offset from the base is a compile-time constant: the sixteen reductions share one address register pair
      if (item_ok) ReadOutReds<D, 0>::run(base, v);
      base += kSplit * kTileM * D;
      --left;
      hg2 ^= 1;
    }
  } else if (warp == 19) {
    setmaxnreg_dec<40>();     // idle
  } else if (warp == 16) {
    // ------------------------------------------------------------------ TMA producer
    setmaxnreg_dec<40>();
    if (lane == 0 && count > 0) {
      tma_prefetch_desc(&mapQ); tma_prefetch_desc(&mapDO); tma_prefetch_desc(&mapQc); tma_prefetch_desc(&mapDOc);
      mbar_expect_tx(&bar->kv_full, 2 * SM::kTileBytes);
      tma_load_4d(sK, &mapK, &bar->kv_full, 0, k0, g * (D / 64), b);
      tma_load_4d(sV, &mapV, &bar->kv_full, 0, k0, g * (D / 64), b);
      ItemCursor<kSplit> cur;
      cur.settle(bar->plan, a.G, rank);
      for (int i = 0; i < count; ++i) {
        const int hg = cur.hg, glb = hg == a.G, row0 = cur.t * kTileM;
        const int hc = glb ? 0 : (g * a.G + hg) * (D / 64), bc = glb ? b * a.Hkv + g : b;
        cur.next(bar->plan, a.G, rank);
        const int st = i & 1;
        const uint32_t ph = ((i >> 1) & 1) ^ 1;
        if (!mbar_wait(&bar->q_empty[st], ph, abort_flag)) break;
        mbar_expect_tx(&bar->q_full[st], SM::kTileBytes);
        tma_load_4d(sQ + st * SM::kTileBytes, glb ? &mapQc : &mapQ, &bar->q_full[st], 0, row0, hc, bc);
        if (!mbar_wait(&bar->do_empty[st], ph, abort_flag)) break;
        mbar_expect_tx(&bar->do_full[st], SM::kTileBytes);
        tma_load_4d(sDO + st * SM::kTileBytes, glb ? &mapDOc : &mapDO, &bar->do_full[st], 0, row0, hc, bc);
      }
    }
    __syncwarp();
  } else if (warp == 18) {
    // ------------------------------------------------------------------ row statistics of each item
    setmaxnreg_dec<40>();
    // lse * log2(e) and Delta of the item's 128 query rows, plus per-quarter mask flags, go to shared memory.
    // The global loads of item i+1 are issued before waiting for its slot, so their latency is hidden.
    float r_lse[4], r_delta[4];
    int r_pos[4], r_lo[4], r_glb = 0, r_row0 = 0;   // r_lo: first token of the row's sequence (packed batches)
    ItemCursor<kSplit> cur;
    cur.settle(bar->plan, a.G, rank);
    auto load_item = [&]() {
      const int hg = cur.hg, glb = hg == a.G, row0 = cur.t * kTileM;
      cur.next(bar->plan, a.G, rank);
      const int n_rows = glb ? n_c * a.G : a.Lq;
      const float* lse = glb ? a.lse_glb : a.lse_loc;
      const float* dl = glb ? a.delta_glb : a.delta_loc;
      r_glb = glb;
      r_row0 = row0;
      // A packed row is (compact index, head of the group): one division a tile, and one by a reciprocal for each row, exact
      // for what is left of it (x G < 2^31).
      const int c0 = glb ? row0 / a.G : row0, rem0 = glb ? row0 - c0 * a.G : 0;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int tile_row = row0 + q * 32 + lane;
        const bool valid = tile_row < n_rows;
        const int x = rem0 + q * 32 + lane;
        const int dc = glb ? (int)__umulhi(2u * x, a.g_inv) : x;
        const int row = c0 + dc;                               // sequence row, or compact index
        const int h = g * a.G + (glb ? x - dc * a.G : hg);
        const int64_t si = ((int64_t)b * a.Hq + h) * a.Lq + (valid ? row : 0);
        // (written by launches of this call that this one may overlap with: not through the read-only path)
        r_lse[q] = valid ? __ldcg(&lse[si]) * kLog2e : 0.f;
        r_delta[q] = valid ? __ldcg(&dl[si]) : 0.f;
        const int token = valid ? (glb ? __ldg(&a.q_idx[(int64_t)b * a.Lq + row]) : row) : 0;
        r_pos[q] = valid ? token - (glb ? a.vis_shift : 0) + a.q_pos_offset : -1;
        r_lo[q] = (valid && a.seq_bounds != nullptr) ? __ldg(&a.seq_bounds[2 * token]) : -0x40000000;
      }
    };
    if (count > 0) load_item();
    for (int i = 0; i < count; ++i) {
      const int s = i & 1;
      if (!__all_sync(0xffffffffu, mbar_wait(&bar->st_empty[s], ((i >> 1) & 1) ^ 1, abort_flag))) break;
      float* st_lse = reinterpret_cast<float*>(smem + SM::kStatOff + s * SM::kStatSlot);
      float* st_delta = st_lse + 128;
      int* st_flags = reinterpret_cast<int*>(st_delta + 128);
      const int w_eff = r_glb ? 0x3fffffff : a.window;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int col = q * 32 + lane;
        st_lse[col] = -r_lse[q];       // negated, like Delta: P = exp2(scale * s + (-lse)) is one fused multiply-add
        st_delta[col] = -r_delta[q];   // negated: dS = P * (dP + (-Delta)) with packed f32x2 arithmetic
        // quarter q needs the element mask unless every (key, query) pair of it is visible
        const bool lane_ok = r_pos[q] >= 0 && (k0 + kTileN - 1 <= r_pos[q]) && (k0 >= max(r_pos[q] - w_eff, r_lo[q]));
        const bool interior = __all_sync(0xffffffffu, lane_ok);
        if (lane == 0) st_flags[q] = interior ? 0 : 1;
      }
      if (lane == 0) { st_flags[4] = r_glb; st_flags[5] = r_row0; }
      __syncwarp();
      mbar_arrive(&bar->st_full[s]);
      if (i + 1 < count) load_item();
    }
  } else if (warp == 17) {
    // ------------------------------------------------------------------ MMA issuer
    // (one elected thread runs the loop)
    setmaxnreg_dec<40>();
    if (elect_one()) {
      constexpr uint32_t tmem = 0;   // checked above: TMEM operand addresses are immediates in this loop
      constexpr uint32_t idesc_s = idesc_bf16_f32(128, 128, 0, 0);
      constexpr uint32_t idesc_acc = idesc_bf16_f32(128, D, 0, 1);
      constexpr uint32_t idesc_dq = idesc_bf16_f32(128, D, 1, 1);     // A = dS read MN-major, B = K read MN-major
      constexpr uint32_t kStageStep = SM::kTileBytes >> 4;
      const uint64_t dk = smem_desc_sw128(smem_u32(sK), 16, 1024), dv = smem_desc_sw128(smem_u32(sV), 16, 1024);
      const uint64_t dkm = smem_desc_sw128(smem_u32(sK), kBoxBytes, 1024);            // K as MN-major B of dQ
      const uint64_t dsm = smem_desc_sw128(smem_u32(sDS), kBoxBytes, 1024);           // dS as MN-major A of dQ
      const uint64_t dq_base = smem_desc_sw128(smem_u32(sQ), 16, 1024);
      const uint64_t ddo_base = smem_desc_sw128(smem_u32(sDO), 16, 1024);
      const uint64_t dqm_base = smem_desc_sw128(smem_u32(sQ), kBoxBytes, 1024);      // Q / dO as MN-major B
      const uint64_t ddom_base = smem_desc_sw128(smem_u32(sDO), kBoxBytes, 1024);
      auto issue_S = [&](int qs) {    // S^T = K Q^T into the T columns
        const uint64_t qd = dq_base + qs * kStageStep;
#pragma unroll
        for (int kk = 0; kk < kKSteps; ++kk) {
          const uint32_t c = ((kk >> 2) * kBoxBytes + (kk & 3) * 32) >> 4;
          mma_ss(tmem + 256, dk + c, qd + c, idesc_s, kk > 0);
        }
        tc_commit(&bar->s_full);
      };
      auto issue_dP = [&](int ds) {   // dP^T = V dO^T into the U columns
        const uint64_t dod = ddo_base + ds * kStageStep;
#pragma unroll
        for (int kk = 0; kk < kKSteps; ++kk) {
          const uint32_t c = ((kk >> 2) * kBoxBytes + (kk & 3) * 32) >> 4;
          mma_ss(tmem + 384, dv + c, dod + c, idesc_s, kk > 0);
        }
        tc_commit(&bar->dp_full);
      };
      auto issue_dQ = [&]() {         // dQ(i) = dS K into the U columns (a fresh accumulator for every item)
#pragma unroll
        for (int kk = 0; kk < 8; ++kk)
          mma_ss(tmem + 384, dsm + ((kk * 2048) >> 4), dkm + ((kk * 2048) >> 4), idesc_dq, kk > 0);
        tc_commit(&bar->dq_full);
        tc_commit(&bar->ds_free);
      };
      auto issue_dV = [&](int ds, bool first) {   // dV += P^T dO, P^T from the T columns
        const uint64_t dod = ddom_base + ds * kStageStep;
#pragma unroll
        for (int kk = 0; kk < 8; ++kk)
          mma_ts(tmem, tmem + 256 + (kk >> 1) * 32 + (kk & 1) * 8, dod + ((kk * 2048) >> 4), idesc_acc,
                 (kk > 0 || !first) ? 1u : 0u);
        tc_commit(&bar->do_empty[ds]);
      };
      auto issue_dK = [&](int qs, bool first) {   // dK += dS^T Q, dS^T from the U columns
        const uint64_t qd = dqm_base + qs * kStageStep;
#pragma unroll
        for (int kk = 0; kk < 8; ++kk)
          mma_ts(tmem + D, tmem + 384 + (kk >> 1) * 32 + (kk & 1) * 8, qd + ((kk * 2048) >> 4), idesc_acc,
                 (kk > 0 || !first) ? 1u : 0u);
        tc_commit(&bar->q_empty[qs]);
      };
      bool ok = count > 0 && mbar_spin(&bar->kv_full, 0, abort_flag) && mbar_spin(&bar->q_full[0], 0, abort_flag) &&
                mbar_spin(&bar->do_full[0], 0, abort_flag);
      if (ok) {
        tc_fence_after();
        issue_S(0);
        issue_dP(0);
      }
      for (int i = 0; ok && i < count; ++i) {
        const bool more = i + 1 < count;
        if (!mbar_spin(&bar->p_full, i & 1, abort_flag)) { ok = false; break; }
        tc_fence_after();
        issue_dV(i & 1, i == 0);
        if (more) {
          // S^T(i+1) overwrites P^T(i): dV(i) precedes it in issue order.  It does not depend on dS(i), so it goes
          // ahead of that wait: the compute warps find the next scores ready when they are done with dS(i)
          if (!mbar_spin(&bar->q_full[(i + 1) & 1], ((i + 1) >> 1) & 1, abort_flag)) { ok = false; break; }
          tc_fence_after();
          issue_S((i + 1) & 1);
        }
        if (!mbar_spin(&bar->ds_full, i & 1, abort_flag)) { ok = false; break; }
        tc_fence_after();
        issue_dK(i & 1, i == 0);
        issue_dQ();                    // over dS^T(i), which dK(i) ahead of it has read
        if (more) {
          const int sn = (i + 1) & 1;
          const uint32_t phn = ((i + 1) >> 1) & 1;
          // dP^T(i+1) overwrites dQ(i): wait for its read-out
          if (!mbar_spin(&bar->u_free, i & 1, abort_flag) ||
              !mbar_spin(&bar->do_full[sn], phn, abort_flag)) { ok = false; break; }
          tc_fence_after();
          issue_dP(sn);
        }
      }
      if (ok) tc_commit(&bar->final_bar);
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------------ P^T, dS and epilogue
    setmaxnreg_inc<80>();
    bool ok = true;
    {                                                  // (scope: nothing of the loop lives on into the epilogue)
    const int q = warp >> 2;                           // query-column quarter of this warp
    const int kr = (warp & 3) * 32 + lane;             // key inside the block == TMEM lane
    const uint32_t lane_base = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const uint32_t s_addr = tmem + lane_base + 256 + q * 32;
    const uint32_t dp_addr = tmem + lane_base + 384 + q * 32;
    for (int i = 0; i < count; ++i) {
      const int s = i & 1;
      // this item's row statistics go to registers before the scores are waited for
      if (!__all_sync(0xffffffffu, mbar_wait(&bar->st_full[s], (i >> 1) & 1, abort_flag))) { ok = false; break; }
      const uint32_t st_base = smem_u32(smem + SM::kStatOff + s * SM::kStatSlot);
      const int* st_flags = reinterpret_cast<const int*>(smem + SM::kStatOff + s * SM::kStatSlot) + 2 * 128;
      float st[32];
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const float4 v = lds128(st_base + (q * 32 + c * 4) * 4);
        st[4 * c] = v.x; st[4 * c + 1] = v.y; st[4 * c + 2] = v.z; st[4 * c + 3] = v.w;
      }
      const bool masked = st_flags[q] != 0;
      // Rows and compact rows ascend in position, so the queries that see this thread's key are one range of them: its
      // bits within this warp's 32 columns.  (Reading position and sequence start of every column instead took an edge
      // tile's probabilities from 1100 to 5900 clk, for one tile in eight at 4K tokens.)
      uint32_t visible = 0;
      if (masked) visible = visible_columns(a, bar->b, bar->n_c, k0 + kr, st_flags[4], st_flags[5] + q * 32);
      if (!__all_sync(0xffffffffu, mbar_wait(&bar->s_full, i & 1, abort_flag))) { ok = false; break; }
      tc_fence_after();
      uint32_t pp[16];
      {
        // the scores come out of TMEM sixteen columns at a time (register budget of the compute warps)
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          uint32_t sv[16];
          tmem_ld16(s_addr + hh * 16, sv);
          tmem_ld_wait();
#pragma unroll
          for (int e8 = 0; e8 < 8; ++e8) {
            const int e = hh * 8 + e8;
            const float2 x = __ffma2_rn(make_float2(__uint_as_float(sv[2 * e8]), __uint_as_float(sv[2 * e8 + 1])),
                                        make_float2(a.scale_log2, a.scale_log2), make_float2(st[2 * e], st[2 * e + 1]));
            pp[e] = pack_bf16(fast_exp2(x.x), fast_exp2(x.y));
          }
          // the element mask is needed only for the few tiles that straddle the causal diagonal or a window edge; it acts on
          // the packed bits, whatever an invisible score's exponential is (a second loop version instead: 965 -> 985 us)
          if (masked) {
#pragma unroll
            for (int e8 = 0; e8 < 8; ++e8) {
              const int e = hh * 8 + e8;
              pp[e] &= ((visible >> (2 * e)) & 1u ? 0xffffu : 0u) | ((visible >> (2 * e + 1)) & 1u ? 0xffff0000u : 0u);
            }
          }
        }
      }
      tmem_st16(s_addr, pp);     // P^T over the first half of this quarter's own S^T columns
      tmem_st_wait();
      tc_fence_before();
      mbar_arrive(&bar->p_full);
      // -Delta of the same rows, again ahead of the wait; after this the statistics slot may be refilled
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const float4 v = lds128(st_base + (128 + q * 32 + c * 4) * 4);
        st[4 * c] = v.x; st[4 * c + 1] = v.y; st[4 * c + 2] = v.z; st[4 * c + 3] = v.w;
      }
      mbar_arrive(&bar->st_empty[s]);
      if (!__all_sync(0xffffffffu, mbar_wait(&bar->dp_full, i & 1, abort_flag))) { ok = false; break; }
      tc_fence_after();
      uint32_t pd[16];
      // dP^T comes out of TMEM sixteen columns at a time: with the 32 statistics and the 16 packed probabilities live,
      // a 32-column load would not fit the compute warps' 80 registers
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        uint32_t dv[16];
        tmem_ld16(dp_addr + hh * 16, dv);
        tmem_ld_wait();
#pragma unroll
        for (int e8 = 0; e8 < 8; ++e8) {
          const int e = hh * 8 + e8;
          // dS uses the bf16-rounded P, the same value the dV product sees; st[] holds -Delta
          const float2 t = __fadd2_rn(make_float2(__uint_as_float(dv[2 * e8]), __uint_as_float(dv[2 * e8 + 1])),
                                      make_float2(st[2 * e], st[2 * e + 1]));
          const float2 ds = __fmul2_rn(make_float2(bf16lo_to_f32(pp[e]), bf16hi_to_f32(pp[e])), t);
          pd[e] = pack_bf16(ds.x, ds.y);
        }
      }
      tmem_st16(dp_addr, pd);    // dS^T over the first half of this quarter's own dP^T columns
      // dS also goes to shared memory, [key][query] with the 128-byte swizzle of a TMA tile (two boxes of 64 queries); the
      // tile of the previous item must have been consumed by dQ(i-1)
      if (i > 0 && !__all_sync(0xffffffffu, mbar_wait(&bar->ds_free, (i - 1) & 1, abort_flag))) { ok = false; break; }
      {
        const uint32_t row = smem_u32(sDS) + (q >> 1) * kBoxBytes + kr * 128;
        const int chunk0 = (q & 1) * 4;
#pragma unroll
        for (int c = 0; c < 4; ++c)
          asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(row + (((chunk0 + c) ^ (kr & 7)) << 4)),
                       "r"(pd[4 * c]), "r"(pd[4 * c + 1]), "r"(pd[4 * c + 2]), "r"(pd[4 * c + 3]) : "memory");
      }
      fence_async_smem();        // the MMA reads the tile through the async proxy
      tmem_st_wait();
      tc_fence_before();         // orders the TMEM accesses above before dK, and before dQ that overwrites the columns
      mbar_arrive(&bar->ds_full);
    }
    }
    // epilogue: quarters 0,1 store the two column halves of dV, quarters 2,3 those of dK
    // (what it needs is read anew: in registers across the items it costs the loop spills)
    const bool own = bar->count > 0; // a CTA whose share is empty issued nothing and adds nothing
    const int q = thread_index() >> 7, kr = thread_index() & 127;
    const uint32_t lane_base = (thread_index() & 96) << 16;
    if (own && ok) ok = __all_sync(0xffffffffu, mbar_wait(&bar->final_bar, 0, abort_flag));
    tc_fence_after();
    if (kSplit > 1) {
      // The accumulators of the cluster's CTAs: quarter q of (dV | dK) belongs to CTA q * kSplit / 4, every other CTA
      // sends it its own into a slot of the Q / dO rings, which nobody reads once all products of the cluster are done.
      const int owner = q * kSplit / 4, me = (int)cluster_rank();
      cluster_sync();
      if (tid == 0) share_abort<kSplit>(abort_flag);
      __syncwarp();
      if (owner != me)
        send_dkv<D, kSplit>(cluster_map(smem_u32(smem + SM::kQOff), owner) +
                            dkv_slot_offset<D, kSplit>((me - owner + kSplit) % kSplit - 1, q, kr),
                            tmem + lane_base + q * (D / 2), own);
      cluster_sync();
      ok = ok && owner == me && *abort_flag == 0;      // (all CTAs have left their waits: the flag is final)
    }
    if (ok) store_dkv<D, kSplit>(a, smem, tmem + lane_base + q * (D / 2), own, bar->b, bar->g, bar->k0 + kr, q, kr);
  }
  if (kSplit > 1 && warp >= kComputeWarps) {   // the other warps' part in the two barriers
    __syncwarp();
    cluster_sync();
    cluster_sync();
  }
  tc_fence_before();
  __syncthreads();
  if (bar->abort_flag) {
    const uint64_t t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
    if (tid == 0) atomicExch(a.status, 1);
    __syncthreads();
  }
  if (warp == 17) tmem_dealloc(tmem, 512);
}

__global__ void __launch_bounds__(256) dq_zero_kernel(float* __restrict__ acc_loc, float* __restrict__ acc_glb,
                                                      const int32_t* __restrict__ n_routed, int B, int Hq, int Hkv, int L,
                                                      int tile_floats) {
  dependency_wait();
  dependents_release();
  zero_accumulators(acc_loc, acc_glb, n_routed, B, Hq, Hkv, L, tile_floats, blockIdx.x, gridDim.x);
}

// fp32 dQ accumulators -> bf16 dQ: dQ_t = scale * (local(t) + d_t * global(prefix[t])), for the row tiles
// [tile_begin, tile_begin + tile_count).  One CTA per (batch, row tile, head); the accumulator blocks are read in their own order (512 contiguous bytes per warp), the bf16 rows leave
// through shared memory as whole 2 D-byte segments.  (The accumulators are neither __restrict__ nor read with __ldg: the
// kernel may start while the one before it still adds to them.)
template <int D>
__global__ void __launch_bounds__(256) dq_merge_kernel(const float* acc_loc, const float* acc_glb,
                                                       const uint8_t* __restrict__ d_mask,
                                                       const int32_t* __restrict__ prefix, bf16* __restrict__ dQ, int B,
                                                       int L, int Hq, int Hkv, float scale, int64_t bs, int64_t ts,
                                                       int tile_begin, int tile_count, int* status) {
  constexpr int kChunks = D / 8;             // 16-byte chunks per bf16 row
  constexpr int kRowBytes = D * 2 + 16;      // padded: conflict-free 16-byte accesses down a column
  __shared__ __align__(16) uint8_t tile_s[kTileM * kRowBytes];
  __shared__ int slot[32];
  if (threadIdx.x < 32) slot[threadIdx.x] = head_slot(threadIdx.x, Hq / Hkv);
  dependency_wait();
  __syncthreads();
  const int n_tiles = (L + kTileM - 1) / kTileM;
  const int h = blockIdx.x % Hq;
  const int tile = tile_begin + (blockIdx.x / Hq) % tile_count;
  const int b = blockIdx.x / (Hq * tile_count);
  const int64_t tile_floats = kTileM * D;
  const int G = Hq / Hkv, kv = h / G, hg = h - kv * G, n_ctiles = compact_tiles(L, G);
  const float* loc = acc_loc ? acc_loc + (((int64_t)b * Hq + h) * n_tiles + tile) * tile_floats : nullptr;
  for (int idx = threadIdx.x; idx < kTileM * kChunks; idx += blockDim.x) {
    const int lane = idx & 31, rq = (idx >> 5) & 3, k = idx >> 7;
    const int r = rq * 32 + lane, t = tile * kTileM + r;
    if (t >= L) continue;
    const int d0 = 8 * k, q = d0 / (D / 4), c = (d0 % (D / 4)) / 4;
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f), y = x;
    if (loc) {
      const float4* p = reinterpret_cast<const float4*>(loc + (q * 4 + rq) * (8 * D) + c * 128 + lane * 4);
      x = __ldcg(p); y = __ldcg(p + 32);
    }
    if (acc_glb && d_mask[(int64_t)b * L + t]) {
      const int cr = prefix[(int64_t)b * (L + 1) + t] * G + hg;
      if (!dbg_in_range(cr >= 0 && cr < n_ctiles * kTileM, status)) continue;
      const float4* p = reinterpret_cast<const float4*>(
          acc_glb + (((int64_t)b * Hkv + kv) * n_ctiles + (cr >> 7)) * tile_floats + (q * 4 + ((cr & 127) >> 5)) * (8 * D) +
          c * 128 + slot[cr & 31] * 4);
      const float4 gx = __ldcg(p), gy = __ldcg(p + 32);
      x.x += gx.x; x.y += gx.y; x.z += gx.z; x.w += gx.w;
      y.x += gy.x; y.y += gy.y; y.z += gy.z; y.w += gy.w;
    }
    *reinterpret_cast<uint4*>(tile_s + r * kRowBytes + k * 16) =
        make_uint4(pack_bf16(x.x * scale, x.y * scale), pack_bf16(x.z * scale, x.w * scale),
                   pack_bf16(y.x * scale, y.y * scale), pack_bf16(y.z * scale, y.w * scale));
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < kTileM * kChunks; idx += blockDim.x) {
    const int r = idx / kChunks, k = idx % kChunks, t = tile * kTileM + r;
    if (t < L)
      *reinterpret_cast<uint4*>(dQ + b * bs + t * ts + (int64_t)h * D + k * 8) =
          *reinterpret_cast<const uint4*>(tile_s + r * kRowBytes + k * 16);
  }
}

}  // namespace
int delta_ctas_per_sm(int D) {
  int per_sm = 0;
  const cudaError_t e = D == 128 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, bwd_delta_kernel<128>, 256, 0)
                                 : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, bwd_delta_kernel<64>, 256, 0);
  return (e != cudaSuccess || per_sm < 1) ? 1 : per_sm;
}
namespace {

size_t rows_bytes(const l2a_params* p) { return align_up((size_t)p->B * p->Lq * p->Hq * p->D * sizeof(bf16), 256); }
size_t stat_bytes(const l2a_params* p) { return align_up((size_t)p->B * p->Hq * p->Lq * sizeof(float), 256); }

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

}  // namespace

int bwd_ranges(int n_kblocks, int n_events, int first[kMaxBwdRanges]) {
  first[0] = 0;
  if (n_events >= 11 && n_kblocks >= 16) {
    first[1] = n_kblocks / 2; first[2] = (3 * n_kblocks) / 4; first[3] = (7 * n_kblocks) / 8;
    return 4;
  }
  if (n_events >= 7 && n_kblocks >= 8) {
    first[1] = (3 * n_kblocks) / 4;
    return 2;
  }
  return 1;
}

// First row tile whose dQ still receives contributions from the key blocks at or after `split`: a row at position p
// only meets keys <= p, so after the key blocks below `split` the rows with p < 128 * split are final.
int dq_final_tiles(int split, int q_pos_offset, int n_tiles) {
  const long long rows = (long long)split * kTileN - q_pos_offset;
  if (rows <= 0) return 0;
  const long long t = rows / kTileM;
  return t > n_tiles ? n_tiles : (int)t;
}

template <int D, int kSplit>
cudaError_t launch_bwd_split(const BwdArgs& a, const CUtensorMap& mapQ, const CUtensorMap& mapDO, const CUtensorMap& mapQc,
                             const CUtensorMap& mapDOc, const CUtensorMap& mapK, const CUtensorMap& mapV, bool overlap,
                             cudaStream_t s) {
  static PerDeviceOnce once;
  cudaError_t e = once.run([] {
    return cudaFuncSetAttribute(bwd_kernel<D, kSplit>, cudaFuncAttributeMaxDynamicSharedMemorySize, BwdSmem<D>::kTotal);
  });
  if (e != cudaSuccess) return e;
  if (kSplit == 1)
    return launch_dependent(bwd_kernel<D, kSplit>, dim3((unsigned)a.kb_count * a.B * a.Hkv), kDkvThreads, BwdSmem<D>::kTotal, s,
                            overlap, mapQ, mapDO, mapQc, mapDOc, mapK, mapV, a);
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kSplit; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)a.kb_count * a.B * a.Hkv * kSplit);
  cfg.blockDim = dim3(kDkvThreads);
  cfg.dynamicSmemBytes = BwdSmem<D>::kTotal;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = overlap ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, bwd_kernel<D, kSplit>, mapQ, mapDO, mapQc, mapDOc, mapK, mapV, a);
}

template <int D>
cudaError_t launch_bwd_kernel(BwdArgs a, const CUtensorMap& mapQ, const CUtensorMap& mapDO, const CUtensorMap& mapQc,
                              const CUtensorMap& mapDOc, const CUtensorMap& mapK, const CUtensorMap& mapV, int sms,
                              bool overlap, cudaStream_t s) {
  // (of the whole sequence, also when the launch is one of several key-block ranges: the results stay the same)
  const int64_t blocks = (int64_t)((a.Lk + kTileN - 1) / kTileN) * a.B * a.Hkv;
  // A cluster per key block where one CTA per block leaves SMs idle or the heaviest block sets the time.  Measured, whole
  // backward with 1 / 2 / 4 CTAs per block at 148 SMs: 32 blocks 224 / 153 / 110 us, 64 blocks 822 / 486 / 461, 128 blocks
  // 750 / 478 / 527 and 272 / 206 / 238, 256 blocks 1435 / 1360 / 1467 and 381 / 399 / 454, 512 blocks 1481 / 1691 / 1907.
  const int split = 2 * blocks < sms ? 4 : 2 * blocks < 3 * sms ? 2 : 1;
  // Below eight waves the heaviest key blocks of every head go first (two sequences of 4096 tokens, 256 blocks: 1.20 ->
  // 0.93 ms); with more waves the tail is short and either order measures the same, so the one with less L2 traffic stays.
  a.kb_outermost = blocks < 8 * sms;
  return split == 1   ? launch_bwd_split<D, 1>(a, mapQ, mapDO, mapQc, mapDOc, mapK, mapV, overlap, s)
         : split == 2 ? launch_bwd_split<D, 2>(a, mapQ, mapDO, mapQc, mapDOc, mapK, mapV, overlap, s)
                      : launch_bwd_split<D, 4>(a, mapQ, mapDO, mapQc, mapDOc, mapK, mapV, overlap, s);
}

template <int D>
cudaError_t launch_bwd(const BwdArgs& base, const CUtensorMap& mapQ, const CUtensorMap& mapDO,
                       const CUtensorMap& mapQc, const CUtensorMap& mapDOc, const CUtensorMap& mapK,
                       const CUtensorMap& mapV, const uint8_t* d_mask, bool zeroed, cudaStream_t s) {
  const DeviceInfo* dev = device_info();
  if (dev == nullptr) return cudaErrorUnknown;
  const int n_tiles = (base.Lq + kTileM - 1) / kTileM;
  const bool overlap = phase_events().n == 0;    // (events between the launches ask for their times one after the other)
  cudaError_t err = cudaSuccess;
  if (!zeroed)
    err = launch_dependent(dq_zero_kernel, dim3(dev->sms * 8), 256, 0, s, overlap, base.dq_acc_loc, base.dq_acc_glb, base.n_routed,
                           base.B, base.Hq, base.Hkv, base.Lq, kTileM * D);
  if (err != cudaSuccess) return err;
  phase_events().mark(s);
  const int n_kblocks = (base.Lk + kTileN - 1) / kTileN;
  // A caller that registered phase events for key-block ranges wants the gradients of the early rows while the rest is
  // computed (to move them to the host): one launch per range, each followed by the merge of the dQ rows it finishes.
  int first[kMaxBwdRanges];
  const int n_ranges = bwd_ranges(n_kblocks, phase_events().n, first);
  int t_done = 0;
  for (int part = 0; part < n_ranges; ++part) {
    BwdArgs a = base;
    const int kb_end = part + 1 < n_ranges ? first[part + 1] : n_kblocks;
    a.kb_begin = first[part];
    a.kb_count = kb_end - first[part];
    const cudaError_t e = launch_bwd_kernel<D>(a, mapQ, mapDO, mapQc, mapDOc, mapK, mapV, dev->sms, overlap, s);
    if (e != cudaSuccess) return e;
    phase_events().mark(s);
    const int t1 = part + 1 < n_ranges ? dq_final_tiles(kb_end, base.q_pos_offset, n_tiles) : n_tiles;
    if (t1 > t_done &&
        (err = launch_dependent(dq_merge_kernel<D>, dim3((unsigned)((t1 - t_done) * base.B * base.Hq)), 256, 0, s, overlap,
                                base.dq_acc_loc, base.dq_acc_glb, d_mask, base.prefix, base.dQ, base.B, base.Lq, base.Hq, base.Hkv,
                                base.scale, base.dq_st.b, base.dq_st.t, t_done, t1 - t_done, base.status)) != cudaSuccess)
      return err;
    if (t1 > t_done) t_done = t1;
    phase_events().mark(s);
  }
  return cudaGetLastError();
}

// Up to this size of an accumulator further CTAs of the Delta kernel clear it, beside Delta where that leaves SMs idle; beyond it a
// kernel behind does (DRAM turns between reads and writes: see Delta).  A step of 706 tokens (4 heads) 55.3 -> 53.2 us, of 2 x 793
// (32/8) 144.6 -> 138.1, 1587 205 -> 198.4, 3000 (28/4) 432 -> 422, layer of 8155 2005 -> 1981, 2 x 4096 the same.
constexpr size_t kZeroByDelta = 128u << 20;

// one fp32 dQ accumulator: whole 128-row tiles
size_t acc_bytes(const l2a_params* p) {
  return align_up((size_t)p->B * p->Hq * ceil_div(p->Lq, kTileM) * kTileM * p->D * sizeof(float), 256);
}
size_t bwd_ws_size(const l2a_params* p) { return kWsHeaderBytes + 2 * rows_bytes(p) + 3 * stat_bytes(p) + 2 * acc_bytes(p); }

}  // namespace l2a

using namespace l2a;

extern "C" l2a_status l2a_backward(const l2a_params* p, const void* Q, const void* K, const void* V,
                                   const uint8_t* d_mask, const int32_t* q_idx, const int32_t* n_routed,
                                   const int32_t* prefix, const void* dO, const void* S_save, const void* A_c,
                                   const float* lse_loc, const float* lse_glb, void* dQ, void* dK, void* dV,
                                   float* dgate, void* bwd_ws, size_t bwd_ws_bytes, void* stream) {
  return l2a_backward_split(p, Q, K, V, d_mask, q_idx, n_routed, prefix, dO, dO, S_save, A_c, lse_loc, lse_glb, dQ, dK,
                            dV, dgate, bwd_ws, bwd_ws_bytes, stream);
}

static l2a_status backward_impl(const l2a_params* p, const void* Q, const void* K, const void* V,
                                const uint8_t* d_mask, const int32_t* q_idx, const int32_t* n_routed,
                                const int32_t* prefix, const void* dO, const void* dS_loc, const void* S_save,
                                const void* A_c, const float* lse_loc, const float* lse_glb, void* dQ, void* dK,
                                void* dV, float* dgate, void* bwd_ws, size_t bwd_ws_bytes, void* stream,
                                bool clear_status);

extern "C" l2a_status l2a_backward_split(const l2a_params* p, const void* Q, const void* K, const void* V,
                                         const uint8_t* d_mask, const int32_t* q_idx, const int32_t* n_routed,
                                         const int32_t* prefix, const void* dO, const void* dS_loc,
                                         const void* S_save, const void* A_c, const float* lse_loc,
                                         const float* lse_glb, void* dQ, void* dK, void* dV, float* dgate,
                                         void* bwd_ws, size_t bwd_ws_bytes, void* stream) {
  return backward_impl(p, Q, K, V, d_mask, q_idx, n_routed, prefix, dO, dS_loc, S_save, A_c, lse_loc, lse_glb, dQ, dK,
                       dV, dgate, bwd_ws, bwd_ws_bytes, stream, true);
}

// Section 3.1: in the paper's layer Global Attention has its own projections of the local output, i.e. its own
// Q/K/V.  One call for both modules: the local module's backward on (Q, K, V), the global module's on (Qg, Kg, Vg).
extern "C" l2a_status l2a_backward_sets(const l2a_params* p, const void* Q, const void* K, const void* V, const void* Qg,
                                        const void* Kg, const void* Vg, const uint8_t* d_mask, const int32_t* q_idx,
                                        const int32_t* n_routed, const int32_t* prefix, const void* dO,
                                        const void* S_save, const void* A_c, const float* lse_loc, const float* lse_glb,
                                        void* dQ, void* dK, void* dV, void* dQg, void* dKg, void* dVg, float* dgate,
                                        void* bwd_ws, size_t bwd_ws_bytes, void* stream) {
  if (!p) return L2A_ERR_INVALID_ARG;
  if (!Qg && !Kg && !Vg)     // one set feeds both modules
    return l2a_backward(p, Q, K, V, d_mask, q_idx, n_routed, prefix, dO, S_save, A_c, lse_loc, lse_glb, dQ, dK, dV, dgate,
                        bwd_ws, bwd_ws_bytes, stream);
  if (!Qg || !Kg || !Vg || !dQg || !dKg || !dVg) return L2A_ERR_INVALID_ARG;
  if (p->flags & (L2A_FLAG_SKIP_LOCAL | L2A_FLAG_SKIP_GLOBAL | L2A_FLAG_FORCE_ALL_GLOBAL)) return L2A_ERR_INVALID_ARG;
  l2a_params q = *p;
  q.flags = (p->flags & ~L2A_FLAG_SHARED_WINDOW) | L2A_FLAG_SKIP_GLOBAL;
  l2a_status st = backward_impl(&q, Q, K, V, nullptr, nullptr, nullptr, nullptr, dO, dO, S_save, nullptr, lse_loc, nullptr,
                                dQ, dK, dV, nullptr, bwd_ws, bwd_ws_bytes, stream, true);
  if (st != L2A_OK) return st;
  q.flags = (p->flags & ~L2A_FLAG_SHARED_WINDOW) | L2A_FLAG_SKIP_LOCAL;
  return backward_impl(&q, Qg, Kg, Vg, d_mask, q_idx, n_routed, prefix, dO, dO, nullptr, A_c, nullptr, lse_glb, dQg, dKg,
                       dVg, dgate, bwd_ws, bwd_ws_bytes, stream, false);
}

static l2a_status backward_impl(const l2a_params* p, const void* Q, const void* K, const void* V,
                                const uint8_t* d_mask, const int32_t* q_idx, const int32_t* n_routed,
                                const int32_t* prefix, const void* dO, const void* dS_loc, const void* S_save,
                                const void* A_c, const float* lse_loc, const float* lse_glb, void* dQ, void* dK,
                                void* dV, float* dgate, void* bwd_ws, size_t bwd_ws_bytes, void* stream,
                                bool clear_status) {
  if (!p) return L2A_ERR_INVALID_ARG;
  if (!dS_loc || !aligned16(dS_loc)) return L2A_ERR_INVALID_ARG;
  size_t need = 0;
  l2a_status st = l2a_workspace_bytes(p, nullptr, nullptr, &need);
  if (st != L2A_OK) return st;
  const bool skip_local = p->flags & L2A_FLAG_SKIP_LOCAL, skip_global = p->flags & L2A_FLAG_SKIP_GLOBAL;
  if (skip_local && skip_global) return L2A_ERR_INVALID_ARG;
  const bool force_all = p->flags & L2A_FLAG_FORCE_ALL_GLOBAL;
  if (!Q || !K || !V || !dO || !dQ || !dK || !dV) return L2A_ERR_INVALID_ARG;
  if (!skip_global && (!d_mask || !q_idx || !n_routed || !prefix || !A_c || !lse_glb)) return L2A_ERR_INVALID_ARG;
  if (!skip_local && (!S_save || !lse_loc)) return L2A_ERR_INVALID_ARG;
  if (force_all && (skip_local || skip_global)) return L2A_ERR_INVALID_ARG;
  if (!aligned16(Q) || !aligned16(K) || !aligned16(V) || !aligned16(dO) || !aligned16(S_save) || !aligned16(A_c) ||
      !aligned16(dQ) || !aligned16(dK) || !aligned16(dV))
    return L2A_ERR_INVALID_ARG;
  if (!bwd_ws || (reinterpret_cast<uintptr_t>(bwd_ws) % 256) != 0 || bwd_ws_bytes < need) return L2A_ERR_WORKSPACE;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  uint8_t* ws = static_cast<uint8_t*>(bwd_ws);
  // the gather, first on the stream where there is one, clears the header (not in the debug build, whose index checks in the
  // same kernel report through it)
#ifdef L2A_DEBUG
  const bool gather_clears = false;
#else
  const bool gather_clears = clear_status && !skip_global;
#endif
  if (clear_status && !gather_clears && cudaMemsetAsync(ws, 0, kWsHeaderBytes, s) != cudaSuccess) return L2A_ERR_CUDA;
  bf16* Qc = reinterpret_cast<bf16*>(ws + kWsHeaderBytes);
  bf16* dOc = reinterpret_cast<bf16*>(ws + kWsHeaderBytes + rows_bytes(p));
  float* delta_loc = reinterpret_cast<float*>(ws + kWsHeaderBytes + 2 * rows_bytes(p));
  float* delta_glb = reinterpret_cast<float*>(ws + kWsHeaderBytes + 2 * rows_bytes(p) + stat_bytes(p));
  float* lse_c = reinterpret_cast<float*>(ws + kWsHeaderBytes + 2 * rows_bytes(p) + 2 * stat_bytes(p));
  float* dq_acc_loc = reinterpret_cast<float*>(ws + kWsHeaderBytes + 2 * rows_bytes(p) + 3 * stat_bytes(p));
  float* dq_acc_glb = reinterpret_cast<float*>(ws + kWsHeaderBytes + 2 * rows_bytes(p) + 3 * stat_bytes(p) + acc_bytes(p));
  // Shared-window backward: the window's share of a routed row's global gradient rides on the local items (see
  // bwd_delta_kernel).  Needs the same gradient for both outputs; the flag permits it, other modes just ignore it.
  const bool share = (p->flags & L2A_FLAG_SHARED_WINDOW) && dS_loc == dO && !skip_local && !skip_global &&
                     !force_all;

  CUtensorMap mapQ, mapDO, mapQc, mapDOc, mapK, mapV;
  const RowStrides qs = resolve_strides(p->q_stride, p->Lq, p->Hq * p->D);
  const RowStrides ks = resolve_strides(p->k_stride, p->Lk, p->Hkv * p->D);
  const RowStrides vs = resolve_strides(p->v_stride, p->Lk, p->Hkv * p->D);
  const RowStrides os = resolve_strides(p->o_stride, p->Lq, p->Hq * p->D);
  if (!encode_rows_map(&mapQ, Q, p->B, p->Lq, p->Hq * p->D, kTileM, p->D, qs.b, qs.t) ||
      !encode_rows_map(&mapDO, dS_loc, p->B, p->Lq, p->Hq * p->D, kTileM, p->D, os.b, os.t) ||   // local items: dL/ds_t
      !encode_rows_map(&mapQc, Qc, p->B * p->Hkv, p->Lq * (p->Hq / p->Hkv), p->D, kTileM, p->D) ||
      !encode_rows_map(&mapDOc, dOc, p->B * p->Hkv, p->Lq * (p->Hq / p->Hkv), p->D, kTileM, p->D) ||
      !encode_rows_map(&mapK, K, p->B, p->Lk, p->Hkv * p->D, kTileN, p->D, ks.b, ks.t) ||
      !encode_rows_map(&mapV, V, p->B, p->Lk, p->Hkv * p->D, kTileN, p->D, vs.b, vs.t))
    return L2A_ERR_CUDA;

  const bool zeroed = (size_t)p->B * p->Hq * p->Lq * p->D * sizeof(float) <= kZeroByDelta;
  PhaseEvents& pe = phase_events();
  struct ClearOnExit { PhaseEvents& p; ~ClearOnExit() { p.clear(); } } clear_on_exit{pe};
  const bool overlap = pe.n == 0;
  pe.mark(s);
  if (!skip_global) {
    if (launch_gather_rows(static_cast<const bf16*>(Q), Qc, q_idx, n_routed, p->B, p->Lq, p->Hq * p->D,
                           p->Hq / p->Hkv, p->D, s, qs, reinterpret_cast<int*>(ws), gather_clears ? reinterpret_cast<int32_t*>(ws) : nullptr,
                           gather_clears ? (int)(kWsHeaderBytes / 4) : 0, false, static_cast<const bf16*>(dO), dOc, os) !=
        cudaSuccess)
      return L2A_ERR_CUDA;
  }
  pe.mark(s);
  {
    // one resident wave of 8-warp CTAs; the warps take the tokens round-robin
    const DeviceInfo* dev = device_info();
    if (dev == nullptr) return L2A_ERR_CUDA;
    auto kern = p->D == 128 ? bwd_delta_kernel<128> : bwd_delta_kernel<64>;
    int64_t blocks = (int64_t)dev->sms * (p->D == 128 ? dev->delta_ctas_128 : dev->delta_ctas_64);
    const int64_t max_blocks = ((int64_t)p->B * p->Lq + 7) / 8;
    if (blocks > max_blocks) blocks = max_blocks;
    const ZeroArgs z = {(int)blocks, skip_local ? nullptr : dq_acc_loc, skip_global ? nullptr : dq_acc_glb, n_routed, p->Hkv};
    if (launch_dependent(kern, dim3((unsigned)(blocks + (zeroed ? 2 * dev->sms : 0))), 256, 0, s, overlap && !skip_global, static_cast<const bf16*>(dO),
                         static_cast<const bf16*>(dS_loc), static_cast<const bf16*>(skip_local ? nullptr : S_save),
                         static_cast<const bf16*>(A_c), skip_global ? nullptr : d_mask, prefix, delta_loc, delta_glb, dgate,
                         p->B, p->Lq, p->Hq, force_all ? 1 : 0, os.b, os.t, lse_loc, lse_glb, share ? lse_c : nullptr, z) !=
        cudaSuccess)
      return L2A_ERR_CUDA;
    if (force_all) {
      dim3 grid((p->Lq + 255) / 256, p->Hq, p->B);
      if (launch_dependent(compact_stat_kernel, grid, 256, 0, s, overlap, lse_glb, lse_c, q_idx, n_routed, p->Lq, p->Hq) !=
          cudaSuccess)
        return L2A_ERR_CUDA;
    }
  }
  BwdArgs a;
  a.B = p->B; a.Lq = p->Lq; a.Lk = p->Lk; a.Hq = p->Hq; a.Hkv = p->Hkv; a.D = p->D;
  a.G = p->Hq / p->Hkv;
  a.g_inv = (uint32_t)(((1ull << 31) + a.G - 1) / a.G);
  a.window = p->window < (1 << 30) ? p->window : (1 << 30);   // any window >= Lk is the same
  a.q_pos_offset = p->q_pos_offset;
  a.scale = p->softmax_scale > 0.f ? p->softmax_scale : 1.0f / sqrtf((float)p->D);
  a.scale_log2 = a.scale * kLog2e;
  a.skip_local = skip_local ? 1 : 0;
  a.skip_global = skip_global ? 1 : 0;
  a.q_idx = q_idx; a.n_routed = n_routed; a.prefix = prefix;
  a.seq_bounds = p->seq_bounds;
  a.lse_loc = share ? lse_c : lse_loc; a.lse_glb = force_all ? lse_c : lse_glb;
  a.vis_shift = share ? (p->window < (1 << 30) ? p->window : (1 << 30)) + 1 : 0; a.delta_loc = delta_loc; a.delta_glb = delta_glb;
  a.dQ = static_cast<bf16*>(dQ); a.dK = static_cast<bf16*>(dK); a.dV = static_cast<bf16*>(dV);
  a.dq_st = qs; a.dk_st = ks; a.dv_st = vs;
  a.dq_acc_loc = !skip_local ? dq_acc_loc : nullptr;
  a.dq_acc_glb = !skip_global ? dq_acc_glb : nullptr;
  a.status = reinterpret_cast<int*>(ws);
  const cudaError_t e =
      p->D == 128 ? launch_bwd<128>(a, mapQ, mapDO, mapQc, mapDOc, mapK, mapV, skip_global ? nullptr : d_mask, zeroed, s)
                  : launch_bwd<64>(a, mapQ, mapDO, mapQc, mapDOc, mapK, mapV, skip_global ? nullptr : d_mask, zeroed, s);
  return e == cudaSuccess ? L2A_OK : L2A_ERR_CUDA;
}
