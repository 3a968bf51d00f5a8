// Decode step of the layer (Section 3.4): one new query token per sequence attends to the last W+1 keys of the
// cache (Local Attention) and, only if its routing decision d = 1, to the whole cache (Global Attention);
// o = s + d * a.  The work is one pass over the K/V cache: HBM-bound.  The cache of every KV head is cut at the window's
// first key and split into chunks processed by independent CTAs; a chunk's partial soft-max (acc, max, sum) inside the
// window serves both modules, those before it exist for routed tokens only.  decode_combine_kernel, whose CTAs (one per
// sequence and query head) are resident when the last chunk ends, combines the chunks: o is one weighted sum of their
// accumulators.  A single chunk stores its result itself.
//
// One CTA = one chunk of keys of one (batch entry, KV head), for all G query heads of the group:
//   producer warp : streams 64-key K and V tiles through a ring of shared-memory stages with TMA (one 4-D copy
//                   per tile, 128-byte swizzle), so tens of KB per SM are in flight whatever the compute warps do.
//   compute warps : each takes 16 keys of every stage.  The G query heads are the rows of a 16-row MMA A operand
//                   (mma.sync m16n8k16, bf16 in, fp32 accumulate): S = Q K^T from ldmatrix'd K rows, running
//                   soft-max in the exp2 domain on the accumulator fragment, O += P V from transposed ldmatrix of
//                   the V rows.  The rows of A that the heads leave free (8..15) take what the rounding of P to bf16 cuts
//                   off: a window key's rounding enters s and a alike, and adds up there.  The tensor cores are used only to keep the instruction count per key low enough
//                   that the copy engine, not instruction issue, sets the pace.
#include <math.h>

#include <algorithm>

#include "l2a_common.cuh"
#include "sm100_prims.cuh"

namespace l2a {

namespace {

constexpr int kDecKeys = 64;                 // keys per pipeline stage
constexpr int kDecStages = 3;
constexpr int kDecComputeWarps = kDecKeys / 16;
constexpr int kDecThreads = (kDecComputeWarps + 1) * 32;   // + the producer warp
constexpr int kMaxGroup = 8;                 // query heads per KV head supported (rows 0..7 of the A operand)

struct DecodeArgs {
  int B, Lk, Hq, Hkv, G;
  int window, q_pos;       // the new token sits at position q_pos (normally Lk - 1)
  float scale_log2;
  int n_win, n_out;        // chunks of the window / of the keys before it
  const bf16* q;           // [B, Hq, D]
  const uint8_t* d;        // [B] routing decision of the new token (NULL = never routed)
  float* part;             // [B, Hkv, n_win + n_out, G, D + 4]  (acc[D], m, l, 2 unused)
  int* failed;             // [B, Hkv] a wait ran out in one of the chunks: nothing is stored
  bf16* O;                 // [B, Hq, D]
  int* status;             // workspace status word
};

struct DecodeBars {
  uint64_t full[kDecStages], empty[kDecStages];
  int abort_flag;
};

constexpr int kMaxWin = 64, kMaxOut = 512;   // chunks at most
template <int D>
constexpr size_t decode_smem_bytes() {
  return (size_t)kDecStages * 2 * kDecKeys * D * 2 + sizeof(DecodeBars);
}
__device__ __forceinline__ void chunk_range(int lo, int hi, int n, int i, int& c_lo, int& c_hi) {
  const int len = hi - lo + 1;
  int per = (len + n - 1) / n;
  per = (per + kDecKeys - 1) / kDecKeys * kDecKeys;
  c_lo = lo + i * per;
  c_hi = min(hi, c_lo + per - 1);
}

__device__ __forceinline__ void ldsm_x4(uint32_t saddr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(saddr));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t saddr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(saddr));
}
// D += A * B, A 16x16 (row), B 16x8 (col), bf16 operands, fp32 accumulators; a0, a2: rows 0..7 of A, a1, a3: rows 8..15.
__device__ __forceinline__ void mma_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                          uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Address of the 16-byte chunk `chunk` (8 columns) of key row `row` inside a 64-key tile stored as D/64
// consecutive 128-byte-swizzled sub-tiles of 64 rows x 64 columns.
__device__ __forceinline__ uint32_t tile_addr(uint32_t tile, int row, int chunk) {
  return tile + (chunk >> 3) * (kDecKeys * 128) + row * 128 + (((chunk & 7) ^ (row & 7)) << 4);
}

template <int D, int G>
__global__ void __launch_bounds__(kDecThreads, 2)
decode_split_kernel(const DecodeArgs a, const __grid_constant__ CUtensorMap mapK,
                    const __grid_constant__ CUtensorMap mapV) {
  constexpr int kTileBytes = kDecKeys * D * 2;
  constexpr int kStageBytes = 2 * kTileBytes;       // K tile, then V tile
  const int item = blockIdx.x, g = blockIdx.y, b = blockIdx.z;
  dependents_release();
  // (Nobody else sets them so early: a wait runs out seconds from here, and a misaligned base below stops every CTA, this one
  // included.)
  if (item == 0 && threadIdx.x == 0) {
    a.failed[b * a.Hkv + g] = 0;
    if (g == 0 && b == 0) *a.status = 0;
  }
  const bool outside = item >= a.n_win;
  const bool routed = a.d != nullptr && a.d[b] != 0;
  if (outside && !routed) return;                              // Global Attention is skipped when d = 0
  const int win_lo = max(0, a.q_pos - a.window);
  int c_lo, c_hi;
  if (outside) chunk_range(0, win_lo - 1, a.n_out, item - a.n_win, c_lo, c_hi);
  else chunk_range(win_lo, a.q_pos, a.n_win, item, c_lo, c_hi);
  const int n_tiles = c_hi >= c_lo ? (c_hi - c_lo) / kDecKeys + 1 : 0;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  extern __shared__ __align__(1024) uint8_t smem[];
  DecodeBars* bar = reinterpret_cast<DecodeBars*>(smem + kDecStages * kStageBytes);
  volatile int* abort_flag = &bar->abort_flag;
  if ((smem_u32(smem) & 1023u) != 0) {       // the swizzled tile addressing needs a 1024-byte-aligned base
    if (tid == 0) mark_failed(a.status, 2, &a.failed[b * a.Hkv + g]);
    return;
  }
  if (tid == 0) {
    for (int s = 0; s < kDecStages; ++s) {
      mbar_init(&bar->full[s], 1);
      mbar_init(&bar->empty[s], kDecComputeWarps);
    }
    bar->abort_flag = 0;
    fence_mbar_init();
  }
  __syncthreads();

  // per-thread soft-max state of head `hr` (accumulator row) over this warp's keys
  const int hr = lane >> 2, t4 = lane & 3;
  float m_run = -INFINITY, l_run = 0.f;
  float acc[D / 8][4];
#pragma unroll
  for (int j = 0; j < D / 8; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;

  if (warp == kDecComputeWarps) {
    // ================================================================= producer
    if (lane == 0) {
      tma_prefetch_desc(&mapK);
      tma_prefetch_desc(&mapV);
      for (int i = 0; i < n_tiles; ++i) {
        const int s = i % kDecStages, ph = (i / kDecStages) & 1;
        if (!mbar_wait(&bar->empty[s], ph ^ 1, abort_flag)) break;
        uint8_t* stage = smem + s * kStageBytes;
        mbar_expect_tx(&bar->full[s], kStageBytes);
        tma_load_4d(stage, &mapK, &bar->full[s], 0, c_lo + i * kDecKeys, g * (D / 64), b);
        tma_load_4d(stage + kTileBytes, &mapV, &bar->full[s], 0, c_lo + i * kDecKeys, g * (D / 64), b);
      }
    }
  } else {
    // ================================================================= compute warps
    // A fragments of Q: row hr = query head g*G + hr (zero rows for hr >= G), all D columns
    uint32_t qa[D / 16][2];
    {
      const bf16* qrow = a.q + ((int64_t)b * a.Hq + g * G + (hr < G ? hr : 0)) * D;
#pragma unroll
      for (int ks = 0; ks < D / 16; ++ks) {
        const uint32_t v0 = *reinterpret_cast<const uint32_t*>(qrow + ks * 16 + 2 * t4);
        const uint32_t v1 = *reinterpret_cast<const uint32_t*>(qrow + ks * 16 + 8 + 2 * t4);
        qa[ks][0] = hr < G ? v0 : 0u;
        qa[ks][1] = hr < G ? v1 : 0u;
      }
    }
    const int r0 = warp * 16;                          // this warp's key rows inside a stage
    const int lm = lane >> 3, lr = lane & 7;           // ldmatrix: lane -> (matrix, row of the matrix)
    const int k_row = r0 + (lm >> 1) * 8 + lr;         // K: matrices (keys lo|d lo), (keys lo|d hi), (keys hi|..)
    const int v_row = r0 + (lm & 1) * 8 + lr;          // V: matrices (keys lo|cols j), (keys hi|cols j), (..|j+1)

    for (int i = 0; i < n_tiles; ++i) {
      const int s = i % kDecStages, ph = (i / kDecStages) & 1;
      if (!mbar_wait_warp(&bar->full[s], ph, abort_flag)) break;
      const uint32_t tK = smem_u32(smem + s * kStageBytes), tV = tK + kTileBytes;
      const int key0 = c_lo + i * kDecKeys + r0;       // first key of this warp's 16
      if (key0 <= c_hi) {
        const bool tail = key0 + 15 > c_hi;
        // ---- S = Q K^T for 16 keys (two 8-key accumulator tiles)
        float s0[4] = {0.f, 0.f, 0.f, 0.f}, s1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks) {
          uint32_t kb[4];
          ldsm_x4(tile_addr(tK, k_row, ks * 2 + (lm & 1)), kb);
          mma_16816(s0, qa[ks][0], 0u, qa[ks][1], 0u, kb[0], kb[1]);
          mma_16816(s1, qa[ks][0], 0u, qa[ks][1], 0u, kb[2], kb[3]);
        }
        // this thread: head hr, keys key0 + 2*t4 + {0, 1} (s0) and key0 + 8 + 2*t4 + {0, 1} (s1)
        float sc[4] = {s0[0] * a.scale_log2, s0[1] * a.scale_log2, s1[0] * a.scale_log2, s1[1] * a.scale_log2};
        uint32_t vm0 = 0xffffffffu, vm1 = 0xffffffffu;
        if (tail) {
          const int kq = key0 + 2 * t4;
          if (kq > c_hi) { sc[0] = -INFINITY; vm0 &= 0xffff0000u; }
          if (kq + 1 > c_hi) { sc[1] = -INFINITY; vm0 &= 0x0000ffffu; }
          if (kq + 8 > c_hi) { sc[2] = -INFINITY; vm1 &= 0xffff0000u; }
          if (kq + 9 > c_hi) { sc[3] = -INFINITY; vm1 &= 0x0000ffffu; }
        }
        float mx = fmaxf(fmaxf(sc[0], sc[1]), fmaxf(sc[2], sc[3]));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        const float m_new = fmaxf(m_run, mx);          // finite: key0 <= c_hi, so key 0 of the 16 is valid
        const float alpha = exp2f(m_run - m_new);      // 0 on the first step (m_run = -inf)
        const float p0 = exp2f(sc[0] - m_new), p1 = exp2f(sc[1] - m_new);
        const float p2 = exp2f(sc[2] - m_new), p3 = exp2f(sc[3] - m_new);
        l_run = l_run * alpha + ((p0 + p1) + (p2 + p3));   // per-thread partial sum, reduced at the end
        m_run = m_new;
        if (__any_sync(0xffffffffu, alpha != 1.f)) {
#pragma unroll
          for (int j = 0; j < D / 8; ++j) { acc[j][0] *= alpha; acc[j][1] *= alpha; acc[j][2] *= alpha; acc[j][3] *= alpha; }
        }
        const uint32_t pa0 = pack_bf16(p0, p1), pa2 = pack_bf16(p2, p3);
        const uint32_t pa1 = pack_bf16(p0 - __uint_as_float(pa0 << 16), p1 - __uint_as_float(pa0 & 0xffff0000u));
        const uint32_t pa3 = pack_bf16(p2 - __uint_as_float(pa2 << 16), p3 - __uint_as_float(pa2 & 0xffff0000u));
        // ---- O += P V: B fragments are the transposed 8x8 blocks of the V rows
#pragma unroll
        for (int jj = 0; jj < D / 16; ++jj) {
          uint32_t vb[4];
          ldsm_x4_t(tile_addr(tV, v_row, jj * 2 + (lm >> 1)), vb);
          if (tail) { vb[0] &= vm0; vb[1] &= vm1; vb[2] &= vm0; vb[3] &= vm1; }   // rows past the chunk may hold anything
          mma_16816(acc[2 * jj], pa0, pa1, pa2, pa3, vb[0], vb[1]);
          mma_16816(acc[2 * jj + 1], pa0, pa1, pa2, pa3, vb[2], vb[3]);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&bar->empty[s]);
    }
  }

  // ---- merge the compute warps of this CTA (stage memory is free once every warp has left the loop), then
  // write the chunk's partial result
  __syncthreads();
  float* red_acc = reinterpret_cast<float*>(smem);                           // [warps][G][D]
  float* red_m = red_acc + kDecComputeWarps * G * D;                         // [warps][G], then the factors of the sums
  float* red_l = red_m + kDecComputeWarps * G;
  float ls = l_run;
  ls += __shfl_xor_sync(0xffffffffu, ls, 1);
  ls += __shfl_xor_sync(0xffffffffu, ls, 2);
  if (warp < kDecComputeWarps && hr < G) {
    if (t4 == 0) { red_m[warp * G + hr] = m_run; red_l[warp * G + hr] = ls; }
#pragma unroll
    for (int j = 0; j < D / 8; ++j)
      // (an infinite value stays what it is: the part cut off may have the other sign or be zero)
      *reinterpret_cast<float2*>(&red_acc[(warp * G + hr) * D + j * 8 + 2 * t4]) =
          make_float2(acc[j][0] + (isfinite(acc[j][0]) ? acc[j][2] : 0.f), acc[j][1] + (isfinite(acc[j][1]) ? acc[j][3] : 0.f));
  }
  __syncthreads();
  const int n_items = a.n_win + a.n_out;
  const bool single = (routed ? n_items : a.n_win) == 1;       // nothing to combine: the result goes straight out
  constexpr int kRow = D + 4;
  float* base = a.part + (((int64_t)b * a.Hkv + g) * n_items + item) * (G * kRow);
  // one thread per head takes the maximum and the sum; it leaves each warp's factor in place of its maximum
  if (tid < G) {
    float M = -INFINITY, L = 0.f;
#pragma unroll
    for (int w = 0; w < kDecComputeWarps; ++w) M = fmaxf(M, red_m[w * G + tid]);
#pragma unroll
    for (int w = 0; w < kDecComputeWarps; ++w) {
      const float mw = red_m[w * G + tid];
      const float f = (mw == -INFINITY) ? 0.f : exp2f(mw - M);
      L += red_l[w * G + tid] * f;
      red_m[w * G + tid] = f;
    }
    if (single) red_l[tid] = routed ? 1.f / L + 1.f / L : 1.f / L;     // routed: window and whole cache are the same keys
    else *reinterpret_cast<float2*>(base + tid * kRow + D) = make_float2(M, L);
  }
  __syncthreads();
  for (int x = tid; x < G * (D / 4); x += kDecThreads) {
    const int h = x / (D / 4), c4 = x % (D / 4);
    float4 A = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int w = 0; w < kDecComputeWarps; ++w) {
      const float4 v = *reinterpret_cast<const float4*>(&red_acc[(w * G + h) * D + c4 * 4]);
      const float f = red_m[w * G + h];
      A.x += v.x * f; A.y += v.y * f; A.z += v.z * f; A.w += v.w * f;
    }
    if (!single) {
      *reinterpret_cast<float4*>(base + h * kRow + c4 * 4) = A;
    } else if (bar->abort_flag == 0) {
      const float w = red_l[h];
      reinterpret_cast<uint2*>(a.O + ((int64_t)b * a.Hq + g * G + h) * D)[c4] =
          make_uint2(pack_bf16(w * A.x, w * A.y), pack_bf16(w * A.z, w * A.w));
    }
  }
  if (bar->abort_flag) {
    // a bounded wait ran out: give copies still in flight time to land before shared memory is released
    const uint64_t t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
    if (tid == 0) mark_failed(a.status, 1, &a.failed[b * a.Hkv + g]);
    __syncthreads();
  }
}

// Combines the chunks of one query head of one sequence:
//   o = sum_win acc_i 2^(m_i - M_win) / L_win + d * sum_all acc_i 2^(m_i - M_all) / L_all
// Bound by latencies, not by the rows it reads: so every thread asks for its share of the first kCombineAhead * 128 / (D / 4)
// chunks (48 for D = 128) before the weights are known, and the launch overlaps with the end of the chunks.  The CTA of a
// (sequence, KV head) that finished last did this before, behind a counter that a memset ahead of the kernel cleared:
// 6.7 of 12.7 us for one sequence of 9001 keys (28/4 heads, routed), and 2.3 us for the memset.
constexpr int kCombineThreads = 128, kCombineAhead = 12;
template <int D>
__global__ void __launch_bounds__(kCombineThreads) decode_combine_kernel(const DecodeArgs a) {
  constexpr int kLanes = D / 4, kGroups = kCombineThreads / kLanes, kRow = D + 4;
  __shared__ float weight[kMaxWin + kMaxOut];
  __shared__ float4 red[kGroups][kLanes];
  __shared__ float2 red_win[kCombineThreads / 32], red_all[kCombineThreads / 32];    // (maximum, sum)
  const int h = blockIdx.x, b = blockIdx.y, G = a.G, g = h / G;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int c4 = tid % kLanes, grp = tid / kLanes;
  const int n_items = a.n_win + a.n_out;
  dependency_wait();
  const bool routed = a.d != nullptr && a.d[b] != 0;
  const int n = routed ? n_items : a.n_win;
  if (n == 1) return;                                            // stored by its only chunk
  const float* base = a.part + (((int64_t)b * a.Hkv + g) * n_items * G + h % G) * kRow;
  const int64_t step = (int64_t)G * kRow;
  float4 v[kCombineAhead];
#pragma unroll
  for (int i = 0; i < kCombineAhead; ++i) {
    const int k = grp + i * kGroups;
    v[i] = k < n ? __ldcg(reinterpret_cast<const float4*>(base + k * step + c4 * 4)) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  const bool failed = has_failed(&a.failed[b * a.Hkv + g]);
  constexpr int kMine = (kMaxWin + kMaxOut + kCombineThreads - 1) / kCombineThreads;
  float2 ml[kMine];
  float m_win = -INFINITY, m_all = -INFINITY;
#pragma unroll
  for (int i = 0; i < kMine; ++i) {
    const int k = tid + i * kCombineThreads;
    ml[i] = k < n ? __ldcg(reinterpret_cast<const float2*>(base + k * step + D)) : make_float2(-INFINITY, 0.f);
    m_all = fmaxf(m_all, ml[i].x);
    if (k < a.n_win) m_win = fmaxf(m_win, ml[i].x);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    m_win = fmaxf(m_win, __shfl_xor_sync(0xffffffffu, m_win, o));
    m_all = fmaxf(m_all, __shfl_xor_sync(0xffffffffu, m_all, o));
  }
  if (lane == 0) { red_win[warp].x = m_win; red_all[warp].x = m_all; }
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kCombineThreads / 32; ++w) {
    m_win = fmaxf(m_win, red_win[w].x);
    m_all = fmaxf(m_all, red_all[w].x);
  }
  float l_win = 0.f, l_all = 0.f;
#pragma unroll
  for (int i = 0; i < kMine; ++i) {
    if (ml[i].x == -INFINITY) continue;                          // (a chunk without keys wrote no maximum)
    l_all += ml[i].y * exp2f(ml[i].x - m_all);
    if (tid + i * kCombineThreads < a.n_win) l_win += ml[i].y * exp2f(ml[i].x - m_win);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    l_win += __shfl_xor_sync(0xffffffffu, l_win, o);
    l_all += __shfl_xor_sync(0xffffffffu, l_all, o);
  }
  if (lane == 0) { red_win[warp].y = l_win; red_all[warp].y = l_all; }
  __syncthreads();
  l_win = 0.f;
  l_all = 0.f;
#pragma unroll
  for (int w = 0; w < kCombineThreads / 32; ++w) {
    l_win += red_win[w].y;
    l_all += red_all[w].y;
  }
#pragma unroll
  for (int i = 0; i < kMine; ++i) {
    const int k = tid + i * kCombineThreads;
    if (k >= n) continue;
    float w = 0.f;
    if (ml[i].x != -INFINITY) {
      if (k < a.n_win) w = exp2f(ml[i].x - m_win) / l_win;
      if (routed) w += exp2f(ml[i].x - m_all) / l_all;
    }
    weight[k] = w;
  }
  __syncthreads();
  float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
  auto add = [&](int k, const float4& x) {
    const float w = weight[k];
    o.x = fmaf(w, x.x, o.x);
    o.y = fmaf(w, x.y, o.y);
    o.z = fmaf(w, x.z, o.z);
    o.w = fmaf(w, x.w, o.w);
  };
#pragma unroll
  for (int i = 0; i < kCombineAhead; ++i)
    if (grp + i * kGroups < n) add(grp + i * kGroups, v[i]);
#pragma unroll 4
  for (int k = grp + kCombineAhead * kGroups; k < n; k += kGroups)
    add(k, __ldcg(reinterpret_cast<const float4*>(base + k * step + c4 * 4)));
  red[grp][c4] = o;
  __syncthreads();
  if (grp == 0 && !failed) {
#pragma unroll
    for (int s = 1; s < kGroups; ++s) {
      const float4 x = red[s][c4];
      o.x += x.x; o.y += x.y; o.z += x.z; o.w += x.w;
    }
    reinterpret_cast<uint2*>(a.O + ((int64_t)b * a.Hq + h) * D)[c4] = make_uint2(pack_bf16(o.x, o.y), pack_bf16(o.z, o.w));
  }
}

// Chunks as long as one resident wave of CTAs (two per SM, 148 SMs) allows, between 256 and 4096 keys: every chunk costs
// its launch and a row per head that the combination reads back.  Measured against four times as many: one sequence of 128K
// keys (28/4 heads) 64 / 87 us, two of 40K 27 / 36, six of 100K with one KV head 63 / 84, 16 of 128K with four routed 342
// (2048 keys at most: 353), 32 of 8000 not routed 90 / 92, one of 9001 16.4 with either.
// Before the window only routed sequences have work, and the host does not know which are.  Chunks there are no longer than
// lets ONE routed sequence fill every SM once, but have 1536 keys: the CTAs of the others cost their launch.  Microseconds
// without this limit / with it (/ with 1024 / 2048 keys): one routed of 16 sequences of 32K (28/4 heads) 68 / 49 (47 / 52),
// of 32 of 60K (8/1) 59 / 39 (37 / 43), of 16 of 128K (8/1) 50 / 37 (35 / 38); none of 32 of 8000 (32/8) 89 / 91 (102 / 90),
// none of 16 of 128K (8/1) 18.7 / 21.6 (22.8 / 20.9); all of 16 of 128K (8/1) 170 / 179 (184 / 176).
// (All of these with the combination by the CTA that finished last.  With decode_combine_kernel, captured calls back to
// back: one sequence of 9001 keys (28/4 heads) routed 16.4 -> 7.6, not routed 14.4 -> 7.3; of 40000 30.4 -> 18.1; of 128K
// (32/8) 96.6 -> 88.0; one routed of 16 of 32K (28/4) 45.7 -> 39.6, of 32 of 60K (8/1) 28.7 -> 19.7; none of 32 of 8000
// (32/8) 92.1 -> 86.7; all of 16 of 128K (8/1) 180.1 -> 165.6; four routed of 16 of 128K (32/8) 346.8 -> 338.5.)
constexpr int kChunkTarget = 2 * 148, kChunkMin = 256, kChunkMax = 4096;
constexpr int kSoloTarget = 148, kSoloMin = 1536;
void window_and_rest(const l2a_params* p, int* win, int* out) {
  *win = std::min(p->q_pos_offset, p->window) + 1;
  *out = p->q_pos_offset + 1 - *win;
}
void plan_chunks(const l2a_params* p, int* n_win, int* n_out) {
  int win, out;
  window_and_rest(p, &win, &out);
  const int64_t pairs = (int64_t)p->B * p->Hkv;
  auto chunk = [](int64_t keys, int target, int least) {     // keys over `target` chunks
    const int64_t per = (keys + target - 1) / target;
    return (int)(per < least ? least : (per > kChunkMax ? kChunkMax : (per + kDecKeys - 1) / kDecKeys * kDecKeys));
  };
  *n_win = std::min(ceil_div(win, chunk(win * pairs, kChunkTarget, kChunkMin)), kMaxWin);
  const int solo = chunk((int64_t)(win + out) * p->Hkv, kSoloTarget, kSoloMin);
  *n_out = std::min(ceil_div(out, std::min(solo, chunk((win + out) * pairs, kChunkTarget, kChunkMin))), kMaxOut);
}
// Chunks of all (sequence, KV head) pairs at any position up to p's and any batch up to p's: a caller sizes the workspace
// once, for the full cache, while the plan of a shorter one can have more chunks (its length is rounded to whole tiles).  A
// chunk has at least kChunkMin keys and at least the share of keys * pairs / kChunkTarget, or kChunkMax; before the window
// it may also have kSoloMin keys, and at least the share of keys * Hkv / kSoloTarget.
int64_t chunks_bound(const l2a_params* p) {
  int win, out;
  window_and_rest(p, &win, &out);
  const int64_t pairs = (int64_t)p->B * p->Hkv;
  auto chunks = [&](int64_t keys, int length) { return pairs * ((keys + length - 1) / length); };
  auto bound = [&](int64_t keys) {
    return std::max(std::min(chunks(keys, kChunkMin), kChunkTarget + pairs), chunks(keys, kChunkMax));
  };
  const int64_t solo = std::min(chunks(out, kSoloMin), (int64_t)p->B * (kSoloTarget + p->Hkv));
  return std::min(bound(win), pairs * kMaxWin) + std::min(std::max(bound(out), solo), pairs * kMaxOut);
}

template <int D, int G>
cudaError_t launch_split(const DecodeArgs& a, const CUtensorMap& mapK, const CUtensorMap& mapV, dim3 grid,
                         cudaStream_t s) {
  constexpr size_t smem = decode_smem_bytes<D>();
  static PerDeviceOnce once;
  const cudaError_t e = once.run([] {
    return cudaFuncSetAttribute(decode_split_kernel<D, G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  });
  if (e != cudaSuccess) return e;
  decode_split_kernel<D, G><<<grid, kDecThreads, smem, s>>>(a, mapK, mapV);
  return cudaGetLastError();
}

template <int D>
cudaError_t launch_split_d(const DecodeArgs& a, const CUtensorMap& mapK, const CUtensorMap& mapV, dim3 grid,
                           cudaStream_t s) {
  switch (a.G) {
    case 1: return launch_split<D, 1>(a, mapK, mapV, grid, s);
    case 2: return launch_split<D, 2>(a, mapK, mapV, grid, s);
    case 3: return launch_split<D, 3>(a, mapK, mapV, grid, s);
    case 4: return launch_split<D, 4>(a, mapK, mapV, grid, s);
    case 5: return launch_split<D, 5>(a, mapK, mapV, grid, s);
    case 6: return launch_split<D, 6>(a, mapK, mapV, grid, s);
    case 7: return launch_split<D, 7>(a, mapK, mapV, grid, s);
    case 8: return launch_split<D, 8>(a, mapK, mapV, grid, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace
}  // namespace l2a

using namespace l2a;

static size_t failed_bytes(const l2a_params* p) { return align_up((size_t)p->B * p->Hkv * sizeof(int), 256); }

static size_t decode_ws_size(const l2a_params* p, int64_t chunks) {
  return kWsHeaderBytes + failed_bytes(p) + align_up((size_t)chunks * (p->Hq / p->Hkv) * (p->D + 4) * sizeof(float), 256);
}

static l2a_status check_decode(const l2a_params* p) {
  size_t unused = 0;
  const l2a_status st = l2a_workspace_bytes(p, &unused, nullptr, nullptr);
  return st != L2A_OK ? st : p->Lq != 1 ? L2A_ERR_INVALID_ARG : L2A_OK;
}

extern "C" l2a_status l2a_decode_workspace_bytes(const l2a_params* p, size_t* ws_bytes) {
  const l2a_status st = check_decode(p);
  if (st != L2A_OK) return st;
  if (!ws_bytes) return L2A_ERR_INVALID_ARG;
  *ws_bytes = decode_ws_size(p, chunks_bound(p));
  return L2A_OK;
}

extern "C" l2a_status l2a_decode(const l2a_params* p, const void* q, const void* K, const void* V, const uint8_t* d,
                                 void* O, void* ws, size_t ws_bytes, void* stream) {
  const l2a_status st = check_decode(p);
  if (st != L2A_OK) return st;
  if (!q || !K || !V || !O) return L2A_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(q) | reinterpret_cast<uintptr_t>(K) | reinterpret_cast<uintptr_t>(V) |
       reinterpret_cast<uintptr_t>(O)) & 15)
    return L2A_ERR_INVALID_ARG;
  if (p->Hq / p->Hkv > kMaxGroup) return L2A_ERR_UNSUPPORTED;
  if (p->seq_bounds) return L2A_ERR_UNSUPPORTED;   // a decode step has one cache per batch entry
  if (p->q_pos_offset >= p->Lk) return L2A_ERR_INVALID_ARG;     // the new token's own key must be in the cache
  DecodeArgs a;
  plan_chunks(p, &a.n_win, &a.n_out);
  if (!ws || (reinterpret_cast<uintptr_t>(ws) % 256) != 0 ||
      ws_bytes < decode_ws_size(p, (int64_t)p->B * p->Hkv * (a.n_win + a.n_out)))
    return L2A_ERR_WORKSPACE;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  CUtensorMap mapK, mapV;
  if (!is_dense(p->q_stride, p->Lq, p->Hq * p->D) || !is_dense(p->o_stride, p->Lq, p->Hq * p->D)) return L2A_ERR_UNSUPPORTED;
  const RowStrides ks = resolve_strides(p->k_stride, p->Lk, p->Hkv * p->D);
  const RowStrides vs = resolve_strides(p->v_stride, p->Lk, p->Hkv * p->D);
  if (!encode_rows_map(&mapK, K, p->B, p->Lk, p->Hkv * p->D, kDecKeys, p->D, ks.b, ks.t) ||
      !encode_rows_map(&mapV, V, p->B, p->Lk, p->Hkv * p->D, kDecKeys, p->D, vs.b, vs.t))
    return L2A_ERR_CUDA;
  a.B = p->B; a.Lk = p->Lk; a.Hq = p->Hq; a.Hkv = p->Hkv; a.G = p->Hq / p->Hkv;
  a.window = p->window;
  a.q_pos = p->q_pos_offset;
  a.scale_log2 = (p->softmax_scale > 0.f ? p->softmax_scale : 1.0f / sqrtf((float)p->D)) * 1.4426950408889634f;
  a.q = static_cast<const bf16*>(q);
  a.d = d;
  a.status = static_cast<int*>(ws);
  a.failed = reinterpret_cast<int*>(static_cast<uint8_t*>(ws) + kWsHeaderBytes);
  a.part = reinterpret_cast<float*>(static_cast<uint8_t*>(ws) + kWsHeaderBytes + failed_bytes(p));
  a.O = static_cast<bf16*>(O);
  const dim3 grid(a.n_win + a.n_out, p->Hkv, p->B);
  cudaError_t e = p->D == 128 ? launch_split_d<128>(a, mapK, mapV, grid, s) : launch_split_d<64>(a, mapK, mapV, grid, s);
  if (e == cudaSuccess && grid.x > 1) {
    const dim3 heads(p->Hq, p->B);
    e = p->D == 128 ? launch_dependent(decode_combine_kernel<128>, heads, kCombineThreads, 0, s, true, a)
                    : launch_dependent(decode_combine_kernel<64>, heads, kCombineThreads, 0, s, true, a);
  }
  return e == cudaSuccess ? L2A_OK : L2A_ERR_CUDA;
}
