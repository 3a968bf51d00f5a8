// Routing decision + query compaction (Eq. 3; Section 3.2; Algorithm 1 step 1), and the row gather
// that consolidates routed rows into a contiguous buffer.
//
// One or two small launches, latency bound:
//   route_count : each CTA thresholds 4096 positions and counts its routed ones (ballot + popc); skipped for short
//                 sequences, whose CTAs count all positions themselves
//   route_scan  : each CTA sums the counts of the CTAs before it and writes d_mask, prefix, q_idx (ascending = stable) and
//                 the -1 tail of its own 4096 positions: a warp takes 512 consecutive ones, 32 at a time (one ballot),
//                 so that every store is contiguous (a thread with 16 consecutive positions of its own, storing with a
//                 stride of 64 bytes, took 9.8 us for a block, this 5 to 8).
// Nothing is read back by the host: the routed count stays on the device.
#include "l2a_common.cuh"
#include "sm100_prims.cuh"

namespace l2a {

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kRounds = kRouteBlockElems / kThreads;     // 32-position rounds of a warp
// Blocks of a sequence up to which every CTA counts them all itself (16384 positions: 64 loads a thread, less than the
// second launch costs).
constexpr int kCountAllBlocks = 4;

__device__ __forceinline__ bool routed_at(const RouteArgs& a, int64_t i) {
  if (a.router_kind == L2A_ROUTER_MASK_U8) return static_cast<const uint8_t*>(a.router)[i] != 0;
  const float z = a.router_kind == L2A_ROUTER_LOGITS_BF16 ? __bfloat162float(static_cast<const bf16*>(a.router)[i])
                                                          : static_cast<const float*>(a.router)[i];   // the upcast is exact
  return z >= a.threshold;             // NaN compares false; -0.0 >= 0.0 is true
}

// routed positions among those of block blk this thread looks at
__device__ __forceinline__ int count_block(const RouteArgs& a, int64_t row_base, int blk) {
  int cnt = 0;
#pragma unroll
  for (int i = 0; i < kRounds; ++i) {
    const int t = blk * kRouteBlockElems + i * kThreads + threadIdx.x;
    if (t < a.L && routed_at(a, row_base + t)) ++cnt;
  }
  return cnt;
}

__global__ void __launch_bounds__(kThreads) route_count_kernel(RouteArgs a) {
  const int b = blockIdx.y, blk = blockIdx.x;
  dependents_release();
  const int cnt = __reduce_add_sync(0xffffffffu, count_block(a, (int64_t)b * a.L, blk));
  __shared__ int warp_cnt[kWarps];
  if ((threadIdx.x & 31) == 0) warp_cnt[threadIdx.x >> 5] = cnt;
  __syncthreads();
  if (threadIdx.x == 0) {
    int s = 0;
    for (int w = 0; w < kWarps; ++w) s += warp_cnt[w];
    a.block_sums[b * a.nblocks + blk] = s;
  }
}

template <bool kCountAll>
__global__ void __launch_bounds__(kThreads) route_scan_kernel(RouteArgs a) {
  const int b = blockIdx.y, blk = blockIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t row_base = (int64_t)b * a.L;
  if (!kCountAll) dependency_wait();
  dependents_release();
  __shared__ int red_before[kWarps], red_total[kWarps], warp_cnt[kWarps];
  if (a.header != nullptr && blk == 0 && b == 0 && threadIdx.x < kWsHeaderBytes / 4) a.header[threadIdx.x] = 0;

  // counts of the other CTAs' positions, and of those before this one's
  int before = 0, total = 0;
  for (int i = kCountAll ? 0 : threadIdx.x; i < a.nblocks; i += kCountAll ? 1 : kThreads) {
    if (i == blk) continue;
    const int v = kCountAll ? count_block(a, row_base, i) : a.block_sums[b * a.nblocks + i];
    total += v;
    if (i < blk) before += v;
  }
  before = __reduce_add_sync(0xffffffffu, before);
  total = __reduce_add_sync(0xffffffffu, total);
  // this warp's 512 positions
  const int t0 = blk * kRouteBlockElems + warp * (32 * kRounds);
  uint32_t words[kRounds];
  int cnt = 0;
#pragma unroll
  for (int i = 0; i < kRounds; ++i) {
    const int t = t0 + i * 32 + lane;
    words[i] = __ballot_sync(0xffffffffu, t < a.L && routed_at(a, row_base + t));
    cnt += __popc(words[i]);
  }
  if (lane == 0) { red_before[warp] = before; red_total[warp] = total; warp_cnt[warp] = cnt; }
  __syncthreads();
  int c = 0;
  total = 0;
  for (int w = 0; w < kWarps; ++w) {
    c += red_before[w];
    total += red_total[w] + warp_cnt[w];
    if (w < warp) c += warp_cnt[w];
  }

  uint8_t* dm = a.d_mask + row_base;
  int32_t* qi = a.q_idx + row_base;
  int32_t* pf = a.prefix + (int64_t)b * (a.L + 1);
#pragma unroll
  for (int i = 0; i < kRounds; ++i) {
    const int t = t0 + i * 32 + lane;
    const int on = (words[i] >> lane) & 1;
    const int ci = c + __popc(words[i] & ((1u << lane) - 1u));
    if (t < a.L) {
      dm[t] = (uint8_t)on;
      pf[t] = ci;
      if (on) qi[ci] = t;
      if (t >= total) qi[t] = -1;  // compact slots past the routed count
    }
    c += __popc(words[i]);
  }
  if (blk == 0 && threadIdx.x == 0) {
    a.n_routed[b] = total;
    pf[a.L] = total;
  }
}

// For the backward (the forward's global pass gathers the rows of a tile itself).  One CTA per routed row (grid-stride); 16-byte chunks; src2, if given, is gathered in the same way.  The heads of a KV group
// (group_chunks chunks of a row) lie together in the result: [batch, KV head, compact row, group_chunks].  No input is
// __restrict__ or read with __ldg: the kernel may start while the one before it (the routing, or whatever produced the queries)
// still writes them.
__global__ void __launch_bounds__(256) gather_rows_kernel(const bf16* src, bf16* dst, const int32_t* q_idx,
                                                          const int32_t* n_routed, int L,
                                                          int row_chunks /* 16-byte chunks per row */,
                                                          int group_chunks, int G, int64_t src_batch_chunks,
                                                          int64_t src_row_chunks, int* status, int32_t* zero,
                                                          int n_zero, const bf16* src2, bf16* dst2,
                                                          int64_t src2_batch_chunks, int64_t src2_row_chunks) {
  const int b = blockIdx.y;
  dependency_wait();
  dependents_release();
  if (blockIdx.x == 0 && b == 0)
    for (int i = threadIdx.x; i < n_zero; i += blockDim.x) zero[i] = 0;
  const int n_c = n_routed[b];
  int n_pad = (int)((compact_groups(n_c, G) * kRowsPerCta + G - 1) / G);
  if (n_pad > L) n_pad = L;
  const uint4* s = reinterpret_cast<const uint4*>(src) + b * src_batch_chunks;   // source strides in 16-byte chunks
  uint4* d = reinterpret_cast<uint4*>(dst) + (int64_t)b * L * row_chunks;
  const uint4* s2 = reinterpret_cast<const uint4*>(src2) + b * src2_batch_chunks;
  uint4* d2 = reinterpret_cast<uint4*>(dst2) + (int64_t)b * L * row_chunks;
  auto place = [&](int i, int c) {        // chunk i of compact row c
    const int kv = i / group_chunks;
    return ((int64_t)kv * L + c) * group_chunks + (i - kv * group_chunks);
  };
  for (int c = blockIdx.x; c < n_pad; c += gridDim.x) {
    if (c < n_c) {
      const int t = q_idx[(int64_t)b * L + c];
      if (!dbg_in_range(t >= 0 && t < L, status)) continue;
      for (int i = threadIdx.x; i < row_chunks; i += blockDim.x) {
        const uint4 x = __ldcg(&s[t * src_row_chunks + i]);
        const int64_t o = place(i, c);
        if (src2 != nullptr) d2[o] = __ldcg(&s2[t * src2_row_chunks + i]);
        d[o] = x;
      }
    } else {
      for (int i = threadIdx.x; i < row_chunks; i += blockDim.x) {
        const int64_t o = place(i, c);
        d[o] = make_uint4(0, 0, 0, 0);
        if (src2 != nullptr) d2[o] = make_uint4(0, 0, 0, 0);
      }
    }
  }
}

// Router logit (Eq. 3).  The grid is sized to the machine: the warps take groups of four tokens round-robin (the
// whole grid reads one contiguous stretch of S at a time), four at a time so that each 32-byte piece of w fetched
// (from L1) serves four 16-byte loads of S and several rows are in flight per warp; fp32 accumulation.
constexpr int kRlTokens = 4;
__global__ void __launch_bounds__(256) router_logits_kernel(const bf16* __restrict__ S, const float* __restrict__ w,
                                                            float bias, float* __restrict__ logits,
                                                            float* __restrict__ sum_sq, int B, int L, int row_elems) {
  const int64_t n_tokens = (int64_t)B * L;
  const int64_t n_warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  const int64_t gw = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  const int64_t t_begin = gw * kRlTokens, t_end = n_tokens;
  const int n_chunks = row_elems / 8;
  const float4* w4 = reinterpret_cast<const float4*>(w);
  // sum of sigmoid^2 of this warp's tokens, flushed with one atomic per batch entry they touch (the batch index
  // never decreases along a warp's tokens)
  float reg_sum = 0.f;
  int64_t reg_b = t_begin < t_end ? t_begin / L : 0;
  for (int64_t token0 = t_begin; token0 < t_end; token0 += n_warps * kRlTokens) {
    const uint4* rows[kRlTokens];
    float acc[kRlTokens];
#pragma unroll
    for (int r = 0; r < kRlTokens; ++r) {
      // rows past the range re-read its last token; their result is not stored
      const int64_t tok = token0 + r < t_end ? token0 + r : t_end - 1;
      rows[r] = reinterpret_cast<const uint4*>(S) + tok * n_chunks;
      acc[r] = 0.f;
    }
#pragma unroll 2
    for (int i = lane; i < n_chunks; i += 32) {
      uint4 v[kRlTokens];
#pragma unroll
      for (int r = 0; r < kRlTokens; ++r) v[r] = __ldg(&rows[r][i]);
      const float4 wa = __ldg(&w4[2 * i]), wb = __ldg(&w4[2 * i + 1]);
      const float ww[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
      for (int r = 0; r < kRlTokens; ++r) {
        const uint32_t u[4] = {v[r].x, v[r].y, v[r].z, v[r].w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          acc[r] = fmaf(__uint_as_float(u[k] << 16), ww[2 * k], acc[r]);
          acc[r] = fmaf(__uint_as_float(u[k] & 0xffff0000u), ww[2 * k + 1], acc[r]);
        }
      }
    }
#pragma unroll
    for (int r = 0; r < kRlTokens; ++r) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], o);
      if (lane == 0 && token0 + r < t_end) {
        const float z = acc[r] + bias;
        logits[token0 + r] = z;
        if (sum_sq != nullptr) {
          const float g = 1.0f / (1.0f + __expf(-z));
          const int64_t bb = (token0 + r) / L;
          if (bb != reg_b) {
            atomicAdd(&sum_sq[reg_b], reg_sum);
            reg_sum = 0.f;
            reg_b = bb;
          }
          reg_sum += g * g;
        }
      }
    }
  }
  if (sum_sq != nullptr && lane == 0 && t_end > t_begin) atomicAdd(&sum_sq[reg_b], reg_sum);
}

// A kernel instead of a memset: it may start under the end of the kernel before it.
__global__ void clear_header_kernel(int32_t* header) {
  dependency_wait();
  header[threadIdx.x] = 0;
}

// Packed variable-length batches: token t belongs to the sequence i with cu[i] <= t < cu[i + 1] (binary search over
// the n_seq + 1 boundaries); tokens at or after cu[n_seq] are sequences of their own.
__global__ void __launch_bounds__(256) pack_sequences_kernel(const int32_t* __restrict__ cu, int n_seq, int L,
                                                             int32_t* __restrict__ seq_bounds) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= L) return;
  int lo = 0, hi = n_seq;                  // invariant: cu[lo] <= t (cu[0] = 0); answer in [lo, hi)
  if (n_seq <= 0 || t >= __ldg(&cu[n_seq])) {
    reinterpret_cast<int2*>(seq_bounds)[t] = make_int2(t, t + 1);
    return;
  }
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (__ldg(&cu[mid]) <= t) lo = mid; else hi = mid;
  }
  int first = __ldg(&cu[lo]), end = __ldg(&cu[lo + 1]);
  // boundaries that are not ascending must still give a range that holds t and stays inside the axis
  first = max(0, min(first, t));
  end = min(L, max(end, t + 1));
  reinterpret_cast<int2*>(seq_bounds)[t] = make_int2(first, end);
}

}  // namespace

cudaError_t launch_router_logits(const bf16* S, const float* w, float bias, float* logits, float* sum_sq, int B, int L,
                                 int row_elems, cudaStream_t stream) {
  int device = 0, sms = 148;
  if (cudaGetDevice(&device) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  int per_sm = 0;   // one resident wave: every CTA of the grid runs at once and owns an equal share
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, router_logits_kernel, 256, 0) != cudaSuccess || per_sm < 1)
    per_sm = 1;
  int64_t blocks = (int64_t)sms * per_sm;
  const int64_t max_blocks = ((int64_t)B * L + 8 * kRlTokens - 1) / (8 * kRlTokens);
  if (blocks > max_blocks) blocks = max_blocks;
  router_logits_kernel<<<(unsigned)blocks, 256, 0, stream>>>(S, w, bias, logits, sum_sq, B, L, row_elems);
  return cudaGetLastError();
}

cudaError_t launch_clear_header(void* ws, bool overlap, cudaStream_t stream) {
  return launch_dependent(clear_header_kernel, dim3(1), (unsigned)(kWsHeaderBytes / 4), 0, stream, overlap, static_cast<int32_t*>(ws));
}

cudaError_t launch_pack_sequences(const int32_t* cu_seqlens, int n_seq, int L, int32_t* seq_bounds, cudaStream_t stream) {
  pack_sequences_kernel<<<ceil_div(L, 256), 256, 0, stream>>>(cu_seqlens, n_seq, L, seq_bounds);
  return cudaGetLastError();
}

cudaError_t launch_route_compact(const RouteArgs& a, cudaStream_t stream) {
  dim3 grid(a.nblocks, a.B);
  if (a.nblocks <= kCountAllBlocks) {
    route_scan_kernel<true><<<grid, kThreads, 0, stream>>>(a);
  } else {
    route_count_kernel<<<grid, kThreads, 0, stream>>>(a);
    const cudaError_t e = launch_dependent(route_scan_kernel<false>, grid, kThreads, 0, stream, true, a);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

cudaError_t launch_gather_rows(const bf16* src, bf16* dst, const int32_t* q_idx, const int32_t* n_routed, int B,
                               int L, int row_elems, int G, int D, cudaStream_t stream, RowStrides src_strides, int* status, int32_t* zero, int n_zero, bool overlap,
                               const bf16* src2, bf16* dst2, RowStrides src2_strides) {
  const int row_chunks = row_elems * 2 / 16;
  const int64_t ts = src_strides.t > 0 ? src_strides.t : row_elems;
  const int64_t bs = src_strides.b > 0 ? src_strides.b : (int64_t)L * ts;
  const int64_t ts2 = src2_strides.t > 0 ? src2_strides.t : row_elems;
  const int64_t bs2 = src2_strides.b > 0 ? src2_strides.b : (int64_t)L * ts2;
  int gx = L < 148 * 16 ? L : 148 * 16;
  dim3 grid(gx, B);
  return launch_dependent(gather_rows_kernel, grid, 256, 0, stream, overlap, src, dst, q_idx, n_routed, L, row_chunks, G * D / 8, G,
                          bs / 8, ts / 8, status, zero, n_zero, src2, dst2, bs2 / 8, ts2 / 8);
}

}  // namespace l2a

// ------------------------------------------------------------------------------------------------
// Variant of the routing/compaction entry point that needs no scratch from the caller and allocates
// nothing: the per-CTA counts live in a fixed array in the library's own device image.
//
// In host code `g_static_route_counts` is only a handle for the runtime, not a device address, so
// the launcher is never given the symbol itself: the address is looked up once per device with
// cudaGetSymbolAddress (with that device current) and cached.
static __device__ __align__(256) int32_t g_static_route_counts[L2A_STATIC_ROUTE_SLOTS];

namespace {
constexpr int kMaxDevices = 64;
int32_t* g_static_counts_addr[kMaxDevices] = {};

// Returns the device address of the static array on the current device (nullptr on failure).
int32_t* static_counts_for_current_device() {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
  int32_t* cached = __atomic_load_n(&g_static_counts_addr[dev], __ATOMIC_ACQUIRE);
  if (cached) return cached;
  void* ptr = nullptr;
  if (cudaGetSymbolAddress(&ptr, g_static_route_counts) != cudaSuccess || ptr == nullptr) return nullptr;
  __atomic_store_n(&g_static_counts_addr[dev], static_cast<int32_t*>(ptr), __ATOMIC_RELEASE);
  return static_cast<int32_t*>(ptr);
}
}  // namespace

extern "C" l2a_status l2a_route_compact_static(const l2a_params* p, const void* router, int router_kind,
                                               float logit_threshold, uint8_t* d_mask, int32_t* q_idx,
                                               int32_t* n_routed, int32_t* prefix, void* stream) {
  // shape checks come from the workspace query (host only, launches nothing)
  size_t unused = 0;
  l2a_status st = l2a_workspace_bytes(p, &unused, nullptr, nullptr);
  if (st != L2A_OK) return st;
  if (!router || !d_mask || !q_idx || !n_routed || !prefix) return L2A_ERR_INVALID_ARG;
  if (router_kind != L2A_ROUTER_MASK_U8 && router_kind != L2A_ROUTER_LOGITS_F32 &&
      router_kind != L2A_ROUTER_LOGITS_BF16)
    return L2A_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(q_idx) | reinterpret_cast<uintptr_t>(n_routed) |
       reinterpret_cast<uintptr_t>(prefix)) & 3)
    return L2A_ERR_INVALID_ARG;
  if (router_kind == L2A_ROUTER_LOGITS_F32 && (reinterpret_cast<uintptr_t>(router) & 3)) return L2A_ERR_INVALID_ARG;
  if (router_kind == L2A_ROUTER_LOGITS_BF16 && (reinterpret_cast<uintptr_t>(router) & 1)) return L2A_ERR_INVALID_ARG;
  const int nblocks = l2a::ceil_div(p->Lq, l2a::kRouteBlockElems);
  if ((int64_t)p->B * nblocks > L2A_STATIC_ROUTE_SLOTS) return L2A_ERR_UNSUPPORTED;  // beyond the fixed scratch
  int32_t* counts = static_counts_for_current_device();
  if (!counts) return L2A_ERR_CUDA;
  l2a::RouteArgs a;
  a.router = router;
  a.router_kind = router_kind;
  a.threshold = logit_threshold;
  a.B = p->B;
  a.L = p->Lq;
  a.d_mask = d_mask;
  a.q_idx = q_idx;
  a.n_routed = n_routed;
  a.prefix = prefix;
  a.block_sums = counts;
  a.nblocks = nblocks;
  return l2a::launch_route_compact(a, static_cast<cudaStream_t>(stream)) == cudaSuccess ? L2A_OK : L2A_ERR_CUDA;
}
