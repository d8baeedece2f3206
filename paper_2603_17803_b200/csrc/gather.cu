// Stage 4a: gather of the selected pages (the cross-tier transfer of Sec. 6, here a copy inside
// HBM), and the index build that produces the per-page min/max key summaries.
//
// Both are pure streaming kernels: 16-byte loads and stores, one contiguous K (or V) block of
// S*256 bytes per (page, kv head), no reuse -- bound by HBM bandwidth.
#include "swarm_internal.cuh"

#include <algorithm>

namespace swarm {
namespace {

// One warp per (b, h, slot j): copies the K block and the V block (adjacent in the pool) of page sel[b][h][j] for head
// kv(h) into rows [j*S, (j+1)*S) of the head's gathered buffers.  Rows of padding tokens and whole
// unused slots are written as zeros.
// Bound by HBM (copies written, distinct pages read).  A warp keeps four 512-byte loads in flight behind one trip for
// the indices, 48 warps per SM.  (A CTA of 256 threads per slot, two loads per thread behind three dependent trips, was
// bound by the turn-over of its CTAs.  157 MB written from 79 MB, behind the selection and the resolution: 55 -> 50 us;
// 645 MB: 187 -> 187 us.  More bytes in flight help a gather that runs by itself, 45 -> 43 us at sixteen loads per lane, and
// hurt one that starts on all SMs at once behind another kernel, 187 -> 197 us.)
constexpr int kGatherThreads = 128, kGatherBatch = 4;
__global__ void __launch_bounds__(kGatherThreads, 12)
gather_kernel(Geometry geo, const uint16_t* __restrict__ kv_pool, const int32_t* __restrict__ sel,
              const int32_t* __restrict__ n_sel, const int64_t* __restrict__ page_base,
              const int32_t* __restrict__ ctx_len, uint16_t* __restrict__ k_out, uint16_t* __restrict__ v_out,
              int32_t* __restrict__ n_tok, uint32_t* __restrict__ status) {
  pdl_wait();                                               // (its launch overlaps what precedes it in the stream)
  pdl_launch_dependents();
  const int lane = threadIdx.x & 31;
  const long long u = (long long)blockIdx.x * (kGatherThreads / 32) + (threadIdx.x >> 5);
  if (u >= (long long)geo.B * geo.Hq * geo.k) return;
  const int bh = (int)(u / geo.k), j = (int)(u - (long long)bh * geo.k), b = bh / geo.Hq, h = bh - b * geo.Hq;
  const int S = geo.S;
  const int len = ctx_len[b], ns = n_sel[bh], chosen = sel[u];
  const int64_t base = page_base[b];
  const int P = pages_of(len, S);
  const int tail = len - S * (P - 1);                       // valid tokens of the last page
  const long long blk = (long long)S * kHeadDim;            // elements per K (or V) block
  int p = j < ns ? chosen : -1;
  if (j < ns && (p < 0 || p >= P)) {
    if (lane == 0) atomicOr(status, SWARM_DEV_BAD_PAGE);
    p = -1;
  }
  // The attention over gathered buffers masks only the end of the last slot: a partial page anywhere else would
  // put its padding rows among the valid tokens.  The library's own selections are ascending, so this can only
  // happen with a selection the caller wrote.
  if (p == P - 1 && tail != S && j != ns - 1) {
    if (lane == 0) atomicOr(status, SWARM_DEV_BAD_PAGE);
    p = -1;
  }
  const int valid = p < 0 ? 0 : (p == P - 1 ? tail : S);
  const uint4 zero = make_uint4(0, 0, 0, 0);
  const uint16_t* src = kv_pool + (((base + max(p, 0)) * geo.Hkv + h / geo.g) * 2) * blk;
  uint4* kd = reinterpret_cast<uint4*>(k_out + u * blk);
  uint4* vd = reinterpret_cast<uint4*>(v_out + u * blk);
  const int vecs = S * kHeadDim / 8;                        // 16-byte vectors per block (16 per token)
  for (int t0 = 0; t0 < S; t0 += kGatherBatch) {            // both blocks: S turns of the warp
    uint4 v[kGatherBatch];
#pragma unroll
    for (int t = 0; t < kGatherBatch; ++t) {
      const int i = (t0 + t) * 32 + lane;
      const bool ok = t0 + t < S && ((i < vecs ? i : i - vecs) >> 4) < valid;
      v[t] = ok ? ldg_nc_v4(src + (long long)i * 8) : zero;
    }
#pragma unroll
    for (int t = 0; t < kGatherBatch; ++t) {
      const int i = (t0 + t) * 32 + lane;
      if (t0 + t < S) *(i < vecs ? kd + i : vd + (i - vecs)) = v[t];
    }
  }
  if (n_tok != nullptr && j == 0 && lane == 0) {
    // sel is ascending, so a partial page can only be the last selected one
    int rows = 0;
    if (ns > 0) {
      const int last = sel[(long long)bh * geo.k + ns - 1];
      rows = ns * S - (last == P - 1 ? S - tail : 0);
    }
    n_tok[bh] = rows;
  }
}

// One warp per (pool page, kv head): lanes 0-15 scan the even tokens, lanes 16-31 the odd tokens,
// each over 8 coordinates; the halves are merged with one shuffle and lanes 0-15 write the 256-byte
// minima row, lanes 16-31 the maxima row.
// Bound by HBM.  The warps of a grid that fills the device once walk the pool in its own order (page, then head), so
// that neighbours read neighbouring blocks, and every warp has eight 512-byte loads in flight.  The minima and maxima are
// taken on pairs of bf16: a block costs a warp about 100 instructions instead of 250, and no registers spill at four CTAs per
// SM.  Summaries and medoid rows of 16 requests of up to 60000 tokens (1061 and 31 MB): 191 us with the values widened to fp32,
// 182 in pairs (the summaries alone at 0.95 of the measured copy bandwidth); five and six CTAs per SM spill, 194 and 258.
__device__ __forceinline__ uint32_t min2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("min.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ uint32_t max2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ void min_max8(const uint4& v, uint32_t (&lo)[4], uint32_t (&hi)[4]) {
  const uint32_t words[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    lo[e] = min2(lo[e], words[e]);
    hi[e] = max2(hi[e], words[e]);
  }
}

constexpr int kSummaryThreads = 256;
__global__ void __launch_bounds__(kSummaryThreads, 4)
summaries_kernel(Geometry geo, const uint16_t* __restrict__ kv_pool, const int64_t* __restrict__ page_base,
                 const int32_t* __restrict__ ctx_len, uint16_t* __restrict__ ksum, uint32_t* __restrict__ status) {
  pdl_wait();                                               // (its launch overlaps what precedes it in the stream)
  pdl_launch_dependents();
  const int lane = threadIdx.x & 31;
  const int S = geo.S;
  if (blockIdx.x == 0) {                                    // lengths that do not fit their pages
    for (int b = threadIdx.x; b < geo.B; b += kSummaryThreads)
      if (ctx_len[b] < 1 || pages_of(ctx_len[b], S) > page_base[b + 1] - page_base[b]) atomicOr(status, SWARM_DEV_BAD_LENGTH);
  }
  const long long first = page_base[0], units = (page_base[geo.B] - first) * geo.Hkv;
  const long long stride = (long long)gridDim.x * (kSummaryThreads / 32);
  long long u = (long long)blockIdx.x * (kSummaryThreads / 32) + (threadIdx.x >> 5);
  long long page = first + u / geo.Hkv;
  int kvh = (int)(u % geo.Hkv);
  const long long step_pages = stride / geo.Hkv;            // (a division per unit costs as much as its arithmetic)
  const int step_heads = (int)(stride % geo.Hkv);
  int b = 0;                                                // request of the unit's page: found once, then carried along
  for (int hi_b = geo.B; hi_b - b > 1;) {
    const int mid = (b + hi_b) / 2;
    if (page_base[mid] <= page) b = mid; else hi_b = mid;
  }
  const int c = lane & 15, half = lane >> 4;
  auto advance = [&]() {
    u += stride;
    page += step_pages;
    kvh += step_heads;
    if (kvh >= geo.Hkv) { kvh -= geo.Hkv; ++page; }
  };
  for (; u < units; advance()) {
    while (b + 1 < geo.B && page_base[b + 1] <= page) ++b;
    const long long base = page_base[b], owned = page_base[b + 1] - base;
    const int len = ctx_len[b], P = pages_of(len, S), p = (int)(page - base);
    if (len < 1 || P > owned || p >= P) continue;
    const int valid = p == P - 1 ? len - S * (P - 1) : S;
    const uint16_t* K = kv_pool + ((page * geo.Hkv + kvh) * 2) * (long long)S * kHeadDim + half * kHeadDim + c * 8;
    uint32_t lo[4], hi[4];                                   // pairs of bf16
#pragma unroll
    for (int e = 0; e < 4; ++e) { lo[e] = 0x7F807F80u; hi[e] = 0xFF80FF80u; }   // +inf, -inf
    for (int t0 = 0; t0 < valid; t0 += 16) {
      uint4 v[8];
      if (t0 + 16 <= valid) {
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = ldg_nc_v4(K + (long long)(t0 + 2 * i) * kHeadDim);
      } else {                                              // the last tokens of a request: the others read the first again
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = ldg_nc_v4(K + (t0 + 2 * i + half < valid ? (long long)(t0 + 2 * i) : -(long long)half) * kHeadDim);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) min_max8(v[i], lo, hi);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      lo[e] = min2(lo[e], __shfl_xor_sync(0xFFFFFFFFu, lo[e], 16));
      hi[e] = max2(hi[e], __shfl_xor_sync(0xFFFFFFFFu, hi[e], 16));
    }
    uint4* dst = reinterpret_cast<uint4*>(ksum + ((page * geo.Hkv + kvh) * 2 + half) * (long long)kHeadDim + c * 8);
    *dst = half ? make_uint4(hi[0], hi[1], hi[2], hi[3]) : make_uint4(lo[0], lo[1], lo[2], lo[3]);
  }
}

}  // namespace

cudaError_t launch_gather(const Geometry& geo, const uint16_t* kv_pool, const int32_t* sel, const int32_t* n_sel,
                          const int64_t* page_base, const int32_t* ctx_len, uint16_t* k_out, uint16_t* v_out,
                          int32_t* n_tok, uint32_t* status, cudaStream_t st) {
  const long long slots = (long long)geo.k * geo.B * geo.Hq;
  const unsigned grid = (unsigned)((slots * 32 + kGatherThreads - 1) / kGatherThreads);
  return launch_pdl(gather_kernel, dim3(grid), dim3(kGatherThreads), 0, st, true, geo, kv_pool, sel, n_sel, page_base, ctx_len, k_out, v_out, n_tok,
                    status);
}

cudaError_t launch_build_summaries(const Geometry& geo, const uint16_t* kv_pool, const int64_t* page_base,
                                   const int32_t* ctx_len, uint16_t* ksum, uint32_t* status, cudaStream_t st) {
  const long long ctas = ((long long)geo.n_pool_pages * geo.Hkv * 32 + kSummaryThreads - 1) / kSummaryThreads;
  const int grid = (int)std::min<long long>(ctas, 4LL * sm_count());   // (the kernel's launch bounds: four per SM)
  return launch_pdl(summaries_kernel, dim3(grid), dim3(kSummaryThreads), 0, st, true, geo, kv_pool, page_base, ctx_len, ksum, status);
}

// Per-step data moved by kernels between the device and host memory the device can address (pinned, unified
// addressing) instead of by copy operations: a copy node between kernels costs several microseconds of
// engine hand-over, a load or store over the bus does not.
//   fetch_kernel    the step's queries, host -> workspace (volatile loads: the host rewrites the buffer between calls)
//   publish_kernel  the step's small results, device -> host; 16-byte vectors for out, words for the rest (used
//                   when the step's last kernel cannot store them itself, see HostMirror)
namespace {
__global__ void __launch_bounds__(256)
fetch_kernel(const uint4* src_h, uint4* __restrict__ dst, int n16) {
  pdl_launch_dependents();                                  // the scorer sets itself up meanwhile
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n16; i += gridDim.x * blockDim.x) {
    uint4 v;
    asm volatile("ld.volatile.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(src_h + i));
    dst[i] = v;
  }
}

__global__ void __launch_bounds__(256)
publish_kernel(const float* __restrict__ out, const float* __restrict__ lse, const int32_t* __restrict__ n_uniq,
               const int32_t* __restrict__ queue_load, float* out_h, float* lse_h, int32_t* n_uniq_h,
               int32_t* queue_load_h, int n_out4, int n_lse, int n_queues) {
  pdl_wait();                                               // the results come from the previous kernel
  const int t = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
  if (out_h != nullptr)
    for (int i = t; i < n_out4; i += stride)
      reinterpret_cast<float4*>(out_h)[i] = __ldcg(reinterpret_cast<const float4*>(out) + i);
  if (lse_h != nullptr)
    for (int i = t; i < n_lse; i += stride) lse_h[i] = __ldcg(lse + i);
  if (queue_load_h != nullptr)
    for (int i = t; i < n_queues; i += stride) queue_load_h[i] = __ldcg(queue_load + i);
  if (n_uniq_h != nullptr && t == 0) *n_uniq_h = __ldcg(n_uniq);
}
}  // namespace

cudaError_t launch_fetch(const void* src_h, void* dst, long long bytes, cudaStream_t st) {
  const int n16 = (int)(bytes / 16);
  const int grid = max(1, min(32, (n16 + 255) / 256));
  fetch_kernel<<<dim3(grid), dim3(256), 0, st>>>(static_cast<const uint4*>(src_h), static_cast<uint4*>(dst), n16);
  return cudaGetLastError();
}

cudaError_t launch_publish(const Geometry& geo, const float* out, const float* lse, const int32_t* n_uniq,
                           const int32_t* queue_load, float* out_h, float* lse_h, int32_t* n_uniq_h,
                           int32_t* queue_load_h, cudaStream_t st) {
  const int n_out4 = geo.B * geo.Hq * kHeadDim / 4;
  const int grid = max(1, min(32, (n_out4 + 255) / 256));
  return launch_pdl(publish_kernel, dim3(grid), dim3(256), 0, st, true, out, lse, n_uniq, queue_load, out_h, lse_h,
                    n_uniq_h, queue_load_h, n_out4, geo.B * geo.Hq, geo.D);
}

}  // namespace swarm
