// Cluster-granular selection through the medoid index (Sec. 4.2, Tier 1 (1)): every cluster is represented
// by its medoid, the medoid is scored against the query, the best clusters are retrieved whole (Sec. 4.1:
// clusters are the retrieval unit) and all of their pages are attended.
//
// The scoring and the top-k are the page kernels run over a context whose "pages" are the clusters: the
// index holds the key summary of each cluster's medoid page, one row per cluster, requests back to back
// exactly like cluster_base.  What this file adds is the glue around them:
//   medoid_rows_kernel     index build: copy the summary rows of the medoid pages into the index, and the pseudo
//                          context lengths (clusters of the request x page size) for the page kernels
//   expand_clusters_kernel (where the selection kernel does not do it itself, see medoid_expand.cuh)
//                          selected clusters -> per-head bitmap of their member pages plus the local window (what
//                          the attention kernel reads) and the cluster flags (what the resolve kernel reads)
#include "medoid_expand.cuh"

namespace swarm {
namespace {

// One warp per cluster: 2 * d bf16 = 512 contiguous bytes per KV head, eight 512-byte rows in flight.  Bound by the chain
// of small loads in front of them (one wave of CTAs at up to 9472 clusters).  The first CTA also writes the pseudo
// lengths.  Launched behind whatever precedes it (in an index build the summaries).
constexpr int kRowThreads = 256;
__global__ void __launch_bounds__(kRowThreads)
medoid_rows_kernel(Geometry geo, const uint16_t* __restrict__ ksum, const int64_t* __restrict__ page_base,
                   const int64_t* __restrict__ cluster_base, const int32_t* __restrict__ medoid_page,
                   uint16_t* __restrict__ medoid_ksum, int32_t* __restrict__ len, uint32_t* __restrict__ status) {
  pdl_wait();
  pdl_launch_dependents();                                  // (behind the wait: the pseudo lengths are read ahead of one)
  if (blockIdx.x == 0)
    for (int b = threadIdx.x; b < geo.B; b += kRowThreads)
      len[b] = (int32_t)min((long long)(cluster_base[b + 1] - cluster_base[b]) * geo.S, 0x7FFFFFFFLL);
  const long long c = (long long)blockIdx.x * (kRowThreads / 32) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (c >= cluster_base[geo.B]) return;
  const int p = medoid_page[c];
  // request of cluster c: the last b with cluster_base[b] <= c, the bases taken 32 at a time
  int b = 0;
  for (int b0 = 0; b0 < geo.B; b0 += 32) {
    const unsigned below = __ballot_sync(0xFFFFFFFFu, b0 + lane < geo.B && cluster_base[b0 + lane] <= c);
    if (below == 0u) break;
    b = b0 + 31 - __clz(below);
  }
  const long long pb = page_base[b];
  const bool ok = p >= 0 && p < page_base[b + 1] - pb;
  if (!ok && lane == 0) atomicOr(status, SWARM_DEV_BAD_PAGE);
  const uint4* src = reinterpret_cast<const uint4*>(ksum + (pb + (ok ? p : 0)) * geo.Hkv * 2 * kHeadDim) + lane;
  uint4* dst = reinterpret_cast<uint4*>(medoid_ksum + c * geo.Hkv * 2 * kHeadDim) + lane;
  for (int h0 = 0; h0 < geo.Hkv; h0 += 8) {
    uint4 v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = ok && h0 + i < geo.Hkv ? src[(h0 + i) * 32] : make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (h0 + i < geo.Hkv) dst[(h0 + i) * 32] = v[i];
  }
}

// One CTA per (request, query head), behind a selection kernel that does not expand its clusters itself.  The head's bitmap row is
// assembled in shared memory (bit p % 8 of byte p / 8, the layout the selection kernel writes) and stored whole, so rows need no
// clearing between steps.
__global__ void __launch_bounds__(256)
expand_clusters_kernel(const ExpandArgs ex, int Hq, int k_c, const int32_t* __restrict__ sel_c, const int32_t* __restrict__ n_sel_c,
                       uint32_t* __restrict__ status) {
  extern __shared__ uint32_t s_row[];
  const int bh = blockIdx.x, b = bh / Hq;
  pdl_launch_dependents();                                  // the attention CTAs set themselves up meanwhile
  const ExpandRequest rq = expand_request(ex, b);          // inputs: read before the wait
  for (int i = threadIdx.x; i < ex.pitch / 4; i += blockDim.x) s_row[i] = 0u;
  pdl_wait();                                               // the cluster selection comes from the previous kernel
  __syncthreads();
  const int32_t* mine = sel_c + (long long)bh * k_c;
  expand_clusters<8>(ex, rq, bh, b, min(n_sel_c[bh], k_c), [&](int j) { return mine[j]; }, s_row, status);
}

}  // namespace

cudaError_t configure_medoid() {
  return cudaFuncSetAttribute(expand_clusters_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxExpandRowBytes);
}

cudaError_t launch_medoid_rows(const Geometry& geo, const uint16_t* ksum, const int64_t* page_base,
                               const int64_t* cluster_base, const int32_t* medoid_page, uint16_t* medoid_ksum,
                               int32_t* len, uint32_t* status, cudaStream_t st) {
  return launch_pdl(medoid_rows_kernel, dim3((unsigned)(((long long)geo.Cmax * 32 + kRowThreads - 1) / kRowThreads)), dim3(kRowThreads), 0, st, true, geo,
                    ksum, page_base, cluster_base, medoid_page, medoid_ksum, len, status);
}

cudaError_t launch_expand_clusters(const ExpandArgs& ex, const Geometry& geo, int k_c, const int32_t* sel_c, const int32_t* n_sel_c, uint32_t* status,
                                   cudaStream_t st, bool overlap) {
  return launch_pdl(expand_clusters_kernel, dim3((unsigned)(geo.B * geo.Hq)), dim3(256), (size_t)ex.pitch, st, overlap, ex, geo.Hq, k_c, sel_c,
                    n_sel_c, status);
}

}  // namespace swarm
