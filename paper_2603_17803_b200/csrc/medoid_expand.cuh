// Selected clusters of one head -> the head's page bitmap and the cluster flags, by all threads of a CTA (Sec. 4.1: clusters are the
// retrieval unit).  Two kernels run it: the selection kernel behind its own selection, where the list of clusters and the bitmap
// row fit its shared memory, and expand_clusters_kernel.
#pragma once
#include "swarm_internal.cuh"

namespace swarm {

// What a head's request looks like; inputs, read before the CTA waits for the selection.
struct ExpandRequest {
  int P;
  long long cb, cn;
};
__device__ __forceinline__ ExpandRequest expand_request(const ExpandArgs& ex, int b) {
  return {pages_of(ex.ctx_len[b], ex.S), ex.cluster_base[b], ex.cluster_base[b + 1]};
}

// cluster_at(j), j < n: the selected clusters (request-local).  s_row: the bitmap row, pitch / 4 words, zeroed (a barrier later).
// kLanes lanes per selected cluster: every cluster costs two dependent trips to memory (its member range, its members), and
// with a warp per cluster four clusters of a warp paid them one after another (7 of the step's 60 us; 32 clusters per head).
template <int kLanes, class F>
__device__ __forceinline__ void expand_clusters(const ExpandArgs& ex, const ExpandRequest& rq, int bh, int b, int n, F cluster_at, uint32_t* s_row,
                                                uint32_t* __restrict__ status) {
  const int tid = threadIdx.x, sub = tid & (kLanes - 1), P = rq.P, pitch = ex.pitch;
  unsigned err = 0u;
  for (int j = tid / kLanes; j < n; j += blockDim.x / kLanes) {
    const int c = cluster_at(j);
    if (c < 0 || c >= rq.cn - rq.cb || rq.cb + c >= ex.Cmax) { err |= SWARM_DEV_BAD_CLUSTER; continue; }
    const long long e0 = ex.cluster_page_ptr[rq.cb + c], e1 = ex.cluster_page_ptr[rq.cb + c + 1];
    if (e0 < 0 || e1 < e0 || e1 > ex.n_member_entries) { err |= SWARM_DEV_BAD_CLUSTER; continue; }   // corrupt member offsets
    // what gets scheduled: the cluster as a whole, or (entry level) each of its pages on its own
    if (sub == 0 && ex.entry_base == nullptr) ex.flags[rq.cb + c] = 1;
    for (long long e = e0 + sub; e < e1; e += 2 * kLanes) {
      int page[2] = {ex.cluster_pages[e], e + kLanes < e1 ? ex.cluster_pages[e + kLanes] : -1};   // both in flight
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int p = page[u];
        if (u == 1 && e + kLanes >= e1) break;
        if (p < 0 || p >= P || p >= pitch * 8) {
          err |= SWARM_DEV_BAD_PAGE;
        } else {
          atomicOr(&s_row[p >> 5], 1u << (p & 31));
          if (ex.entry_base != nullptr) {
            const long long unit = ex.entry_base[b] + p;
            if (unit < ex.Cmax) ex.flags[unit] = 1;
            else err |= SWARM_DEV_BAD_CLUSTER;
          }
        }
      }
    }
  }
  // the local window (Sec. 4.2, Tier 1 (2)): the last W pages of the request join every head's set and are
  // scheduled like the members of the selected clusters
  for (int p = max(0, P - ex.W) + tid; p < P && p < pitch * 8; p += blockDim.x) {
    atomicOr(&s_row[p >> 5], 1u << (p & 31));
    if (ex.entry_base != nullptr) {
      const long long unit = ex.entry_base[b] + p;
      if (unit < ex.Cmax) ex.flags[unit] = 1;
      else err |= SWARM_DEV_BAD_CLUSTER;
    } else {
      const int c = ex.page2cluster[ex.page_base[b] + p];
      if (c < 0 || c >= rq.cn - rq.cb || rq.cb + c >= ex.Cmax) err |= SWARM_DEV_BAD_CLUSTER;
      else ex.flags[rq.cb + c] = 1;
    }
  }
  if (err) atomicOr(status, err);
  __syncthreads();
  uint32_t* row = reinterpret_cast<uint32_t*>(ex.selmap + (long long)bh * pitch);
  for (int i = tid; i < pitch / 4; i += blockDim.x) row[i] = s_row[i];
}

}  // namespace swarm
