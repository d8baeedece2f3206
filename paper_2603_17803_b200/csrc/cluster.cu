// Algorithm 1: offline co-activation clustering on a given distance matrix (Sec. 4.1, Steps 3 and 4).
//
//   density_kernel   rho[i] = #{ j != i : D[i][j] <= tau } -- one warp per row, 16-byte loads; the only pass over the
//                    whole n x n matrix, bound by HBM bandwidth (4 n^2 bytes read once)
//   rounds_kernel    everything else in one cooperative launch
//
// The listing walks the entries by (rho descending, index ascending) and grows a cluster from every entry that no
// earlier cluster has covered.  What a cluster contains depends on its medoid and the matrix alone (covered entries
// remain candidates, which is where the paper's replicas come from), so clusters can be grown before it is known
// whether the walk will want them.  The kernel works in rounds: the next uncovered entries of the walk, one per CTA, are
// all grown side by side, and each CTA notes which of the round's entries its cluster holds.  Behind a barrier every CTA
// repeats the walk over those notes (a few hundred bits per step), which settles who is a medoid, and the medoids' CTAs
// write their clusters to their final places.  Clusters that the walk does not want are dropped: they cost SMs that had
// nothing else to do.  8192 entries in 64 topics: 102 clusters in 5 rounds.
//
// Growing one cluster: the candidates are sorted by (distance, index) in shared memory and visited in that order; one
// joins when its running sum is within tau * |C|.  A CTA does this 32 candidates at a time, a thread per candidate: the
// warp that owns the 32 decides them one after the other (a ballot and an add per join, operands in a tile in shared memory), the
// others then add the rows of those that joined.  The matrix entries a thread will need for the next 32 are loaded while
// the present ones are decided.  Bound by those gathers: n_c^2 / 2 scattered words per cluster of n_c candidates, about
// one 32-byte sector per two cycles and SM.  (As a walk that went to memory for every join it took 1.3 us per join.)  Lists
// that hold much of the matrix take whole rows instead.
// A candidate's sum is a plain fp32 accumulation in joining order over D[member][candidate], so every decision is the
// one a sequential fp32 walk takes.
#include "swarm_internal.cuh"

#include <algorithm>
#include <type_traits>

namespace swarm {
namespace {

struct ClusterArgs {
  const float* dist;
  int n;
  float tau;
  int32_t* rho;
  // scratch (see build_clusters_workspace_bytes)
  int32_t* queue;        // [n] entries in the order of the walk
  int32_t* place;        // [n] and back: where an entry stands in it
  uint32_t* covered;     // bit p: the entry at place p is covered
  uint32_t* holds;       // [grid][kNoteWords] bit j of row i: the cluster grown by CTA i holds the round's entry j
  int32_t* size;         // [grid] its size
  unsigned* ctl;         // kCtl* below
  // outputs
  int32_t* ptr;
  int32_t* members;
  long long members_cap;
  int32_t* medoid;
  int32_t* n_clusters;
  int32_t* dev_status;   // 0 ok, 1 members_cap too small, 2 a bounded wait ran out
};
constexpr int kCtlArrived = 0, kCtlFailed = 1, kCtlWords = 64;
constexpr int kMaxPicks = 256;                            // entries grown per round: one per CTA
constexpr int kNoteWords = kMaxPicks / 32;
__host__ __device__ inline int bit_words(int n) { return (n + 31) / 32; }

__global__ void __launch_bounds__(256) density_kernel(ClusterArgs a) {
  const int lane = threadIdx.x & 31, n = a.n;
  if (blockIdx.x == 0 && threadIdx.x < kCtlWords) a.ctl[threadIdx.x] = 0u;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < bit_words(n); i += gridDim.x * blockDim.x) a.covered[i] = 0u;
  const int row = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
  if (row >= n) return;
  const float* r = a.dist + (long long)row * n;
  int cnt = 0;
  if ((n & 3) == 0) {                                     // rows are 16-byte aligned
#pragma unroll 4
    for (int j = lane * 4; j < n; j += 128) {
      const uint4 v = ldg_nc_v4(r + j);
      cnt += (__uint_as_float(v.x) <= a.tau && j != row) + (__uint_as_float(v.y) <= a.tau && j + 1 != row) +
             (__uint_as_float(v.z) <= a.tau && j + 2 != row) + (__uint_as_float(v.w) <= a.tau && j + 3 != row);
    }
  } else {
#pragma unroll 4
    for (int j = lane; j < n; j += 32) cnt += (__ldg(r + j) <= a.tau && j != row);
  }
  cnt = __reduce_add_sync(0xFFFFFFFFu, cnt);
  if (lane == 0) a.rho[row] = cnt;
}

// ---- rounds ----------------------------------------------------------------------------------------------------
// 384 threads: with 512 the two blocks of operands that a thread holds spill (36 against 32 us for the largest clusters of
// 8192 entries in 64 topics); more candidates than threads are rare and kept in shared memory.
constexpr int kRoundThreads = 384, kRoundWarps = kRoundThreads / 32;
constexpr int kCountedCand = 1024;                        // up to here candidates are sorted by counting
constexpr unsigned kGridWaitLimit = 1u << 23;

// Order-preserving key of a distance (-0 folded onto +0) and back.
__device__ __forceinline__ uint32_t dist_key(float d) {
  uint32_t u = __float_as_uint(d);
  if (u == 0x80000000u) u = 0u;
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_dist(uint32_t k) { return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k); }

struct RoundShared {
  int warp_tot[kRoundWarps];
  int n_cand, failed;
  int my_clu;                                             // where this CTA's cluster goes, -1: nowhere
  long long my_fill;
  int pick[kMaxPicks];                                    // the round's entries, in the order of the walk
  int pick_size[kMaxPicks];
  uint32_t holds[kMaxPicks][kNoteWords];
  uint32_t taken[kNoteWords];                             // the medoids among them
  uint32_t joined[1024];                                  // bit k of word b: candidate 32 b + k is a member
  uint32_t likely[kRoundWarps];                           // candidates of the first 384 whose rows are worth loading ahead
};

// Exclusive prefix of v over the CTA and the total (two barriers).
__device__ __forceinline__ int block_prefix(RoundShared& sh, int v, int& total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += t;
  }
  __syncthreads();
  if (lane == 31) sh.warp_tot[warp] = incl;
  __syncthreads();
  int before = 0;
  total = 0;
#pragma unroll
  for (int w = 0; w < kRoundWarps; ++w) {
    if (w < warp) before += sh.warp_tot[w];
    total += sh.warp_tot[w];
  }
  return before + incl - v;
}

// Every CTA of the (cooperative) grid has arrived for the nth time; false when that wait ran out.
__device__ __forceinline__ void grid_arrive(const ClusterArgs& a) {
  __syncthreads();
  if (threadIdx.x == 0) red_release_add(a.ctl + kCtlArrived, 1u);
}
__device__ __forceinline__ bool grid_wait(const ClusterArgs& a, RoundShared& sh, unsigned nth) {
  if (threadIdx.x == 0) {
    unsigned* p = a.ctl + kCtlArrived;
    const unsigned target = nth * gridDim.x;
    unsigned polls = 0, v = 0;
    do {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    } while ((int)(v - target) < 0 && ++polls < kGridWaitLimit);
    if ((int)(v - target) < 0) atomicExch(a.ctl + kCtlFailed, 1u);
    if (*reinterpret_cast<volatile unsigned*>(a.ctl + kCtlFailed) != 0u) sh.failed = 1;
  }
  __syncthreads();
  return sh.failed == 0;
}

// Ascending bitonic sort of (key, index) pairs, `m` a power of two.
__device__ __forceinline__ void sort_pairs(uint32_t* key, uint16_t* idx, int m) {
  for (int k = 2; k <= m; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      __syncthreads();
      for (int t = threadIdx.x; t < m / 2; t += kRoundThreads) {
        const int lo = ((t & ~(j - 1)) << 1) | (t & (j - 1)), hi = lo | j;
        const uint32_t ka = key[lo], kb = key[hi];
        const uint16_t ia = idx[lo], ib = idx[hi];
        const bool after = ka > kb || (ka == kb && ia > ib);
        if (after == ((lo & k) == 0)) { key[lo] = kb; key[hi] = ka; idx[lo] = ib; idx[hi] = ia; }
      }
    }
  }
  __syncthreads();
}

// One thread's operands for the 32 candidates of block b: value k is D[row of candidate 32 b + k][entry c], loaded for
// the candidates in `want` that stand in front of candidate i (the ones this thread's sum can still need).
__device__ __forceinline__ void load_block(const ClusterArgs& a, const uint16_t* idx, int b, uint32_t want, int i, int c, float (&val)[32]) {
  const uint4* rows = reinterpret_cast<const uint4*>(idx + 32 * b);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const uint4 r = rows[q];                              // eight 16-bit entries
    const uint32_t words[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int h = 0; h < 8; ++h) {
      const int k = 8 * q + h;
      const uint32_t e = (h & 1) ? words[h >> 1] >> 16 : words[h >> 1] & 0xFFFFu;
      val[k] = (((want >> k) & 1u) && 32 * b + k < i) ? __ldg(a.dist + (long long)e * a.n + c) : 0.f;
    }
  }
}

// Grows the cluster of medoid m (all threads of the CTA).  Returns its size; its members behind the medoid are the
// candidates whose bits are set in sh.joined, and a bit each in `mark`.  `smem`: the CTA's dynamic shared memory.
__device__ int grow(const ClusterArgs& a, RoundShared& sh, unsigned char* smem, int cap, int m, uint32_t* mark) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = a.n;
  const float* row_m = a.dist + (long long)m * n;
  const int n_cand = a.rho[m];
  const bool counted = n_cand <= kCountedCand;
  uint32_t* key = reinterpret_cast<uint32_t*>(smem);      // [cap] distance keys; then the running sums; then the members
  uint16_t* idx = reinterpret_cast<uint16_t*>(smem + cap * 4);           // [cap] entries
  uint32_t* raw_key = reinterpret_cast<uint32_t*>(smem + cap * 6);       // as collected, if counted
  uint32_t* raw_entry = raw_key + kCountedCand;
  static_assert(kCountedCand >= 1024, "32 x 32 operands take its place, the marks of 32768 entries the keys'");

  // ---- candidates in any order ----
  if (tid == 0) sh.n_cand = 0;
  __syncthreads();
  // (whole warps; each thread's are counted first, so that a warp asks for room once)
  auto append = [&](uint32_t mask, auto entry_of, auto dist_of, auto count) {
    int before = __popc(mask);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xFFFFFFFFu, before, o);
      if (lane >= o) before += t;
    }
    int at = 0;
    if (lane == 31 && before > 0) at = atomicAdd(&sh.n_cand, before);
    at = __shfl_sync(0xFFFFFFFFu, at, 31) + before - __popc(mask);
    if (mask == 0u) return;
#pragma unroll
    for (int u = 0; u < decltype(count)::value; ++u) {
      if (((mask >> u) & 1u) && at < n_cand) {
        const uint32_t k = dist_key(dist_of(u));
        if (counted) { raw_key[at] = k; raw_entry[at] = (uint32_t)entry_of(u); }
        else { key[at] = k; idx[at] = (uint16_t)entry_of(u); }
        ++at;
      }
    }
  };
  if ((n & 3) == 0) {
    for (int j0 = 4 * tid; j0 < (n + 127 & ~127); j0 += kRoundThreads * 24) {   // (a warp's 32 threads together)
      float v[24];
#pragma unroll
      for (int u = 0; u < 6; ++u) {                       // six loads in flight
        const int j = j0 + u * kRoundThreads * 4;
        const float4 f = j < n ? __ldg(reinterpret_cast<const float4*>(row_m + j)) : make_float4(0.f, 0.f, 0.f, 0.f);
        v[4 * u] = f.x; v[4 * u + 1] = f.y; v[4 * u + 2] = f.z; v[4 * u + 3] = f.w;
      }
      auto entry_of = [&](int u) { return j0 + (u >> 2) * kRoundThreads * 4 + (u & 3); };
      uint32_t mask = 0u;
#pragma unroll
      for (int u = 0; u < 24; ++u) mask |= (v[u] <= a.tau && entry_of(u) < n && entry_of(u) != m ? 1u : 0u) << u;
      append(mask, entry_of, [&](int u) { return v[u]; }, std::integral_constant<int, 24>());
    }
  } else {
    for (int j0 = tid; j0 < (n + 31 & ~31); j0 += kRoundThreads) {
      const float v = j0 < n ? __ldg(row_m + j0) : 0.f;
      append(j0 < n && v <= a.tau && j0 != m ? 1u : 0u, [&](int) { return j0; }, [&](int) { return v; }, std::integral_constant<int, 1>());
    }
  }
  __syncthreads();
  // ---- sorted by (distance, index) ----
  if (counted) {
    // Each candidate's place by counting the keys up to its own, four lanes per candidate.  Equal keys land on one place
    // and leave another unfilled; then the count is repeated with the entries in it.
    const int padded = (n_cand + 15) & ~15;
    for (int i = n_cand + tid; i < padded; i += kRoundThreads) raw_key[i] = 0xFFFFFFFFu;
    for (int i = tid; i < n_cand; i += kRoundThreads) idx[i] = 0xFFFFu;
    __syncthreads();
    auto place = [&](bool ties) {
      for (int t0 = 0; t0 < 4 * n_cand; t0 += kRoundThreads) {
        const int i = (t0 + tid) >> 2, part = tid & 3;
        const uint32_t mine = i < n_cand ? raw_key[i] : 0u, e = i < n_cand ? raw_entry[i] : 0u;
        int at = 0;
#pragma unroll 4
        for (int j = 4 * part; j < padded; j += 16) {
          const uint4 k = *reinterpret_cast<const uint4*>(raw_key + j);
          at += (k.x <= mine) + (k.y <= mine) + (k.z <= mine) + (k.w <= mine);
          if (ties) {
            const uint4 o = *reinterpret_cast<const uint4*>(raw_entry + j);
            at -= (k.x == mine && o.x > e) + (k.y == mine && o.y > e) + (k.z == mine && o.z > e) + (k.w == mine && o.w > e);
          }
        }
        at += __shfl_xor_sync(0xFFFFFFFFu, at, 1);
        at += __shfl_xor_sync(0xFFFFFFFFu, at, 2);
        if (part == 0 && i < n_cand) { key[at - 1] = mine; idx[at - 1] = (uint16_t)e; }
      }
      __syncthreads();
    };
    place(false);
    bool open = false;
    for (int i = tid; i < n_cand; i += kRoundThreads) open = open || idx[i] == 0xFFFFu;
    if (__syncthreads_or(open)) place(true);
  } else {
    int m2 = 1;
    while (m2 < n_cand) m2 <<= 1;
    for (int i = n_cand + tid; i < m2; i += kRoundThreads) { key[i] = 0xFFFFFFFFu; idx[i] = 0xFFFFu; }
    sort_pairs(key, idx, m2);
  }

  // ---- the walk over the candidates, 32 at a time ----
  const int blocks = (n_cand + 31) / 32;
  // Candidate t's sum lies in a register of thread t; candidates from kRoundThreads on have theirs in shared memory.
  const float kNever = __int_as_float(0x7FFFFFFF);        // no candidate: NaN passes no bound
  for (int i = n_cand + tid; i < 32 * blocks; i += kRoundThreads) idx[i] = (uint16_t)m;
  float s = tid < n_cand ? key_dist(key[tid]) : kNever;
  if (tid < kRoundWarps) sh.likely[tid] = 0xFFFFFFFFu;
  for (int w = tid; w < bit_words(n); w += kRoundThreads) mark[w] = 0u;   // (where the collected candidates were)
  __syncthreads();
  const int c0 = tid < 32 * blocks ? idx[tid] : m;
  float* tile = reinterpret_cast<float*>(raw_entry);      // the operands of the block being decided
  int size = 1;
  // Block b's members, by the warp that holds the sums x of its candidates and their operands val.
  auto decide = [&](int b, float x, float (&val)[32]) {
    // A link of the chain is a load from shared memory, an add, a compare and a ballot, and there is one per member:
    // candidates that no join lets in are passed over on the ballot of the last one.  (Unrolled over the 32 registers
    // the warp waited for instructions: 2900 cycles per 32 candidates.)
#pragma unroll
    for (int k = 0; k < 32; ++k) tile[32 * k + lane] = val[k];
    uint32_t joined = 0u, above = 0xFFFFFFFFu;
    float members = (float)size + 1.f, bound = a.tau * (float)size, next = a.tau * members;
    for (;;) {
      const uint32_t pass = __ballot_sync(0xFFFFFFFFu, x <= bound) & above;
      if (pass == 0u) break;
      const int k = __ffs(pass) - 1;
      const float v = tile[32 * k + lane];                // (written by this lane)
      joined |= 1u << k;
      above = 0xFFFFFFFEu << k;
      x += v;                                             // (of no account for the lanes up to k)
      bound = next;
      members += 1.f;
      next = a.tau * members;
    }
    if (lane == 0) sh.joined[b] = joined;
  };
  float cur[32], nxt[32];
  uint32_t cur_have = 0u, nxt_have = 0u;                  // rows loaded (a row is left out while its candidate looks hopeless)
  const int first = min(blocks, kRoundWarps);             // blocks in registers
  auto fetch = [&](int b, float (&val)[32], uint32_t& loaded) {
    loaded = 0u;
    if (b < first && warp >= b && warp < first) {
      loaded = warp == b ? 0xFFFFFFFFu : *reinterpret_cast<volatile uint32_t*>(&sh.likely[b]);
      load_block(a, idx, b, loaded, tid, c0, val);
    }
  };
  auto step = [&](int b, float (&val)[32], uint32_t loaded) {
    if (warp == b) decide(b, s, val);
    __syncthreads();
    const uint32_t joined = sh.joined[b];
    size += __popc(joined);
    if (warp > b && warp < first) {                       // the sums of the candidates behind the block
      uint32_t late = joined & ~loaded;
      while (late) {                                      // (joined against expectation: loaded now)
        const int k = __ffs(late) - 1;
        late &= late - 1u;
        const float v = __ldg(a.dist + (long long)idx[32 * b + k] * n + c0);
#pragma unroll
        for (int q = 0; q < 32; ++q) if (q == k) val[q] = v;
      }
#pragma unroll
      for (int k = 0; k < 32; ++k) if ((joined >> k) & 1u) s += val[k];
      const unsigned hint = __ballot_sync(0xFFFFFFFFu, s <= 1.25f * a.tau * (float)size);
      if (lane == 0) sh.likely[warp] = hint;              // an average a quarter above the radius is not about to join
    }
  };

  // ---- the candidates behind those ----
  // A member costs the remaining candidates a gather of a 32-byte sector each, or all entries its whole row, n / 8 sectors
  // in order: rows while more than an eighth of the matrix remains, on sums that lie by entry then.  (Gathers alone against
  // this: one cluster of 8192 entries 22.9 and 7.4 ms, of 16384 entries 259 and 29, 8192 entries in 8 topics 3.05 and
  // 3.13.  A quarter as the line: 24000 entries in 8 topics 62 -> 129 ms; a sixteenth: 8192 in 16 topics 0.93 -> 1.14.)
  float* sum = reinterpret_cast<float*>(key);
  const bool more = n_cand > kRoundThreads;
  auto rows_pay = [&](int b) { return 8 * (n_cand - max(32 * (b + 1), kRoundThreads)) > n; };
  const bool by_entry = more && rows_pay(0);
  if (by_entry) {                                         // (all keys that are still wanted have been read)
    for (int e = tid; e < n; e += kRoundThreads) sum[e] = __ldg(row_m + e);
  } else {
    for (int i = tid + kRoundThreads; i < n_cand; i += kRoundThreads) sum[i] = key_dist(key[i]);   // (thread i mod 384, as below)
  }
  auto fetch_tile = [&](int b) {                          // by the warp that decides block b, a block ahead
    if (b < blocks && warp == b % kRoundWarps) load_block(a, idx, b, 0xFFFFFFFFu, 32 * b + lane, idx[32 * b + lane], cur);
  };
  // block b's members join the sums
  auto add = [&](int b) {
    const uint32_t joined = sh.joined[b];
    if (joined == 0u) return;
    if (rows_pay(b)) {
      for (int e0 = tid; e0 < n; e0 += 4 * kRoundThreads) {
        float x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = e0 + u * kRoundThreads < n ? sum[e0 + u * kRoundThreads] : 0.f;
        for (uint32_t todo = joined; todo != 0u;) {
          float v[8][4];                                  // eight rows by four entries in flight, added in joining order
#pragma unroll
          for (int r = 0; r < 8; ++r) {
            const bool has = todo != 0u;
            const float* row = a.dist + (long long)idx[32 * b + (has ? __ffs(todo) - 1 : 0)] * n;
            todo &= todo - 1u;                            // 0 stays 0
#pragma unroll
            for (int u = 0; u < 4; ++u)
              v[r][u] = has && e0 + u * kRoundThreads < n ? __ldg(row + e0 + u * kRoundThreads) : 0.f;
          }
#pragma unroll
          for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int u = 0; u < 4; ++u) x[u] += v[r][u];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) if (e0 + u * kRoundThreads < n) sum[e0 + u * kRoundThreads] = x[u];
      }
    } else {
      for (int i = tid + kRoundThreads; i < n_cand; i += kRoundThreads) {
        if (i < 32 * (b + 1)) continue;
        const int c = idx[i], at = by_entry ? c : i;
        float v[32], x = sum[at];
        load_block(a, idx, b, joined, i, c, v);
#pragma unroll
        for (int k = 0; k < 32; ++k) if ((joined >> k) & 1u) x += v[k];
        sum[at] = x;
      }
    }
  };

  fetch(0, cur, cur_have);
  for (int b = 0; b < first; b += 2) {
    fetch(b + 1, nxt, nxt_have);
    step(b, cur, cur_have);
    if (b + 1 >= first) break;
    fetch(b + 2, cur, cur_have);
    step(b + 1, nxt, nxt_have);
    if (more) {                                           // (fills the wait for the next block's operands)
      for (int q = b; q < b + 2; ++q) add(q);
    }
  }
  if (more) {
    fetch_tile(kRoundWarps);
    for (int b = kRoundWarps; b < blocks; ++b) {
      if (by_entry) __syncthreads();                      // (rows leave an entry's sum with another thread than gathers and decisions)
      if (warp == b % kRoundWarps) {
        const int i = 32 * b + lane;                      // this lane's candidate
        decide(b, i < n_cand ? sum[by_entry ? idx[i] : i] : kNever, cur);
      }
      __syncthreads();
      size += __popc(sh.joined[b]);
      fetch_tile(b + 1);
      add(b);
    }
  }
  __syncthreads();
  for (int i = tid; i < n_cand; i += kRoundThreads)
    if ((sh.joined[i >> 5] >> (i & 31)) & 1u) atomicOr(&mark[idx[i] >> 5], 1u << (idx[i] & 31));
  __syncthreads();
  return size;
}

// The members of the cluster grown last behind its medoid: member i >= 1 is list[i] (shared memory, the sums' place).
__device__ const uint16_t* list_members(RoundShared& sh, unsigned char* smem, int cap, int n_cand) {
  uint16_t* list = reinterpret_cast<uint16_t*>(smem);
  const uint16_t* idx = reinterpret_cast<const uint16_t*>(smem + cap * 4);
  const int blocks = (n_cand + 31) / 32;
  int at = 1;
  for (int b0 = 0; b0 < blocks; b0 += kRoundThreads) {    // (at most three turns)
    const int b = b0 + threadIdx.x;
    uint32_t j = b < blocks ? sh.joined[b] : 0u;
    int total;
    int p = at + block_prefix(sh, __popc(j), total);
    for (; j; j &= j - 1u) list[p++] = idx[32 * b + __ffs(j) - 1];
    at += total;
  }
  __syncthreads();
  return list;
}

__global__ void __launch_bounds__(kRoundThreads, 1) rounds_kernel(ClusterArgs a, int cap) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ RoundShared sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = a.n, bwords = bit_words(n), G = gridDim.x, me = blockIdx.x;
  if (tid == 0) sh.failed = 0;
  if (me == 0 && tid == 0) a.ptr[0] = 0;

  // ---- the order of the walk: places by counting ----
  // Every CTA counts the entries of each density, those in front of its own stretch of entries apart (two counts to a word), and
  // adds up the denser ones; an entry's place is what is denser, what is as dense in front of the stretch, and what is as dense
  // in front of it inside the stretch.  Bound by barriers and the atomics on a few popular counts.  (8192 entries: 7 us; comparing every
  // entry with every other, 12 us.  The whole call, both in turn three times: 8192 entries in 128 topics 264-269 -> 255-256, 16384 in 128
  // 622 -> 597, 32768 in 256 1885 -> 1758; 3911 entries and fewer take the same time either way.)
  {
    uint32_t* hist = reinterpret_cast<uint32_t*>(dyn);     // [n] by n - 1 - density: all entries << 16 | those in front of the stretch
    const int stretch = (n + G - 1) / G, first = min(n, me * stretch), last = min(n, first + stretch);
    for (int i = tid; i < n; i += kRoundThreads) hist[i] = 0u;
    __syncthreads();
#pragma unroll 6
    for (int i = 4 * tid; i < n; i += 4 * kRoundThreads) {
      int r[4];
      if (i + 4 <= n) {
        const int4 v = *reinterpret_cast<const int4*>(a.rho + i);
        r[0] = v.x; r[1] = v.y; r[2] = v.z; r[3] = v.w;
      } else {
        for (int j = 0; j < 4; ++j) r[j] = i + j < n ? a.rho[i + j] : -1;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (r[j] >= 0) atomicAdd(&hist[n - 1 - r[j]], i + j < first ? 0x10001u : 0x10000u);
    }
    __syncthreads();
    const int per = (n + kRoundThreads - 1) / kRoundThreads, b0 = min(n, tid * per), b1 = min(n, b0 + per);
    int sum = 0, total;
    for (int i = b0; i < b1; ++i) sum += (int)(hist[i] >> 16);
    int run = block_prefix(sh, sum, total);
    for (int i = b0; i < b1; ++i) {
      const uint32_t h = hist[i];
      hist[i] = (uint32_t)run + (h & 0xFFFFu);
      run += (int)(h >> 16);
    }
    __syncthreads();
    for (int e = first + tid; e < last; e += kRoundThreads) {
      const int r = a.rho[e];
      int p = (int)hist[n - 1 - r];
      for (int j = first; j < e; ++j) p += a.rho[j] == r;
      a.queue[p] = e;
      a.place[e] = p;
    }
  }
  unsigned nth = 0;
  grid_arrive(a);
  bool fine = grid_wait(a, sh, ++nth);
  int n_clu = 0, from = 0, status = 0;                     // clusters written; bitmap words before `from` are all covered
  long long fill = 0;

  while (fine) {
    // ---- the round's entries: the first G uncovered ones ----
    int n_picks = 0;
    for (int w0 = from; w0 < bwords && n_picks < G; w0 += kRoundThreads) {
      const int w = w0 + tid;
      uint32_t b = 0u;
      if (w < bwords) b = (w * 32 + 32 <= n ? 0xFFFFFFFFu : (1u << (n - w * 32)) - 1u) & ~__ldcg(a.covered + w);
      int total;
      int rank = n_picks + block_prefix(sh, __popc(b), total);
      for (; b && rank < G; b &= b - 1u, ++rank) sh.pick[rank] = w * 32 + __ffs(b) - 1;
      n_picks = min(G, n_picks + total);
    }
    __syncthreads();
    if (tid < n_picks) sh.pick[tid] = __ldcg(a.queue + sh.pick[tid]);   // (places first: their entries in one trip)
    __syncthreads();
    if (n_picks == 0) break;                               // (uniform over the grid: nobody covers before the next barrier)
    // ---- every CTA grows one and notes which of the others its cluster holds ----
    int size = 0;
    const uint16_t* members = nullptr;
    if (me < n_picks) {
      const int m = sh.pick[me];
      uint32_t* mark = reinterpret_cast<uint32_t*>(dyn + cap * 6);
      size = grow(a, sh, dyn, cap, m, mark);
      if (tid < kMaxPicks) {
        const int e = tid < n_picks ? sh.pick[tid] : m;
        const uint32_t w = __ballot_sync(0xFFFFFFFFu, tid < n_picks && ((mark[e >> 5] >> (e & 31)) & 1u));
        if (lane == 0) a.holds[me * kNoteWords + warp] = w;
      }
      if (tid == 0) a.size[me] = size;
    }
    grid_arrive(a);
    if (me < n_picks) members = list_members(sh, dyn, cap, a.rho[sh.pick[me]]);
    if (!(fine = grid_wait(a, sh, ++nth))) break;
    // ---- the walk over them ----
    for (int i = tid; i < n_picks * kNoteWords; i += kRoundThreads) (&sh.holds[0][0])[i] = __ldcg(a.holds + i);
    if (tid < n_picks) sh.pick_size[tid] = __ldcg(a.size + tid);
    __syncthreads();
    if (warp == 0) {
      // lane w: word w of the entries still in the walk, and of the ones taken
      uint32_t open = lane * 32 < n_picks ? (lane * 32 + 32 <= n_picks ? 0xFFFFFFFFu : (1u << (n_picks & 31)) - 1u) : 0u, taken = 0u;
      for (;;) {
        const int i = __reduce_min_sync(0xFFFFFFFFu, open ? lane * 32 + __ffs(open) - 1 : kMaxPicks);
        if (i >= n_picks) break;
        if (lane == (i >> 5)) { taken |= 1u << (i & 31); open &= ~(1u << (i & 31)); }
        if (lane < kNoteWords) open &= ~sh.holds[i][lane];
      }
      if (lane < kNoteWords) sh.taken[lane] = taken;
    }
    __syncthreads();
    // ---- where the taken ones go ----
    const bool is = tid < n_picks && ((sh.taken[tid >> 5] >> (tid & 31)) & 1u);
    int n_taken, n_members;
    const int clu = n_clu + block_prefix(sh, is, n_taken);
    const int at = block_prefix(sh, is ? sh.pick_size[tid] : 0, n_members);
    const bool fits = is && fill + at + sh.pick_size[tid] <= a.members_cap;   // the first that does not fit ends the output
    if (tid == me) { sh.my_clu = fits ? clu : -1; sh.my_fill = fill + at; }
    const int n_fit = __syncthreads_count(fits);
    status = n_fit < n_taken;
    n_clu += n_fit;
    fill += n_members;
    const int my_clu = me < n_picks ? sh.my_clu : -1;
    const long long my_fill = sh.my_fill;
    if (my_clu >= 0) {
      const int m = sh.pick[me];
      if (tid == 0) {
        a.medoid[my_clu] = m;
        a.ptr[my_clu + 1] = (int32_t)(my_fill + size);
        a.members[my_fill] = m;
        const int p = a.place[m];
        atomicOr(a.covered + (p >> 5), 1u << (p & 31));
      }
      for (int i = 1 + tid; i < size; i += kRoundThreads) {
        const int e = members[i], p = a.place[e];
        a.members[my_fill + i] = e;
        atomicOr(a.covered + (p >> 5), 1u << (p & 31));
      }
    }
    if (status != 0) break;                                // (uniform over the grid)
    grid_arrive(a);
    fine = grid_wait(a, sh, ++nth);
    from = __ldcg(a.place + sh.pick[0]) >> 5;              // everything in front of this round's first entry is covered
  }
  if (me == 0 && tid == 0) {
    *a.n_clusters = fine ? n_clu : 0;
    *a.dev_status = fine ? status : 2;
  }
}

}  // namespace

// ---- admission to the fast tier (Sec. 4.2, Tier 1 (3)): clusters in descending Eq. 6 score while they fit -------
namespace {

constexpr int kAdmitThreads = 1024;
constexpr int kAdmitBins = 4096;
constexpr int kAdmitDigit = 12;

// The admitted set is everything above a threshold score plus, in index order, the first clusters at it, so nothing has
// to be sorted: a radix select whose bins hold pages instead of counts finds the score at which the running page count
// leaves the capacity (12-bit digits relative to the scores' own range), an ordered scan the place inside its ties.
// One CTA; latency-bound, n * 4 bytes from L2 per level.  (A full sort by counting took n^2 compares: 84 + 20 us at
// 7 K clusters.)
__global__ void __launch_bounds__(kAdmitThreads)
admit_kernel(const float* __restrict__ score, const uint16_t* __restrict__ size, int n, long long capacity,
             uint8_t* __restrict__ resident, int32_t* __restrict__ info) {
  __shared__ uint32_t hist[kAdmitBins];                    // pages per digit (at most 65536 * 65535 in all)
  __shared__ uint32_t s_warp[32], s_lo[32], s_hi[32];
  __shared__ uint32_t s_base;
  __shared__ int s_bits, s_all, s_admitted;
  __shared__ long long s_left;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  auto key_of = [&](int c) -> uint32_t {
    uint32_t u = __float_as_uint(__ldg(score + c));
    if (u == 0x80000000u) u = 0u;
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
  };
  for (int i = tid; i < kAdmitBins; i += kAdmitThreads) hist[i] = 0u;
  pdl_wait();                                               // (its launch, and that of the kernel behind it, overlap)
  pdl_launch_dependents();
  uint32_t lo = 0xFFFFFFFFu, hi = 0u;
#pragma unroll 4
  for (int c = tid; c < n; c += kAdmitThreads) {
    const uint32_t k = key_of(c);
    lo = min(lo, k);
    hi = max(hi, k);
  }
  lo = __reduce_min_sync(0xFFFFFFFFu, lo);
  hi = __reduce_max_sync(0xFFFFFFFFu, hi);
  if (lane == 0) { s_lo[warp] = lo; s_hi[warp] = hi; }
  __syncthreads();
  if (warp == 0) {
    lo = __reduce_min_sync(0xFFFFFFFFu, s_lo[lane]);
    hi = __reduce_max_sync(0xFFFFFFFFu, s_hi[lane]);
    if (lane == 0) { s_base = lo; s_bits = 32 - __clz(hi - lo); s_left = capacity; s_all = 0; s_admitted = 0; }
  }
  __syncthreads();

  // s_left: capacity behind everything above the candidates, which are the keys with key - base < 2^bits
  for (bool first = true; first || s_bits > 0; first = false) {
    const uint32_t base = s_base;
    const int bits = s_bits, shift = max(bits - kAdmitDigit, 0);
    const long long left = s_left;
    const uint32_t width_m1 = bits >= 32 ? 0xFFFFFFFFu : ((1u << bits) - 1u);
#pragma unroll 4
    for (int c = tid; c < n; c += kAdmitThreads) {
      const uint32_t rel = key_of(c) - base;
      // bin b from the top at word (b % 4) * threads + b / 4: thread t owns bins 4t .. 4t + 3
      if (rel <= width_m1) {
        const uint32_t b = (uint32_t)(kAdmitBins - 1) - (rel >> shift);
        atomicAdd(&hist[(b & 3u) * kAdmitThreads + (b >> 2)], (uint32_t)size[c]);
      }
    }
    __syncthreads();
    uint32_t p[4], sum = 0u;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      p[j] = hist[j * kAdmitThreads + tid];
      hist[j * kAdmitThreads + tid] = 0u;
      sum += p[j];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    uint32_t before = 0u, total = 0u;
    {
      const uint32_t v = s_warp[lane];
      total = __reduce_add_sync(0xFFFFFFFFu, v);
      before = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? v : 0u);
    }
    long long above = (long long)before + incl - sum;
    if ((long long)total <= left) {                        // (only at the first level: everything fits)
      if (tid == 0) { s_all = 1; s_left = left - total; s_bits = 0; }
    } else if (above <= left && left < above + sum) {      // one thread holds the bin in which the capacity ends
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (above <= left && left < above + p[j]) {
          s_base = base + ((uint32_t)(kAdmitBins - 1 - (4 * tid + j)) << shift);
          s_bits = shift;
          s_left = left - above;
          break;
        }
        above += p[j];
      }
    }
    __syncthreads();
  }

  const uint32_t T = s_base;
  const bool all = s_all != 0;
  // ties at T in index order: warp w owns a contiguous span
  const int seg = ((n + 31) / 32 + 31) & ~31;
  const int w_lo = min(n, warp * seg), w_hi = min(n, w_lo + seg);
  uint32_t ties = 0u;
  if (!all) {
#pragma unroll 4
    for (int c = w_lo + lane; c < w_hi; c += 32)
      if (key_of(c) == T) ties += size[c];
  }
  ties = __reduce_add_sync(0xFFFFFFFFu, ties);
  if (lane == 0) s_warp[warp] = ties;
  __syncthreads();
  long long left = s_left;                                 // capacity left for this warp's ties
  left -= (long long)__reduce_add_sync(0xFFFFFFFFu, lane < warp ? s_warp[lane] : 0u);
  __shared__ uint32_t s_tie_pages;
  if (tid == 0) s_tie_pages = 0u;
  __syncthreads();
  int admitted = 0;
  uint32_t tie_pages = 0u;
  for (int c0 = w_lo; c0 < w_hi; c0 += 32) {
    const int c = c0 + lane;
    const uint32_t k = c < w_hi ? key_of(c) : 0u;
    bool in = c < w_hi && (all || k > T);
    const bool tie = !all && c < w_hi && k == T;
    if (__any_sync(0xFFFFFFFFu, tie)) {
      const uint32_t mine = tie ? size[c] : 0u;
      uint32_t incl = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += t;
      }
      if (tie && (long long)incl <= left) { in = true; tie_pages += mine; }
      left -= (long long)__shfl_sync(0xFFFFFFFFu, incl, 31);
    }
    if (c < w_hi) resident[c] = in ? 1 : 0;
    admitted += in;
  }
  if (info != nullptr) {
    admitted = __reduce_add_sync(0xFFFFFFFFu, admitted);
    tie_pages = __reduce_add_sync(0xFFFFFFFFu, tie_pages);
    if (lane == 0) { atomicAdd(&s_admitted, admitted); atomicAdd(&s_tie_pages, tie_pages); }
    __syncthreads();
    if (tid == 0) {
      info[0] = s_admitted;
      info[1] = (int32_t)min(capacity - s_left + (long long)s_tie_pages, 0x7FFFFFFFLL);
    }
  }
}

}  // namespace

long long cache_admit_workspace_bytes(int n) { return ((long long)n * 4 + 255) / 256 * 256; }

cudaError_t launch_cache_admit(const float* score, const uint16_t* size, int n, long long capacity, void* workspace,
                               uint8_t* resident, int32_t* info, cudaStream_t st) {
  (void)workspace;                                         // nothing is sorted any more; the interface keeps it
  return launch_pdl(admit_kernel, dim3(1), dim3(kAdmitThreads), 0, st, true, score, size, n, capacity, resident, info);
}

namespace {
long long padded(long long bytes) { return (bytes + 255) / 256 * 256; }
}  // namespace

long long build_clusters_workspace_bytes(int n) {
  return 2 * padded(4LL * n) + padded(4LL * bit_words(n)) + padded(4LL * kMaxPicks * kNoteWords) + padded(4LL * kMaxPicks) +
         padded(4LL * kCtlWords);
}

cudaError_t launch_build_clusters(const float* dist, int n, float tau, void* workspace, int32_t* rho, int32_t* ptr,
                                  int32_t* members, long long members_cap, int32_t* medoid, int32_t* n_clusters,
                                  int32_t* dev_status, cudaStream_t st) {
  char* ws = static_cast<char*>(workspace);
  auto take = [&](long long bytes) { char* p = ws; ws += padded(bytes); return p; };
  ClusterArgs a;
  a.dist = dist; a.n = n; a.tau = tau; a.rho = rho;
  a.queue = reinterpret_cast<int32_t*>(take(4LL * n));
  a.place = reinterpret_cast<int32_t*>(take(4LL * n));
  a.covered = reinterpret_cast<uint32_t*>(take(4LL * bit_words(n)));
  a.holds = reinterpret_cast<uint32_t*>(take(4LL * kMaxPicks * kNoteWords));
  a.size = reinterpret_cast<int32_t*>(take(4LL * kMaxPicks));
  a.ctl = reinterpret_cast<unsigned*>(take(4LL * kCtlWords));
  a.ptr = ptr; a.members = members; a.members_cap = members_cap; a.medoid = medoid; a.n_clusters = n_clusters;
  a.dev_status = dev_status;

  density_kernel<<<dim3((n + 7) / 8), dim3(256), 0, st>>>(a);   // (first: the rest of the host's work runs beside it)
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  int cap = 1024;                                          // power of two >= n: the candidates of one cluster
  while (cap < n) cap <<= 1;
  const int smem = cap * 6 + std::max(kCountedCand * 8, bit_words(n) * 4);
  int dev = 0, sms = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(rounds_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(std::max(1, std::min({sms, n, kMaxPicks})));   // one CTA per SM, each grows one cluster per round
  cfg.blockDim = dim3(kRoundThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;             // the rounds end in barriers over the grid
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, rounds_kernel, a, cap);
}

}  // namespace swarm
