// Stage 3: cluster resolution, global merge and load-balanced bucket scheduling (Eq. 8; Sec. 5.1), written as
// a device function that two kernels run: resolve_kernel (swarm_resolve_clusters) and, inside the fused step,
// block 0 of the attention kernel (beside the attention CTAs; as a kernel of its own on a second stream it
// lost about 2 us whenever the attention kernel started).
//
//   mark     (all CTAs; inside the fused step the selection kernel has done it and this phase is skipped)
//            every selected (request, page) -> global cluster id; flag[id] = 1.
//            Idempotent byte stores: concurrent writers store the same value, so the dedup needs no
//            atomics.  Four independent slots per thread keep the dependent loads overlapped.
//   tail     (the CTA that finishes marking last, found with one ticket counter)
//     compact  ordered compaction of the flags -> uniq[] ascending by id: rows of 1024 clusters (flags, replica
//              masks, sizes) travel through a cp.async ring in shared memory, one scan over the CTA places a
//              row's ids; the flags are cleared on the way so the next call starts from zeros.  The clusters
//              that need the serial pass are packed, with their output slots, into one dense list (shared
//              memory; longer ones in global memory).
//              With cache state attached (swarm_set_cache) the same pass drops the activated clusters
//              that are resident (Eq. 8) and updates the activation frequencies and Eq. 6 scores.
//     route    single-replica clusters go to their queue (integer histogram, order-free).  Clusters
//              with R >= 2 replicas are visited by (R ascending, id ascending), each going to its
//              least-loaded replica, ties to the lowest queue id: a chain, because every choice depends on
//              the loads left by the one before it.  It bounds the serial step.  Three forms of it, all
//              bit-identical: lanes_pass (two replicas, equal weights, up to 8 queues), levels_pass (two
//              replicas, any weights, up to 16 queues), and for everything else one warp with a link per
//              cluster -- lane j keeps (load[j] << 5 | j), one redux.min over the lanes named by the
//              replica mask picks the queue.  Under SWARM_ORDER_BY_ID that warp visits every cluster in
//              id order instead.
//     submit   (optional output) the batched submission order of Sec. 5.1, see the end of the body.
#pragma once
#include "swarm_internal.cuh"

namespace swarm {
namespace resolve_detail {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kSlotsPerThread = 4;
constexpr size_t kResolveSmemBytes = 192 * 1024;         // operands of the serial pass, its tables, keys of the submission order

// ---- the serial pass over equally heavy clusters with two replicas, 32 stretches at a time ------------------------------
// The greedy is a chain: every choice depends on the loads the one before it left, and a link costs 44 cycles through
// the lanes of a warp.  But with equal weights its loads forget where they came from: two runs over the same clusters
// from different (equally heavy) loads fall into step after some tens to hundreds of clusters, because every choice they
// take differently brings them closer.  So the list is cut into 32 stretches, one per lane, and each lane runs its own
// from a guess -- the loads levelled out as far as the starting loads allow.  Then every lane takes the loads its left
// neighbour ended with as its start, and the warp runs again until no start changes any more.  That state is the
// sequential greedy's: lane 0 starts from the true loads and every other lane from where its neighbour ended.  It takes
// at most 32 turns (lane i is right after i turns whatever the guess): 560 clusters on 8 queues 8 turns of 19 links,
// 1600 (half of them two-replica, 8 queues) 6 of 51.
// A lane holds the loads of up to 8 queues as bytes of two registers, counted in clusters above the least of them.  A
// byte that reaches 128 ends the attempt (the caller then takes levels_pass); levels_pass is also what more queues take.
// Operands in shared memory, cluster k of stretch l at l * pitch + k (an odd pitch: the lanes read different banks); a
// stretch is filled up to a multiple of 4 with clusters that change nothing (shift 255).
//   sel     byte-permute selectors of the lower queue's byte and (upper half) the higher queue's; the other bytes of the
//           result are copies of a sign bit that is zero
//   shift   8 * lower queue | 8 * higher queue << 16
//   choice  4 bits per byte: bit k % 4 of byte (k / 4) * 32 + l is 1 where the lower queue was taken
//   load    lane q: queue q's load in clusters
constexpr int kLanesQueues = 8;
__device__ __forceinline__ uint32_t shared_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t lds(uint32_t at) {    // (32-bit addresses: generic ones cost the chains below a third)
  uint32_t r;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(r) : "r"(at) : "memory");
  return r;
}
// N bytes (16: past L1) of which the first `have` are read, the others arrive as zeros
template <int N>
__device__ __forceinline__ void copy_async(uint32_t to, const void* from, int have) {
  if (N == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to), "l"(from), "r"(have) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(to), "l"(from), "n"(N), "r"(have) : "memory");
}
__device__ __forceinline__ void sts(uint32_t at, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(at), "r"(v) : "memory"); }
__device__ __forceinline__ void sts8(uint32_t at, uint32_t v) { asm volatile("st.shared.u8 [%0], %1;" ::"r"(at), "r"(v) : "memory"); }
__host__ __device__ constexpr int lanes_seg(int n) { return (n + 31) / 32; }            // clusters of a stretch
__host__ __device__ constexpr int lanes_pitch(int n) { return ((lanes_seg(n) + 3) & ~3) + 1; }
__host__ __device__ constexpr int lanes_words(int n) { return 64 * lanes_pitch(n) + 64 + (lanes_seg(n) + 3) / 4 * 8; }
__device__ __forceinline__ uint32_t byte_perm(uint32_t x, uint32_t y, uint32_t sel) {   // (the intrinsic drops the sign mode)
  uint32_t r;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(x), "r"(y), "r"(sel));
  return r;
}
__device__ __forceinline__ uint32_t shl_or_zero(uint32_t x, uint32_t n) {   // (0 for n >= 32)
  uint32_t r;
  asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(n));
  return r;
}
__device__ __forceinline__ bool lanes_pass(const uint32_t* sel, const uint32_t* shift, const uint32_t* choice, int n, int D, unsigned load) {
  const int lane = threadIdx.x & 31;
  const int seg = lanes_seg(n), first = min(n, lane * seg), last = min(n, first + seg);
  const uint32_t sel_at = shared_addr(sel + lane * lanes_pitch(n)), shift_at = shared_addr(shift + lane * lanes_pitch(n));
  const uint32_t choice_at = shared_addr(choice) + lane;
  const uint32_t unused0 = D >= 4 ? 0u : 0x7F7F7F7Fu << (8 * D), unused1 = D >= 8 ? 0u : D <= 4 ? 0x7F7F7F7Fu : 0x7F7F7F7Fu << (8 * (D - 4));
  const uint32_t used0 = unused0 ? ~(0xFFFFFFFFu << (8 * D)) : 0xFFFFFFFFu;
  const uint32_t used1 = D >= 8 ? 0xFFFFFFFFu : D <= 4 ? 0u : ~(0xFFFFFFFFu << (8 * (D - 4)));
  // the guess: level L with sum of max(load, L) = all loads so far
  unsigned total = __reduce_add_sync(0xFFFFFFFFu, lane < D ? load : 0u) + (unsigned)first;
  unsigned level = total / (unsigned)D, rest = total % (unsigned)D;
  const unsigned l_max = __reduce_max_sync(0xFFFFFFFFu, lane < D ? load : 0u), l_min = __reduce_min_sync(0xFFFFFFFFu, lane < D ? load : ~0u);
  if (l_max != l_min) {
    for (int turn = 0; turn < D; ++turn) {
      unsigned above = 0u, n_above = 0u;
      for (int q = 0; q < D; ++q) {
        const unsigned l = __shfl_sync(0xFFFFFFFFu, load, q);
        if (l > level) { above += l; ++n_above; }
      }
      const unsigned left = total - above, among = (unsigned)D - n_above;   // (never all of them: the level is at most the mean)
      const bool lower = left / among < level;
      level = left / among;
      rest = left % among;
      if (!__any_sync(0xFFFFFFFFu, lower)) break;
    }
  }
  // the start as bytes above `base`
  unsigned base = lane > 0 ? level : l_min;
  uint32_t s0 = 0u, s1 = 0u, over = 0u;
  for (int q = 0; q < D; ++q) {
    const unsigned l = __shfl_sync(0xFFFFFFFFu, load, q);
    unsigned v = l;
    if (lane > 0 && l <= level) {
      v = level + (rest > 0u ? 1u : 0u);
      if (rest > 0u) --rest;
    }
    v -= base;
    if (v > 127u) over = 0x80u;
    if (q < 4) s0 |= (v & 127u) << (8 * q);
    else s1 |= (v & 127u) << (8 * (q - 4));
  }
  s0 |= unused0;
  s1 |= unused1;
  for (int turn = 0; turn <= 32; ++turn) {
    uint32_t F0 = s0, F1 = s1, x[4], y[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) { x[u] = lds(sel_at + 4 * u); y[u] = lds(shift_at + 4 * u); }
    for (int k = 0; k < seg; k += 4) {
      uint32_t xn[4], yn[4], lower4 = 0u;                 // (the last fetch runs past the stretch: not used)
#pragma unroll
      for (int u = 0; u < 4; ++u) { xn[u] = lds(sel_at + 4 * (k + 4 + u)); yn[u] = lds(shift_at + 4 * (k + 4 + u)); }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t la = byte_perm(F0, F1, x[u]), lb = byte_perm(F0, F1, x[u] >> 16);
        const bool lower = la <= lb;                      // a tie goes to the lower queue
        const uint32_t at = lower ? (y[u] & 0xFFu) : (y[u] >> 16);
        F0 += shl_or_zero(1u, at);
        F1 += shl_or_zero(1u, at - 32u);
        over |= F0 | F1;
        if (lower) lower4 |= 1u << u;
      }
      sts8(choice_at + 8 * k, lower4);
#pragma unroll
      for (int u = 0; u < 4; ++u) { x[u] = xn[u]; y[u] = yn[u]; }
    }
    over &= 0x80808080u;
    if (__any_sync(0xFFFFFFFFu, over != 0u)) return false;
    uint32_t n0 = __shfl_up_sync(0xFFFFFFFFu, F0, 1), n1 = __shfl_up_sync(0xFFFFFFFFu, F1, 1);
    unsigned nb = __shfl_up_sync(0xFFFFFFFFu, base, 1);
    if (lane == 0) { n0 = s0; n1 = s1; nb = base; }
    uint32_t low = __vminu4(n0 | unused0, n1 | unused1);  // (unused bytes: 127, never the least)
    low = min(min(low & 0xFFu, (low >> 8) & 0xFFu), min((low >> 16) & 0xFFu, low >> 24));
    n0 = ((n0 - low * 0x01010101u) & used0) | unused0;
    n1 = ((n1 - low * 0x01010101u) & used1) | unused1;
    nb += low;
    const bool moved = lane > 0 && first < last && (n0 != s0 || n1 != s1 || nb != base);
    if (!__any_sync(0xFFFFFFFFu, moved)) return true;
    if (lane > 0) { s0 = n0; s1 = n1; base = nb; }
  }
  return false;                                           // (not reached: 32 turns settle every lane)
}
// x / d for d >= 2 and x * d < 2^32 (inverse = ceil(2^32 / d)): an integer division by a variable takes ~40 instructions
__device__ __forceinline__ uint32_t inverse_of(int d) { return 0xFFFFFFFFu / (uint32_t)d + 1u; }
__device__ __forceinline__ int divide(int x, uint32_t inverse) { return (int)__umulhi((uint32_t)x, inverse); }
// Whether lanes_pass gave cluster i to its lower queue (seg = lanes_seg(n) and its inverse).
__device__ __forceinline__ bool lanes_choice(const uint32_t* choice, int seg, uint32_t seg_inverse, int i) {
  const int l = divide(i, seg_inverse), k = i - l * seg;
  return (reinterpret_cast<const uint8_t*>(choice)[(k >> 2) * 32 + l] >> (k & 3)) & 1;
}
// The operands of lanes_pass, by all threads of the CTA.
__device__ __forceinline__ void lanes_operands(const uint32_t* mask, int n, uint32_t* sel, uint32_t* shift) {
  const int seg = lanes_seg(n), pitch = lanes_pitch(n);
  const uint32_t inverse = inverse_of(pitch);
  for (int at0 = threadIdx.x; at0 < 32 * pitch; at0 += 4 * kThreads) {
    unsigned m[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int at = at0 + u * kThreads, l = divide(at, inverse), k = at - l * pitch, i = l * seg + k;
      m[u] = k < seg && l < 32 && i < n ? mask[i] : 0u;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int at = at0 + u * kThreads;
      const unsigned lo = (unsigned)__ffs(m[u]) - 1u, hi = 31u - (unsigned)__clz(m[u]);
      if (at < 32 * pitch) {
        sel[at] = m[u] ? 0x88808880u | lo | hi << 16 : 0x88888888u;
        shift[at] = m[u] ? 8u * lo | hi << 19 : 0x00FF00FFu;
      }
    }
  }
}
constexpr int kPairsMin = 48;                            // fewer clusters than this: one after the other is as quick

// ---- the serial pass over two-replica clusters of any weights, level by level ---------------------------------------------
// Clusters without a common queue do not wait for one another.  The list is cut into stretches of 11 clusters, a lane of a
// building warp each, which gives every cluster a level: one more than the last level of its stretch that uses one of its
// two queues.  Another warp, a lane per queue, walks the levels: a lane fetches the key (load << 5 | queue) of the queue its
// cluster of this level has in common with it and takes the cluster if its own key is the smaller one.  Two levels make
// one link of the chain: a lane also works out for itself what its partner of the second level does in the first, so that
// all three keys of a link are fetched at once.  A link takes 72 cycles; a cluster takes 0.5 levels on 8 queues, 0.35 on
// 16, 0.8 on 4, so it costs 19, 12 or 30 cycles against 44 one after the other.
constexpr int kStretch = 11;                             // (odd: the building lanes read different banks)
constexpr int kChunk = 32 * kStretch;                    // clusters a building warp takes at a time
constexpr int kLevelQueues = 16;                         // (4 bits of two registers each while levels are assigned)
constexpr int kBuilders = 3;                             // warps, and table buffers
constexpr int kTableRows = kChunk + 6;                   // levels of a chunk at most; the walk reads up to two links past the end
constexpr int kTakenWords = (kChunk + 15) / 16 * 32;     // a bit per level and queue
constexpr int kPassWords = kBuilders * (kTableRows * kLevelQueues + kTakenWords);
__device__ __forceinline__ unsigned key_of_lane(unsigned key, unsigned from) {   // (the upper bits of `from` do not count)
  unsigned r;
  asm volatile("shfl.sync.idx.b32 %0, %1, %2, 31, 0xffffffff;" : "=r"(r) : "r"(key), "r"(from));
  return r;
}
__device__ __forceinline__ void warps_sync(int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void warps_arrive(int id) { asm volatile("bar.arrive %0, 64;" ::"r"(id) : "memory"); }

// Levels and table of the clusters [first, min(n, first + kChunk)) (one warp).  Returns the number of levels; the
// cluster's level goes into the bits of wgt (weight << 5) from 21 on.  Rolled loops that look at the lists twice: what the code
// costs is its fetch, once per step on an SM that has not run it since the step before.  (Unrolled over the 11 clusters, in registers: a
// separate call on 983 clusters, 116.5 us with the calls around it, now 114.3; the medoid step of 1950 clusters 54.1, now 53.3; six
// ragged requests of up to 80K tokens 36.2, now 35.5.  Code that has just run is the slower one for it: the separate call over and over
// 22.4, now 23.0.)
__device__ __forceinline__ int levels_build(const uint32_t* mask, uint32_t* wgt, int n, int first, uint32_t* table) {
  const int lane = threadIdx.x & 31;
  const int i0 = first + lane * kStretch, i1 = min(n, i0 + kStretch);
  uint32_t f0 = 0u, f1 = 0u;                              // 4 bits per queue: levels of this stretch that end with it
  int rows = 0;
#pragma unroll 1
  for (int i = i0; i < i1; ++i) {
    const uint32_t m = mask[i];
    const unsigned lo = (unsigned)__ffs(m) - 1u, hi = 31u - (unsigned)__clz(m), at_lo = 4u * (lo & 7u), at_hi = 4u * (hi & 7u);
    const unsigned a = ((lo & 8u ? f1 : f0) >> at_lo) & 15u, b = ((hi & 8u ? f1 : f0) >> at_hi) & 15u, l = max(a, b);
    const uint32_t da = (l + 1u - a) << at_lo, db = (l + 1u - b) << at_hi;
    f0 += (lo & 8u ? 0u : da) + (hi & 8u ? 0u : db);
    f1 += (lo & 8u ? da : 0u) + (hi & 8u ? db : 0u);
    wgt[i] = (wgt[i] & 0x1FFFE0u) | l << 21;
    rows = max(rows, (int)l + 1);
  }
  int incl = rows;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += t;
  }
  const int n_rows = __shfl_sync(0xFFFFFFFFu, incl, 31);
  for (int i = 4 * lane; i < (n_rows + 1) * kLevelQueues; i += 128)  // no cluster: weight 0 (and one level more: links are pairs)
    *reinterpret_cast<uint4*>(table + i) = make_uint4(0u, 0u, 0u, 0u);
  __syncwarp();
#pragma unroll 1
  for (int i = i0; i < i1; ++i) {
    const uint32_t m = mask[i], at = wgt[i], w = at & 0x1FFFE0u;
    const unsigned lo = (unsigned)__ffs(m) - 1u, hi = 31u - (unsigned)__clz(m), row = (at >> 21) + (unsigned)(incl - rows);
    table[row * kLevelQueues + lo] = hi | w;
    table[row * kLevelQueues + hi] = lo | w;
    wgt[i] = w | row << 21;
  }
  return n_rows;
}

// One link: rows with the entries e1 and e2 of this lane; er: the first-level entry of its partner of the second level.
__device__ __forceinline__ unsigned levels_link(unsigned key, unsigned e1, unsigned e2, unsigned er, uint32_t& bits, uint32_t bit) {
  const unsigned p = key_of_lane(key, e1), x = key_of_lane(key, e2), xp = key_of_lane(key, er);
  const bool win1 = key < p, winx = x < xp;
  unsigned k1 = key, x1 = x;
  if (win1) k1 += e1 & ~31u;
  if (winx) x1 += er & ~31u;
  const bool win2 = k1 < x1;
  if (win1) bits |= bit;
  if (win2) bits |= bit << 1;
  return win2 ? k1 + (e2 & ~31u) : k1;
}
// The walk over a chunk's levels (one warp).  taken: bit (row % 16) of word (row / 16) * 32 + queue.
__device__ __forceinline__ unsigned levels_walk(const uint32_t* table, uint32_t* taken, int D, int rows, unsigned key) {
  constexpr uint32_t kRow = 4 * kLevelQueues;
  const int lane = threadIdx.x & 31;
  uint32_t row = shared_addr(table), own = row + (lane < D ? 4 * lane : 0), out = shared_addr(taken) + 4 * lane;
  uint32_t e1 = lds(own), e2 = lds(own + kRow), er = lds(row + 4 * (e2 & 31u));
  uint32_t b1 = lds(own + 2 * kRow), b2 = lds(own + 3 * kRow);   // the next link
  auto step = [&](uint32_t at, uint32_t& bits, uint32_t bit) {   // at: bytes from the first to this link
    const uint32_t c1 = lds(own + at + 4 * kRow), c2 = lds(own + at + 5 * kRow);   // the link after the next
    const uint32_t br = lds(row + at + 2 * kRow + 4 * (b2 & 31u));
    key = levels_link(key, e1, e2, er, bits, bit);
    e1 = b1; e2 = b2; er = br;
    b1 = c1; b2 = c2;
  };
  int r = 0;
  for (; r + 16 <= rows; r += 16) {
    uint32_t bits = 0u;
#pragma unroll
    for (int u = 0; u < 8; ++u) step(2 * u * kRow, bits, 1u << (2 * u));
    sts(out, bits);
    out += 128;
    row += 16 * kRow;
    own += 16 * kRow;
  }
  if (r < rows) {
    uint32_t bits = 0u;
    for (int u = 0; r + u < rows; u += 2) step(u * kRow, bits, 1u << u);
    sts(out, bits);
  }
  return key;
}

// Warp 0 walks (and returns the final keys); warps 1 .. kBuilders build, and put the chosen queues into the low bits of wgt.
// Chunk c lies in buffer c % kBuilders; named barriers 1 + b (built) and 1 + kBuilders + b (walked).
__device__ __forceinline__ unsigned levels_pass(uint32_t* mask, uint32_t* wgt, int n, int D, unsigned load, uint32_t* space, int* s_rows) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int chunks = (n + kChunk - 1) / kChunk;
  uint32_t* takens = space + kBuilders * kTableRows * kLevelQueues;
  unsigned key = load << 5 | (unsigned)lane;
  if (warp == 0) {
    for (int c = 0, b = 0; c < chunks; ++c, b = b + 1 == kBuilders ? 0 : b + 1) {
      warps_sync(1 + b);
      key = levels_walk(space + b * kTableRows * kLevelQueues, takens + b * kTakenWords, D, s_rows[b], key);
      warps_arrive(1 + kBuilders + b);
    }
  } else {
    const int b = warp - 1;
    uint32_t* table = space + b * kTableRows * kLevelQueues;
    const uint32_t* taken = takens + b * kTakenWords;
    for (int c = b; c < chunks; c += kBuilders) {
      const int rows = levels_build(mask, wgt, n, c * kChunk, table);
      if (lane == 0) s_rows[b] = rows;
      __syncwarp();
      warps_arrive(1 + b);
      warps_sync(1 + kBuilders + b);
      for (int i = c * kChunk + lane; i < min(n, (c + 1) * kChunk); i += 32) {
        const unsigned m = mask[i], w = wgt[i], r = w >> 21;
        const unsigned lo = (unsigned)__ffs(m) - 1u, hi = 31u - (unsigned)__clz(m);
        wgt[i] = (w & 0x1FFFE0u) | ((taken[(r >> 4) * 32 + lo] >> (r & 15u)) & 1u ? lo : hi);
      }
    }
  }
  return key;
}

// Dynamic shared memory, in words: the tables of the two passes above, then what the serial pass works on, `cap` words
// each -- replica masks and weight << 5 (the chosen queue joins it in the low bits), both with kBlanks words of room behind
// them, output slots -- and, if a submission order is wanted, its keys and ranks.
constexpr int kBlanks = 16;                              // blank clusters that follow the list: the flat loop fetches that far ahead
__host__ __device__ constexpr int serial_cap(bool submit) {
  return (((int)(kResolveSmemBytes / 4) - kPassWords) / (submit ? 5 : 3) - 24) & ~7;
}
__host__ __device__ constexpr int serial_words(bool submit) {
  return kPassWords + 2 * (serial_cap(submit) + kBlanks) + (submit ? 3 : 1) * serial_cap(submit);
}
static_assert(serial_words(false) * 4 <= (int)kResolveSmemBytes && serial_words(true) * 4 <= (int)kResolveSmemBytes,
              "the lists and their blanks fit behind the tables");

// `cta` of `n_ctas` CTAs of kThreads threads run the body with kResolveSmemBytes of dynamic shared memory.
template <bool kCached>
__device__ __forceinline__ void resolve_body(const ResolveArgs& r, int cta, int n_ctas) {
  const Geometry& geo = r.geo;
  const swarm_cache& cache = r.cache;
  const int32_t* __restrict__ sel = r.sel;
  const int32_t* __restrict__ n_sel = r.n_sel;
  const int64_t* __restrict__ page_base = r.page_base;
  const int32_t* __restrict__ page2cluster = r.page2cluster;
  const int64_t* __restrict__ cluster_base = r.cluster_base;
  const uint32_t* __restrict__ replica_mask = r.replica_mask;
  const uint16_t* __restrict__ cluster_size = r.cluster_size;
  uint8_t* __restrict__ flags = r.flags;                 // (the overlapped tail picks one of two arrays below)
  unsigned* __restrict__ ticket = r.ticket;
  uint4* __restrict__ items = r.items;
  int32_t* uniq = r.uniq;
  uint8_t* queue_of = r.queue_of;
  int32_t* __restrict__ n_uniq = r.n_uniq;
  int32_t* __restrict__ queue_load = r.queue_load;
  uint32_t* __restrict__ status = r.status;
  (void)n_sel;
  extern __shared__ uint4 s_dyn[];
  const int cap = serial_cap(r.submit_order != nullptr);
  uint32_t* s_pass = reinterpret_cast<uint32_t*>(s_dyn);
  uint32_t* s_mask = s_pass + kPassWords;
  uint32_t* s_wgt = s_mask + cap + kBlanks;
  uint32_t* s_slot = s_wgt + cap + kBlanks;
  __shared__ int s_tot[2][kWarps];                       // clusters to fetch | those for the serial pass << 16, per warp, of two rows
  __shared__ int s_rows[kBuilders];
  __shared__ bool s_even;
  __shared__ int s_load[32];
  __shared__ unsigned s_classes, s_wmin, s_wmax;         // of the serial pass: replica classes, smallest and largest weight
  __shared__ unsigned s_item_m[32], s_item_w[32];
  __shared__ bool s_last;
  constexpr int kDryClusters = 128;
  __shared__ struct { int32_t uniq[kDryClusters], freq[kDryClusters]; float score[kDryClusters]; uint8_t queue_of[kDryClusters]; } s_dry;
  __shared__ int s_hits;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (sel != nullptr) {                                  // on its own any input may come from the previous kernel
    pdl_wait();
    pdl_launch_dependents();                             // the next kernel in the stream may be scheduled while this one runs
  }
  const long long c_all = cluster_base[geo.B];           // inside a step an input table: not written by the previous kernel
  const int C = (int)min((long long)geo.Cmax, c_all);
  unsigned err = 0u, step_no = 0u;
  // Every instruction below runs once per step, on an SM that has not fetched it since the step before, and while the
  // attention kernel streams a fetch from L2 takes 2-3 us.  A CTA that is resident before its selection has finished runs
  // the body once on the first clusters of the tables, as if they were all activated: nothing but scratch is written.
  // A rehearsal takes about 10 us.  It pays where
  // the CTA waits as long anyway and the resolution ends the step: one request at 128K tokens 28.7 -> 28.1 us, at 32K tokens 18.0 -> 17.8;
  // with cache state 16 ragged requests of up to 128K tokens and an admission 125.0 -> 124.6, 37 of 55K 177.8 -> 177.4, 3 of 114K 80.8 ->
  // 79.0, 12 of 33K 43.3 -> 42.4.  Steps of several waves without cache state: 36.6 -> 36.9 (the attention ends them);
  // the medoid step, which has 4 us to wait: 10 us longer.  Not in a kernel of its own, which does not know what it waits for: on an idle
  // stream the call takes 35 us, 41 with a rehearsal on made-up clusters; 64 requests x 32 heads x 128 pages (256 CTAs) 34, and 41;
  // 16 x 64 x 512 (512 CTAs) 45, and 64; only four separate calls in a row gained by it (114.2 us, and 113.7).
  for (bool dry = r.rehearse; ; dry = false) {
  int n_clusters = min(C, kDryClusters);
  int32_t* freq_out = cache.freq;
  float* score_out = cache.score;
  if (dry) {
    uniq = s_dry.uniq;
    // (With cache state in global memory: where the pointer may be into either, the pass over a list too long for shared memory, 16384
    // clusters of 64 requests, was compiled slower: the step 645 us instead of 585.  So it was without cache state, 757 instead of 663,
    // when code only a kernel of its own runs was left out of the attention kernel.)
    queue_of = kCached ? reinterpret_cast<uint8_t*>(items) : s_dry.queue_of;
    freq_out = s_dry.freq;
    score_out = s_dry.score;
  } else {
  uniq = r.uniq;
  queue_of = r.queue_of;
  if (sel == nullptr) {
    pdl_wait();                                          // the flags come from the previous kernel
    pdl_launch_dependents();
  }
  n_clusters = C;
  err = (c_all > geo.Cmax) ? SWARM_DEV_BAD_CLUSTER : 0u;
  // Overlapped tail: nothing after this kernel in the step waits for it, so it runs beside the next step's
  // scoring and selection.  That selection marks the other one of two flag arrays (the selection kernel counts
  // the steps it has marked; step n uses array (n - 1) & 1), and this kernel first lets the resolution of the
  // step before finish, which shares its outputs and scratch.
  if (r.tail_ctl != nullptr) {
    step_no = *reinterpret_cast<volatile unsigned*>(r.tail_ctl + kCtlMarked);
    flags += ((step_no - 1u) & 1u) * r.flags_alt;
    if (tid == 0 && !wait_at_least(r.tail_ctl + kCtlResolved, step_no - 1u)) err |= SWARM_DEV_TIMEOUT;
    __syncthreads();
  }

  SWARM_STAMP(status, 0);
  SWARM_KERNEL_BEGIN(status, 3);
  // ---- mark (skipped when the selection kernel already set the flags: sel == nullptr) -------------
  if (sel != nullptr) {
    const long long slots = (long long)geo.B * geo.Hq * geo.k;
    const long long base = (long long)cta * (kThreads * kSlotsPerThread) + tid;
    int p[kSlotsPerThread], bh[kSlotsPerThread];
    bool live[kSlotsPerThread];
#pragma unroll
    for (int u = 0; u < kSlotsPerThread; ++u) {
      const long long idx = base + (long long)u * kThreads;
      live[u] = idx < slots;
      bh[u] = live[u] ? (int)(idx / geo.k) : 0;
      p[u] = live[u] ? sel[idx] : -1;
    }
#pragma unroll
    for (int u = 0; u < kSlotsPerThread; ++u) {
      const long long idx = base + (long long)u * kThreads;
      live[u] = live[u] && (int)(idx - (long long)bh[u] * geo.k) < n_sel[bh[u]];
    }
    long long cid[kSlotsPerThread];
#pragma unroll
    for (int u = 0; u < kSlotsPerThread; ++u) {
      cid[u] = -1;
      if (!live[u]) continue;
      const int b = bh[u] / geo.Hq;
      const long long pb = page_base[b];
      if (p[u] < 0 || p[u] >= page_base[b + 1] - pb) { err |= SWARM_DEV_BAD_PAGE; continue; }
      const int c = page2cluster[pb + p[u]];
      const long long cb = cluster_base[b];
      if (c < 0 || c >= cluster_base[b + 1] - cb || cb + c >= C) { err |= SWARM_DEV_BAD_CLUSTER; continue; }
      cid[u] = cb + c;
    }
#pragma unroll
    for (int u = 0; u < kSlotsPerThread; ++u)
      if (cid[u] >= 0) flags[cid[u]] = 1;
  }
  if (err) atomicOr(status, err);
  err = 0u;

  // ---- which CTA is last? -------------------------------------------------------------------------
  if (n_ctas > 1) {
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = (atomicAdd(ticket, 1u) == (unsigned)n_ctas - 1u);
    __syncthreads();
    if (!s_last) return;
    __threadfence();
  } else {
    __syncthreads();   // one CTA: its own marks are visible to all of its threads after the barrier
  }
  SWARM_STAMP_ANY_CTA(status, 1);
  }

  // ---- compact (flags are read past L1: other CTAs wrote them) -------------------------------------
  // A row is 1024 clusters, four per thread: one word of flags with the replica masks and sizes of its clusters.  The rows
  // travel through a ring in shared memory, kDepth of them requested ahead: under the attention kernel's load a trip
  // to L2 takes 2-3 us.  Per row one scan over the CTA places
  // the ids, ascending; the flags are cleared on the way, each cluster's replica mask is validated, the single-replica
  // ones are routed, and the clusters that need the serial pass are packed, in id order, into one list.
  constexpr int kRow = 4 * kThreads;
  constexpr int kDepth = kCached ? 5 : 8;
  constexpr int kRowBytes = kThreads * (kCached ? 48 : 28);
  static_assert(kDepth * kRowBytes + kRow * 6 <= kPassWords * 4, "the ring lies where the serial pass's tables go");
  // a row's places: the cluster (within the row) of every id, and of every serial item with its place among the ids
  uint16_t* s_src = reinterpret_cast<uint16_t*>(s_pass + kDepth * kRowBytes / 4);
  uint32_t* s_ser = reinterpret_cast<uint32_t*>(s_src + kRow);
  if (tid < 32) s_load[tid] = 0;
  if (tid == 0) { s_classes = 0u; s_wmin = 0xFFFFFFFFu; s_wmax = 0u; s_hits = 0; }
  const unsigned valid_bits = geo.D == 32 ? 0xFFFFFFFFu : ((1u << geo.D) - 1u);
  const bool by_id = (geo.flags & SWARM_ORDER_BY_ID) != 0;
  const bool unit = (geo.flags & SWARM_UNIT_LOAD) != 0;
  // vector loads of the cache state need its arrays aligned like the library's own tables
  const bool cache_vec = kCached && (reinterpret_cast<uintptr_t>(cache.resident) & 3u) == 0 &&
                         (reinterpret_cast<uintptr_t>(cache.freq) & 15u) == 0 && (reinterpret_cast<uintptr_t>(cache.score) & 15u) == 0;
  const bool need_score = kCached && cache.score != nullptr;
  const bool need_sz = !unit || need_score;   // unit loads need no size table, Eq. 6 does
  const int rows = (n_clusters + kRow - 1) / kRow;
  const uint32_t ring = shared_addr(s_pass);
  auto request = [&](int row) {                            // (entries beyond the tables arrive as zeros)
    const int c = row * kRow + 4 * tid, have = min(4, n_clusters - c);
    if (row < rows && have > 0) {
      const uint32_t at = ring + (row % kDepth) * kRowBytes;
      copy_async<16>(at + 16 * tid, replica_mask + c, 4 * have);
      if (need_sz) copy_async<8>(at + kThreads * 16 + 8 * tid, cluster_size + c, 2 * have);
      if ((tid & 3) == 0) copy_async<16>(at + kThreads * 24 + 4 * tid, flags + c, 16);   // (the flag array is padded to 16 bytes)
      if (kCached && cache_vec) {
        copy_async<16>(at + kThreads * 28 + 16 * tid, cache.freq + c, 4 * have);
        copy_async<4>(at + kThreads * 44 + 4 * tid, cache.resident + c, have);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  for (int row = 0; row < kDepth; ++row) request(row);
  int n = 0, n_serial = 0;                                 // clusters to fetch so far, and those for the serial pass
  const bool spill = n_clusters > cap;                     // the list may outgrow shared memory: it is written to global memory as well
  // submission order (optional): (replica class, queue) keys, kept in shared memory so that the ordering pass at the
  // end does not have to read the results back from global memory
  uint32_t* order_key = s_slot + cap;
  const bool order_keys = r.submit_order != nullptr;
  unsigned classes = 0u, wmin = 0xFFFFFFFFu, wmax = 0u;
  int hits = 0;                                            // activated clusters that are resident
  for (int row = 0; row < rows; ++row) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kDepth - 1) : "memory");
    __syncthreads();
    const int c0 = row * kRow + 4 * tid;
    uint32_t f = 0u, mk[4] = {0u, 0u, 0u, 0u}, sz[2] = {0u, 0u}, res = 0u;
    int fr[4] = {0, 0, 0, 0};
    if (c0 < n_clusters) {
      const uint32_t* at = s_pass + (row % kDepth) * (kRowBytes / 4);
      const uint4 m4 = *reinterpret_cast<const uint4*>(at + 4 * tid);
      mk[0] = m4.x; mk[1] = m4.y; mk[2] = m4.z; mk[3] = m4.w;
      if (need_sz) {
        const uint2 s2 = *reinterpret_cast<const uint2*>(at + kThreads * 4 + 2 * tid);
        sz[0] = s2.x; sz[1] = s2.y;
      }
      f = at[kThreads * 6 + tid];
      if (dry) f = c0 + 4 <= n_clusters ? 0x01010101u : 0u;
      else if (f) __stcg(reinterpret_cast<uint32_t*>(flags + c0), 0u);   // leave zeros for the next call
      if (kCached) {
        if (cache_vec) {
          const int4 f4 = *reinterpret_cast<const int4*>(at + kThreads * 7 + 4 * tid);
          fr[0] = f4.x; fr[1] = f4.y; fr[2] = f4.z; fr[3] = f4.w;
          res = at[kThreads * 11 + tid];
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (c0 + j < n_clusters) {
              res |= (cache.resident[c0 + j] != 0 ? 1u : 0u) << (8 * j);
              fr[j] = cache.freq[c0 + j];
            }
          }
        }
      }
    }
    if (kCached && c0 < n_clusters) {
      // cache bookkeeping of Sec. 5.2 for every cluster, activated or not; four clusters' words in one store where the
      // arrays allow it and all four counters move (eight stores of a word per thread and row: 16 ragged requests of up to 128K tokens
      // and an admission 128.9 us, now 125.0; 37 of 55K 187.9, now 177.8; both without the rehearsal)
      float score[4];
      unsigned moved = 0u;                                 // only these counters are written: the others may be somebody else's to move
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const bool on = ((f >> (8 * j)) & 0xFFu) != 0u, is_res = ((res >> (8 * j)) & 0xFFu) != 0u;
        fr[j] += on ? 1 : is_res ? -1 : 0;
        moved |= (on || is_res ? 1u : 0u) << j;
        hits += on && is_res ? 1 : 0;
        const float size_f = (float)((sz[j >> 1] >> (16 * (j & 1))) & 0xFFFFu);
        score[j] = need_score ? (float)fr[j] * (cache.t_base + size_f * cache.t_transfer) / size_f : 0.f;
      }
      const bool vec = cache_vec && !dry && c0 + 4 <= n_clusters;
      if (vec && moved == 15u) *reinterpret_cast<int4*>(freq_out + c0) = make_int4(fr[0], fr[1], fr[2], fr[3]);
      if (vec && need_score) *reinterpret_cast<float4*>(score_out + c0) = make_float4(score[0], score[1], score[2], score[3]);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (((moved >> j) & 1u) && !(vec && moved == 15u) && c0 + j < n_clusters) freq_out[c0 + j] = fr[j];
        if (need_score && !vec && c0 + j < n_clusters) score_out[c0 + j] = score[j];
      }
    }
    // bit j: cluster j of the word is fetched (activated, and with cache state not resident: Eq. 8) / needs the serial pass
    unsigned fetch_bits = 0u, serial_bits = 0u;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const unsigned m = mk[j];
      const bool fetch = ((f >> (8 * j)) & 0xFFu) != 0u && !(kCached && ((res >> (8 * j)) & 0xFFu) != 0u);
      const bool valid = m != 0u && !(m & ~valid_bits);
      fetch_bits |= (fetch ? 1u : 0u) << j;
      serial_bits |= (fetch && valid && (by_id || (m & (m - 1u)) != 0u) ? 1u : 0u) << j;
    }
    // one scan for both places: ids in the low half, serial items in the high half
    const int mine = __popc(fetch_bits) | (__popc(serial_bits) << 16);
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) s_tot[row & 1][warp] = incl;
    __syncthreads();
    int before = incl - mine, total = 0;
#pragma unroll
    for (int w2 = 0; w2 < kWarps; ++w2) {
      const int t = s_tot[row & 1][w2];
      if (w2 < warp) before += t;
      total += t;
    }
    // first only who goes where, then every thread takes ids (and serial items) of the dense lists: per set bit in the
    // thread that holds it the work below took 0.9 us a row
    {
      int at = before & 0xFFFF, ser = before >> 16;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if ((fetch_bits >> j) & 1u) s_src[at] = (uint16_t)(4 * tid + j);
        if ((serial_bits >> j) & 1u) s_ser[ser] = (uint32_t)(4 * tid + j) | (uint32_t)at << 16;
        at += (fetch_bits >> j) & 1;
        ser += (serial_bits >> j) & 1;
      }
    }
    __syncthreads();
    const uint32_t* row_mask = s_pass + (row % kDepth) * (kRowBytes / 4);
    const uint16_t* row_size = reinterpret_cast<const uint16_t*>(row_mask + kThreads * 4);
    for (int k = tid; k < (total & 0xFFFF); k += kThreads) {
      const int src = s_src[k], i = n + k;
      const unsigned m = row_mask[src];
      uniq[i] = row * kRow + src;
      const bool valid = m != 0u && !(m & ~valid_bits);
      if (!valid || (!by_id && (m & (m - 1u)) == 0u)) {     // nothing to decide: a single replica, or none that exists
        const unsigned qd = valid ? (unsigned)__ffs(m) - 1u : 0xFFu;
        queue_of[i] = (uint8_t)qd;
        if (valid) atomicAdd(&s_load[qd], unit ? 1 : (int)row_size[src]);
        else err |= SWARM_DEV_BAD_REPLICA;
        if (order_keys && i < cap) order_key[i] = valid ? 32u + qd : 0xFFFFFFFFu;
      }
    }
    for (int k = tid; k < (total >> 16); k += kThreads) {
      const uint32_t src = s_ser[k];
      const int spos = n_serial + k;
      const unsigned m = row_mask[src & 0xFFFFu], wgt = unit ? 1u : row_size[src & 0xFFFFu], slot = (unsigned)n + (src >> 16);
      classes |= 1u << (__popc(m) - 1);
      wmin = min(wmin, wgt);
      wmax = max(wmax, wgt);
      if (spos < cap) {                                    // the serial pass then never waits on global memory
        s_mask[spos] = m;
        s_wgt[spos] = wgt << 5;
        s_slot[spos] = slot;
      }
      if (spill) items[spos] = make_uint4(m, wgt << 5, slot, 0u);
    }
    n += total & 0xFFFF;
    n_serial += total >> 16;
    __syncthreads();                                       // everyone is done with the row
    request(row + kDepth);
  }
  const bool staged = n_serial <= cap;
  const bool order_keys_early = order_keys && staged && n <= cap;
  SWARM_STAMP_ANY_CTA(status, 2);
  if (classes) {
    atomicOr(&s_classes, classes);
    atomicMin(&s_wmin, wmin);
    atomicMax(&s_wmax, wmax);
  }
  if (kCached && hits) atomicAdd(&s_hits, hits);
  if (err && !dry) atomicOr(status, err);
  err = 0u;
  if (staged && tid < kBlanks) s_mask[n_serial + tid] = s_wgt[n_serial + tid] = 0u;
  __syncthreads();
  SWARM_STAMP_ANY_CTA(status, 3);

  // ---- everything left for the serial pass has two replicas: see lanes_pass and levels_pass ------------
  const bool pairs = staged && s_classes == 2u && n_serial >= kPairsMin && geo.D <= kLevelQueues;   // (uniform over the CTA)
  const unsigned todo = by_id ? 1u : (s_classes & ~1u);   // replica classes the serial pass visits
  const bool flat = staged && !pairs && __popc(todo) <= 1;
  if (pairs) {
    bool even = geo.D <= kLanesQueues && lanes_words(n_serial) <= kPassWords && s_wmin == s_wmax && s_wmin > 0u;
    if (even)
      for (int q = 0; q < geo.D; ++q) even = even && (unsigned)s_load[q] % s_wmin == 0u;
    if (even) {
      const unsigned unit_w = s_wmin;
      uint32_t *sel = s_pass, *shift = sel + 32 * lanes_pitch(n_serial) + 32, *choice = shift + 32 * lanes_pitch(n_serial) + 32;
      lanes_operands(s_mask, n_serial, sel, shift);
      __syncthreads();
      SWARM_STAMP_ANY_CTA(status, 8);
      if (warp == 0) {
        const bool ok = lanes_pass(sel, shift, choice, n_serial, geo.D, (unsigned)s_load[lane] / unit_w);
        if (lane == 0) s_even = ok;
      }
      __syncthreads();
      SWARM_STAMP_ANY_CTA(status, 9);
      even = s_even;
      if (even) {
        const int seg = lanes_seg(n_serial);
        const uint32_t inverse = inverse_of(seg);
        for (int i = tid; i < n_serial; i += kThreads) {
          const unsigned m = s_mask[i];
          const unsigned q = lanes_choice(choice, seg, inverse, i) ? (unsigned)__ffs(m) - 1u : 31u - (unsigned)__clz(m);
          s_wgt[i] |= q;
          atomicAdd(&s_load[q], (int)unit_w);
        }
      }
    }
    if (!even && warp <= kBuilders) {
      const unsigned key = levels_pass(s_mask, s_wgt, n_serial, geo.D, (unsigned)s_load[lane], s_pass, s_rows);
      if (warp == 0 && lane < geo.D) s_load[lane] = (int)(key >> 5);
    }
  } else if (warp == 0) {
    // ---- the ordered greedy, one warp ----------------------------------------------------------------
    unsigned L = ((unsigned)s_load[lane] << 5) | (unsigned)lane;     // (load, queue id) in one comparable word
    // Common case: everything the serial pass has to visit is of one replica class (or the order is by id) and
    // sits in shared memory.  The list then is the visit order, and the pass is a flat loop over it: the operands
    // of the next eight clusters are fetched while eight are decided, lane u keeps the queue of the u-th.
    if (flat && n_serial > 0) {
      constexpr int kAhead = 8;
      static_assert(2 * kAhead <= kBlanks, "a turn that starts in the list fetches up to two turns' clusters");
      const uint32_t m_at = shared_addr(s_mask), w_at = shared_addr(s_wgt);
      unsigned m[kAhead], w[kAhead];
#pragma unroll
      for (int u = 0; u < kAhead; ++u) { m[u] = lds(m_at + 4 * u); w[u] = lds(w_at + 4 * u); }
      for (int i = 0; i < n_serial; i += kAhead) {         // (blank clusters follow the list: no lane takes part)
        unsigned m2[kAhead], w2[kAhead], best[kAhead];
#pragma unroll
        for (int u = 0; u < kAhead; ++u) { m2[u] = lds(m_at + 4 * (i + kAhead + u)); w2[u] = lds(w_at + 4 * (i + kAhead + u)); }
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
          const unsigned key = ((m[u] >> lane) & 1u) ? L : 0xFFFFFFFFu;
          best[u] = __reduce_min_sync(0xFFFFFFFFu, key);   // shuffle-, ballot- and register-based
          if (key == best[u]) L += w[u];                   // variants measured slower on sm_100
        }
        unsigned mine = best[0];
#pragma unroll
        for (int u = 1; u < kAhead; ++u) mine = lane == u ? best[u] : mine;
        if (lane < kAhead && i + lane < n_serial) sts(m_at + 4 * (i + lane), mine & 31u);   // (in the mask's place)
#pragma unroll
        for (int u = 0; u < kAhead; ++u) { m[u] = m2[u]; w[u] = w2[u]; }
      }
    }
    // Several replica classes (one after the other), or a list in global memory: 32 clusters at a time are staged in
    // shared memory so that the serial loop is a plain counted loop whose operands are fetched one step ahead of
    // the dependent chain select -> redux.min -> compare -> add.
    for (int R = by_id ? 0 : 2; R <= (by_id ? 0 : geo.D) && !flat; ++R) {
      if (!by_id && !((todo >> (R - 1)) & 1u)) continue;
      // (mask, weight, output slot) of 32 clusters per step, fetched two steps ahead of their use
      auto item_at = [&](int k) -> uint4 {
        if (k >= n_serial) return make_uint4(0u, 0u, 0u, 0u);
        return staged ? make_uint4(s_mask[k], s_wgt[k] & ~31u, 0u, 0u) : items[k];
      };
      uint4 pre0 = item_at(lane);
      uint4 pre1 = item_at(32 + lane);
      for (int k0 = 0; k0 < n_serial; k0 += 32) {
        const unsigned m = pre0.x, wgt = pre0.y, slot = pre0.z;
        pre0 = pre1;
        pre1 = item_at(k0 + 64 + lane);
        const bool mine = m != 0u && (by_id || __popc(m) == R);
        const unsigned pending = __ballot_sync(0xFFFFFFFFu, mine);
        const int cnt_p = __popc(pending);
        if (cnt_p == 0) continue;
        const int rank = __popc(pending & ((1u << lane) - 1u));
        if (mine) { s_item_m[rank] = m; s_item_w[rank] = wgt; }
        __syncwarp();
        unsigned my_q = 0u;
        unsigned mm = s_item_m[0], ww = s_item_w[0];
        for (int rr = 0; rr < cnt_p; ++rr) {
          const unsigned mm_next = s_item_m[min(rr + 1, 31)], ww_next = s_item_w[min(rr + 1, 31)];
          const unsigned key = ((mm >> lane) & 1u) ? L : 0xFFFFFFFFu;
          const unsigned best = __reduce_min_sync(0xFFFFFFFFu, key);
          if (L == best) L += ww;
          if (rank == rr) my_q = best & 31u;
          mm = mm_next;
          ww = ww_next;
        }
        // From shared memory the choice stays with the item and is written out after the pass: a global
        // store issued while the attention kernel starts or retires was measured to hold this warp for 2 us.
        if (mine) {
          if (staged) s_wgt[k0 + lane] |= my_q;
          else queue_of[slot] = (uint8_t)my_q;
        }
        __syncwarp();
      }
    }
    if (lane < geo.D) s_load[lane] = (int)(L >> 5);
    SWARM_KERNEL_END(status, 3);
  }
  __syncthreads();
  SWARM_STAMP_ANY_CTA(status, 4);
  if (staged) {
    for (int k = tid; k < n_serial; k += kThreads) {
      const unsigned q = (flat ? s_mask[k] : s_wgt[k]) & 31u, slot = s_slot[k];
      queue_of[slot] = (uint8_t)q;
      // (pairs and flat lists are of one replica class: bit R - 1 of todo)
      if (order_keys_early) order_key[slot] = (by_id ? 0u : pairs || flat ? (unsigned)__ffs(todo) * 32u : (unsigned)__popc(s_mask[k]) * 32u) + q;
    }
  }
  if (dry) {                                               // (the barrier: nobody still reads what the next turn rewrites)
    __syncthreads();
    continue;
  }
  if (tid < geo.D) {
    queue_load[tid] = s_load[tid];
    if (r.host.queue_load_h != nullptr) r.host.queue_load_h[tid] = s_load[tid];
  }
  if (tid == 0) {
    if (r.host.n_uniq_h != nullptr) *r.host.n_uniq_h = n;
    *n_uniq = n;
    if (kCached && cache.n_hit != nullptr) *cache.n_hit = s_hits;
    if (n_ctas > 1) *ticket = 0u;                          // ready for the next call
  }
  SWARM_STAMP_ANY_CTA(status, 5);

  // ---- batched submission order (Sec. 5.1, last paragraph; only when the caller attached the output) ------
  // Bucket q holds its clusters in assignment order: (replica count ascending, position in uniq ascending), or
  // position alone under SWARM_ORDER_BY_ID.  Batch r takes the r-th cluster of every bucket that has one, in
  // queue order.  Three steps: every thread forms the (class, queue) key of its clusters; the warps walk the
  // keys in position order and rank each cluster inside its (class, queue) group; every thread then turns
  // (class, queue, rank) into the cluster's place in the submission order with the bucket sizes alone.
  if (r.submit_order != nullptr) {
    __shared__ int s_group[33 * 32];                       // clusters per (class, queue); then the start of each group in its bucket
    __shared__ int s_bucket[32];                           // clusters per queue
    uint32_t* key_of = order_keys_early ? order_key : reinterpret_cast<uint32_t*>(items);
    uint32_t* rank_of = key_of + (order_keys_early ? cap : n);
    for (int i = tid; i < 33 * 32; i += kThreads) s_group[i] = 0;
    __syncthreads();                                       // also: every queue_of entry is written
    if (!order_keys_early) {
      // from global memory: four clusters per thread and turn, so that the two dependent reads of each
      // (its id, then that id's replica mask) overlap with the others'
      for (int i0 = tid; i0 < n; i0 += 4 * kThreads) {
        unsigned q[4], m[4];
        int id[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = i0 + u * kThreads;
          q[u] = i < n ? __ldcg(queue_of + i) : 0xFFu;
          id[u] = (i < n && !by_id) ? __ldcg(uniq + i) : -1;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) m[u] = id[u] >= 0 ? replica_mask[id[u]] : 0u;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = i0 + u * kThreads;
          // clusters with a bad replica mask are not submitted
          if (i < n) key_of[i] = q[u] >= 32u ? 0xFFFFFFFFu : ((unsigned)__popc(m[u]) * 32u + q[u]);
        }
      }
    }
    __syncthreads();
    // Every warp ranks a stretch of the clusters with counters of its own, then the counters of the warps in front are
    // added: a turn of the walk is 32 clusters in about 250 cycles, most of them the match.  (By one warp 3300
    // clusters took 13 us, behind everything else the step does.)  The keys come from shared memory; when they live in
    // global memory (more clusters than the lists hold) they are brought in a stage at a time.
    constexpr int kGroups = 33 * 32, kCountWords = kWarps * kGroups;
    static_assert(kCountWords <= kPassWords, "the counters lie where the serial pass's tables were");
    uint32_t *s_count = s_pass, *s_keys = s_pass + kCountWords;
    const int walk_cap = order_keys_early ? max(n, 1) : (int)(kResolveSmemBytes / 4) - kCountWords;
    for (int c0 = 0; c0 < n; c0 += walk_cap) {
      const int m_keys = min(walk_cap, n - c0);
      const uint32_t* keys = order_keys_early ? key_of : s_keys;
      if (!order_keys_early)
        for (int i = tid; i < m_keys; i += kThreads) s_keys[i] = key_of[c0 + i];
      for (int i = tid; i < kCountWords; i += kThreads) s_count[i] = 0u;
      __syncthreads();
      const int per = (m_keys + kThreads - 1) / kThreads * 32;   // clusters of a warp
      const int lo = warp * per, hi = min(m_keys, lo + per);
      uint32_t* mine = s_count + warp * kGroups;
      const unsigned lt = (1u << lane) - 1u;
      for (int i0 = lo; i0 < hi; i0 += 32) {
        const int i = i0 + lane;
        const uint32_t key = i < hi ? keys[i] : 0xFFFFFFFFu;
        const unsigned same = __match_any_sync(0xFFFFFFFFu, key);
        if (key != 0xFFFFFFFFu) rank_of[c0 + i] = mine[key] + __popc(same & lt);
        __syncwarp();
        if (key != 0xFFFFFFFFu && (same & lt) == 0u) mine[key] += __popc(same);   // the group's first lane
        __syncwarp();
      }
      __syncthreads();
      for (int g = tid; g < kGroups; g += kThreads) {
        int run = s_group[g];
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
          const int t = (int)s_count[w * kGroups + g];
          s_count[w * kGroups + g] = (uint32_t)run;
          run += t;
        }
        s_group[g] = run;
      }
      __syncthreads();
      for (int i = lane; i < hi - lo; i += 32) {
        const uint32_t key = keys[lo + i];
        if (key != 0xFFFFFFFFu) rank_of[c0 + lo + i] += mine[key];
      }
      __syncthreads();
    }
    if (tid < 32) {                                        // bucket sizes; group counts -> group starts
      int run = 0;
      for (int c = 0; c <= 32; ++c) {
        const int t = s_group[c * 32 + tid];
        s_group[c * 32 + tid] = run;
        run += t;
      }
      s_bucket[tid] = run;
    }
    __syncthreads();
    int submitted = 0, rounds = 0;
    for (int q = 0; q < geo.D; ++q) {
      submitted += s_bucket[q];
      rounds = max(rounds, s_bucket[q]);
    }
    for (int i0 = tid; i0 < n; i0 += 4 * kThreads) {       // four per turn: the reads of key and rank overlap
      uint32_t key4[4], rank4[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * kThreads;
        key4[u] = i < n ? key_of[i] : 0xFFFFFFFFu;
        rank4[u] = i < n ? rank_of[i] : 0u;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t key = key4[u];
        if (key == 0xFFFFFFFFu) continue;
        const int q = (int)(key & 31u);
        const int depth = s_group[key] + (int)rank4[u];    // position inside bucket q
        int pos = 0;
        for (int q2 = 0; q2 < geo.D; ++q2) pos += min(s_bucket[q2], depth) + ((q2 < q && s_bucket[q2] > depth) ? 1 : 0);
        r.submit_order[pos] = i0 + u * kThreads;
      }
    }
    if (tid == 0 && r.submit_info != nullptr) {
      r.submit_info[0] = rounds;
      r.submit_info[1] = submitted;
    }
  }
  if (r.host.done_h != nullptr) {                          // host step: the resolution's results are in host memory
    __syncthreads();
    if (tid == 0) host_arrive(r.host);
  }
  if (r.tail_ctl != nullptr) {                             // overlapped tail: this step's resolution has finished
    __syncthreads();
    if (tid == 0) st_release(r.tail_ctl + kCtlResolved, step_no);
  }
  break;
  }
}

}  // namespace resolve_detail
}  // namespace swarm
