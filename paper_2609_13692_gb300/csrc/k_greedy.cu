// Agglomerative common-intersection hierarchy (Sec. 6.2; H_g of Thm 6) and
// the spanning-tree lower bound (Sec. 6.3), for request counts far beyond the
// exact recurrence (m up to 16384).
//
// Greedy: every request starts as a cluster with signature R_i; the two active
// clusters with the heaviest common signature w(I(A) cap I(B)) merge, the
// merged signature being that intersection.  A cluster lives in the slot of
// its smallest request; ties go to the smallest slot pair (a, b), a < b, and
// the merged cluster keeps slot a.  The layout walks the hierarchy as in the
// Thm 1 proof.  Lower bound: sum_i w(R_i) - MaxSpanningTree(w(R_i cap R_j)).
//
// Merging in rounds.  Order the slot pairs by (weight, then the smaller pair):
// keys are distinct, and a merge never raises a key (the merged signature is
// part of both, and keeps the smaller slot).  So when a and b are each other's
// best pair, theirs stays the best of both until they merge, and the greedy
// sequence merges exactly that pair at exactly that key; all such pairs can
// merge in the same round.  A merge's key is above every key it leaves behind,
// so the greedy sequence is the merges of all rounds in decreasing key order.
// Once no pair shares weight, the rest is forced: the smallest slot takes in
// the others in increasing order, with empty signatures.  3,000 requests of 8
// passages from pools of 60 need 19 rounds.  The merges one after the other in
// one block took 25.7 of the 27.6 ms of a call (8.6 us each: some twenty block
// barriers); the rounds take 0.9 ms, bound by their launches and the latency of
// the row scans.
//
// Where one passage is in every request, or weights are equal, pairs tie and the
// slot order lets one or two merge per round: what is left then goes to one
// block (k_merge_rest).  3,000 requests with nothing in common but one passage:
// 96 ms in rounds alone, 14.4 so (22.9 in one block from the start); 12,000 of
// them 1,755 and 165 ms (319).
//
// Kernels: k_pair_weights fills W[i][j] = w(R_i cap R_j); Borůvka rounds find
// the maximum spanning tree of W; k_row_best, k_match and k_reweigh are one
// round of merges, k_merge_rest merges one by one; k_rank orders them; k_tail
// appends the forced ones; k_count and k_leaf_order give the left-to-right leaf
// order; k_greedy_emit climbs each (request, chunk) occurrence to the highest
// node whose signature still holds the chunk, and k_greedy_rank orders each
// request's chunks by (that node, chunk id).
#include "../../include/mpt.h"
#include "mpt_internal.cuh"

#include <algorithm>
#include <vector>

namespace mpt {
namespace {

constexpr int kSigMax = 128;       // longest request accepted
constexpr int kMaxGreedyM = 16384;  // slot ids fit in 14 bits
constexpr int kGreedyThreads = 1024;
constexpr int kAhead = 8;  // loads of a row of W that a thread keeps in flight (rows are mostly zeros)

// key of pair {d, e} with common weight v: larger is better (weight, then the
// smaller slot pair)
__device__ __forceinline__ unsigned long long pair_key(uint32_t d, uint32_t e, uint32_t v) {
  const uint32_t a = min(d, e), b = max(d, e);
  return ((unsigned long long)v << 28) | (unsigned long long)((1u << 28) - 1u - ((a << 14) | b));
}
__device__ __forceinline__ void key_pair(unsigned long long k, uint32_t* a, uint32_t* b) {
  const uint32_t p = (1u << 28) - 1u - (uint32_t)(k & ((1u << 28) - 1u));
  *a = p >> 14;
  *b = p & ((1u << 14) - 1u);
}

// Position of x in the sorted signature s[0 .. n), or -1.
__device__ __forceinline__ int find_in(const int32_t* s, int n, int32_t x) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (s[mid] < x) lo = mid + 1; else hi = mid;
  }
  return lo < n && s[lo] == x ? lo : -1;
}

// W of 32 rows by 256 columns per block: the rows' chunks set their row's bit
// in a table by the chunk's low bits; a column's chunks look their rows up
// there (checked by binary search, as chunks share table entries) and add
// their weight to the block's tile.  Both orders of a pair are computed, so
// that W is only written along rows: 178 -> 37 us at m = 3,000 against one
// thread merging the two signatures of a pair and writing it twice, once down a
// column.
constexpr int kPwRows = 32, kPwCols = 256, kPwTable = 4096;
constexpr int kPwSmem = (kPwTable + kPwRows * kSigMax + kPwRows * kPwCols) * 4;

__global__ void __launch_bounds__(kPwCols)
k_pair_weights(int m, const int64_t* __restrict__ off, const int32_t* __restrict__ sig, const int64_t* __restrict__ w,
               uint32_t* __restrict__ W) {
  extern __shared__ __align__(16) uint32_t pw[];
  uint32_t* table = pw;
  int32_t* rsig = reinterpret_cast<int32_t*>(table + kPwTable);
  uint32_t* tile = table + kPwTable + kPwRows * kSigMax;
  __shared__ int rlen[kPwRows];
  const int t = threadIdx.x, i0 = blockIdx.y * kPwRows, j = blockIdx.x * kPwCols + t;
  for (int q = t; q < kPwTable; q += kPwCols) table[q] = 0;
  for (int q = t; q < kPwRows * kPwCols; q += kPwCols) tile[q] = 0;
  if (t < kPwRows) rlen[t] = i0 + t < m ? (int)(off[i0 + t + 1] - off[i0 + t]) : 0;
  __syncthreads();
  for (int q = t; q < kPwRows * kSigMax; q += kPwCols) {
    const int r = q / kSigMax, k = q % kSigMax;
    if (k < rlen[r]) {
      const int32_t x = sig[off[i0 + r] + k];
      rsig[q] = x;
      atomicOr(&table[x & (kPwTable - 1)], 1u << r);
    }
  }
  __syncthreads();
  if (j < m) {
    for (int64_t q = off[j]; q < off[j + 1]; ++q) {
      const int32_t x = sig[q];
      for (uint32_t rr = table[x & (kPwTable - 1)]; rr; rr &= rr - 1) {
        const int r = __ffs(rr) - 1;
        if (i0 + r != j && find_in(rsig + r * kSigMax, rlen[r], x) >= 0) tile[r * kPwCols + t] += (uint32_t)w[x];
      }
    }
    for (int r = 0; r < kPwRows && i0 + r < m; ++r) W[(size_t)(i0 + r) * m + j] = tile[r * kPwCols + t];
  }
}

// Maximum spanning tree of W (Borůvka).  Edges are ordered by pair_key
// (weight, then the smaller slot pair), so every edge key is distinct and the
// tree is unique; its weight is the maximum spanning-tree weight (Sec. 6.3).
// Edges of no weight add nothing and are left out, so the rounds end at a
// spanning forest of the others.
// A round: each vertex's heaviest edge to another component (warp per row),
// each component's heaviest (atomicMax), components hook along them (a pair
// of components that chose the same edge keeps the smaller id as root, and
// that edge is counted once), then every vertex jumps to its root.  Every
// round at least halves the number of components.
__global__ void k_bv_vertex_best(int m, const uint32_t* __restrict__ W, const int32_t* __restrict__ comp,
                                 unsigned long long* __restrict__ cbest, const int32_t* __restrict__ state) {
  const int lane = threadIdx.x & 31;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  if (*state < 0) return;  // no component found an edge last round
  for (int v = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < m; v += warps) {
    const int cv = comp[v];
    unsigned long long b = 0;
    for (int u0 = lane; u0 < m; u0 += 32 * kAhead) {
      uint32_t x[kAhead];
#pragma unroll
      for (int q = 0; q < kAhead; ++q) x[q] = u0 + 32 * q < m ? W[(size_t)v * m + u0 + 32 * q] : 0u;
#pragma unroll
      for (int q = 0; q < kAhead; ++q) {
        const int u = u0 + 32 * q;
        if (x[q] != 0 && comp[u] != cv) b = max(b, pair_key((uint32_t)v, (uint32_t)u, x[q]));
      }
    }
    for (int off = 16; off > 0; off >>= 1) b = max(b, __shfl_xor_sync(0xFFFFFFFFu, b, off));
    if (lane == 0 && b) atomicMax(&cbest[cv], b);
  }
}

// The rest of a round, one block: components hook, vertices jump to their
// roots, the bests are reset.  *state: -1 when nothing hooked, and from then on.
__global__ void __launch_bounds__(kGreedyThreads)
k_bv_step(int m, int32_t* __restrict__ comp, unsigned long long* __restrict__ cbest, int32_t* __restrict__ parent,
          unsigned long long* __restrict__ total, int32_t* __restrict__ state) {
  if (*state < 0) return;
  unsigned long long sum = 0;
  bool any = false;
  for (int c = threadIdx.x; c < m; c += kGreedyThreads) {
    if (comp[c] != c) continue;  // not a component root
    const unsigned long long k = cbest[c];
    if (k == 0) {
      parent[c] = c;
      continue;
    }
    any = true;
    uint32_t a, b;
    key_pair(k, &a, &b);
    const int o = comp[a] == c ? comp[b] : comp[a];
    const bool mutual = cbest[o] == k;
    parent[c] = (mutual && c < o) ? c : o;
    if (!(mutual && o < c)) sum += k >> 28;
  }
  any = __syncthreads_or(any);
  for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, off);
  if ((threadIdx.x & 31) == 0 && sum) atomicAdd(total, sum);
  if (!any) {
    if (threadIdx.x == 0) *state = -1;
    return;
  }
  for (int v = threadIdx.x; v < m; v += kGreedyThreads) {
    int r = comp[v];
    for (int step = 0; step < m && parent[r] != r; ++step) r = parent[r];
    comp[v] = r;
    cbest[v] = 0;
  }
}

// ---------------------------------------------------------------------------
// Rounds of merges.
// ---------------------------------------------------------------------------
struct Slots {
  int m;
  const int64_t* off;         // signatures of the slots, in place of the requests' sorted chunks
  int32_t* sig;
  int32_t* len;
  uint32_t* W;
  unsigned long long* best;   // best pair key of an active slot; 0: it shares weight with none
  uint8_t* act;
  int32_t* mark;              // last round that merged the slot
  int32_t* top;               // the slot's node: a merge's record, or ~request
  // records, in the order they were made
  unsigned long long* rec_key;
  int2* rec_child;            // nodes of both slots before
  int32_t* rec_sig;           // [kSigMax] merged signature
  int32_t* rec_len;
  int32_t* counts;            // 0: records; 1, 2: records before this round, by its parity
};

__global__ void k_slots_init(Slots s, int32_t* __restrict__ comp, unsigned long long* __restrict__ cbest) {
  for (int d = blockIdx.x * blockDim.x + threadIdx.x; d < s.m; d += gridDim.x * blockDim.x) {
    s.len[d] = (int32_t)(s.off[d + 1] - s.off[d]);
    s.best[d] = 0;
    s.act[d] = 1;
    s.mark[d] = -1;
    s.top[d] = ~d;
    comp[d] = d;
    cbest[d] = 0;
  }
}

// Round 1 of 3: the best pair of every slot that needs looking for (all in the
// first round; then those that merged, or whose best partner did, unless it
// kept its slot and their pair its weight: other keys only fell).  Block per
// slot: a slot's scan is a chain of loads, and few slots have one, so the
// threads of a block share it.
constexpr int kBestThreads = 128;
__global__ void __launch_bounds__(kBestThreads) k_row_best(Slots s, int round) {
  __shared__ unsigned long long warp_best[kBestThreads / 32];
  const int before = s.counts[1 + ((round + 1) & 1)], now = s.counts[0];
  if (blockIdx.x == 0 && threadIdx.x == 0) s.counts[1 + (round & 1)] = now;
  if (round > 0 && now == before) return;  // no merge last round: done
  for (int d = blockIdx.x; d < s.m; d += gridDim.x) {
    if (!s.act[d]) continue;  // the same decisions in every thread
    if (round > 0 && s.mark[d] != round - 1) {
      const unsigned long long k = s.best[d];
      if (k == 0) continue;
      uint32_t a, b;
      key_pair(k, &a, &b);
      const uint32_t p = (int)a == d ? b : a;
      if (s.mark[p] != round - 1 || (s.act[p] && s.W[(size_t)d * s.m + p] == (uint32_t)(k >> 28))) continue;
    }
    unsigned long long best = 0;
    const uint32_t* row = s.W + (size_t)d * s.m;
    for (int e0 = threadIdx.x; e0 < s.m; e0 += kBestThreads * kAhead) {
      uint32_t v[kAhead];
#pragma unroll
      for (int q = 0; q < kAhead; ++q) v[q] = e0 + kBestThreads * q < s.m ? row[e0 + kBestThreads * q] : 0u;
#pragma unroll
      for (int q = 0; q < kAhead; ++q) {
        const int e = e0 + kBestThreads * q;
        if (v[q] != 0 && s.act[e]) best = max(best, pair_key((uint32_t)d, (uint32_t)e, v[q]));
      }
    }
    for (int off = 16; off > 0; off >>= 1) best = max(best, __shfl_xor_sync(0xFFFFFFFFu, best, off));
    if ((threadIdx.x & 31) == 0) warp_best[threadIdx.x >> 5] = best;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int q = 1; q < kBestThreads / 32; ++q) best = max(best, warp_best[q]);
      s.best[d] = best;
    }
    __syncthreads();
  }
}

// 2 of 3: slots that are each other's best merge; warp per smaller slot.
// Only the pair's own warp touches its slots.
__global__ void __launch_bounds__(256) k_match(Slots s, int round) {
  const int lane = threadIdx.x & 31, warps = (gridDim.x * blockDim.x) >> 5;
  for (int a = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; a < s.m; a += warps) {
    const unsigned long long k = s.best[a];
    if (k == 0 || !s.act[a]) continue;
    uint32_t ka, kb;
    key_pair(k, &ka, &kb);
    const int b = (int)kb;
    if ((int)ka != a || s.best[b] != k || !s.act[b]) continue;
    int r = 0;
    if (lane == 0) r = atomicAdd(&s.counts[0], 1);
    r = __shfl_sync(0xFFFFFFFFu, r, 0);
    // merged signature: the chunks of a that b holds, in order
    const int la = s.len[a], lb = s.len[b];
    int32_t* sa = s.sig + s.off[a];
    const int32_t* sb = s.sig + s.off[b];
    int n = 0;
    for (int base = 0; base < la; base += 32) {
      const int q = base + lane;
      const int32_t x = q < la ? sa[q] : 0;
      const bool keep = q < la && find_in(sb, lb, x) >= 0;
      const uint32_t bal = __ballot_sync(0xFFFFFFFFu, keep);
      const int o = n + __popc(bal & ((1u << lane) - 1u));
      if (keep) {
        sa[o] = x;  // o <= q, and this round of the loop has read up to base + 31
        s.rec_sig[(size_t)r * kSigMax + o] = x;
      }
      n += __popc(bal);
      __syncwarp();
    }
    if (lane == 0) {
      s.len[a] = n;
      s.rec_len[r] = n;
      s.rec_key[r] = k;
      s.rec_child[r] = make_int2(s.top[a], s.top[b]);
      s.top[a] = r;
      s.act[b] = 0;
      s.mark[a] = round;
      s.mark[b] = round;
    }
  }
}

// 3 of 3: the weights of the merged slots, block per merge of this round.
// A weight is zero where either slot's was (the merged signature is part of
// both); the others come from the signatures.  Two merged slots compute their
// pair's weight twice, and the zero tests hold for old and new weights, so
// the order of the blocks does not matter.
__global__ void __launch_bounds__(256) k_reweigh(Slots s, const int64_t* __restrict__ w, int round) {
  __shared__ int32_t s_new[kSigMax];
  const int first = s.counts[1 + (round & 1)], end = s.counts[0];
  for (int r = first + (int)blockIdx.x; r < end; r += gridDim.x) {
    uint32_t a, b;
    key_pair(s.rec_key[r], &a, &b);
    const int ln = s.rec_len[r];
    __syncthreads();
    for (int q = threadIdx.x; q < ln; q += blockDim.x) s_new[q] = s.rec_sig[(size_t)r * kSigMax + q];
    __syncthreads();
    for (int d0 = threadIdx.x; d0 < s.m; d0 += 256 * kAhead) {
      uint32_t wa[kAhead];
#pragma unroll
      for (int k = 0; k < kAhead; ++k) wa[k] = d0 + 256 * k < s.m ? s.W[(size_t)a * s.m + d0 + 256 * k] : 0u;
#pragma unroll
      for (int k = 0; k < kAhead; ++k) {
        const int d = d0 + 256 * k;
        if (wa[k] == 0 || d == (int)b || !s.act[d]) continue;
        uint32_t v = 0;
        if (s.W[(size_t)b * s.m + d] != 0) {
          const int32_t* sd = s.sig + s.off[d];
          for (int q = 0; q < s.len[d]; ++q)
            if (find_in(s_new, ln, sd[q]) >= 0) v += (uint32_t)w[sd[q]];
        }
        s.W[(size_t)a * s.m + d] = v;
        s.W[(size_t)d * s.m + a] = v;
      }
    }
  }
}

// The remaining merges one after the other, in one block.  best[d] is an upper
// bound on slot d's best key (keys only fall), kept in shared memory as sb,
// with gmax[g] the largest of sb[32 g .. 32 g + 31].  The largest key is merged
// only if it is still exact; otherwise the rows of its two slots are scanned
// again and the search repeats.  2 to 5 us a merge up to 3,000 requests with
// signatures of 8 chunks, mostly barriers; with 100 chunks (nested requests) 54
// us, 70 with a thread per other slot instead of kShare.
constexpr int kMaxGroups = kMaxGreedyM / 32;
constexpr int kNoRounds = 32, kFewRounds = 64;  // requests
constexpr int kShare = 16;
size_t rest_smem_bytes(int m) { return (size_t)m * 8 + (size_t)kMaxGroups * 8 + (size_t)m * 2 + (size_t)m; }

__device__ unsigned long long block_max_u64(unsigned long long v, unsigned long long* red) {
  for (int off = 16; off > 0; off >>= 1) v = max(v, __shfl_xor_sync(0xFFFFFFFFu, v, off));
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) red[warp] = v;
  __syncthreads();
  if (warp == 0) {
    v = lane < kGreedyThreads / 32 ? red[lane] : 0ull;
    for (int off = 16; off > 0; off >>= 1) v = max(v, __shfl_xor_sync(0xFFFFFFFFu, v, off));
    if (lane == 0) red[32] = v;
  }
  __syncthreads();
  const unsigned long long r = red[32];
  __syncthreads();
  return r;
}

__global__ void __launch_bounds__(kGreedyThreads) k_merge_rest(Slots s, const int64_t* __restrict__ w) {
  extern __shared__ __align__(16) unsigned char gsm[];
  unsigned long long* sb = reinterpret_cast<unsigned long long*>(gsm);  // [m]
  unsigned long long* gmax = sb + s.m;                                  // [kMaxGroups]
  uint16_t* live = reinterpret_cast<uint16_t*>(gmax + kMaxGroups);      // [m]
  uint8_t* act = reinterpret_cast<uint8_t*>(live + s.m);                // [m]
  __shared__ int live_n;
  __shared__ unsigned long long red[33];
  __shared__ int32_t s_b[kSigMax], s_new[kSigMax];
  __shared__ int warp_n[kSigMax / 32];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, m = s.m, groups = (m + 31) / 32;
  // the largest of a group's bounds; by the first warp
  auto refresh = [&](int g) {
    if (t < 32) {
      const int d = g * 32 + t;
      unsigned long long v = d < m ? sb[d] : 0ull;
      for (int off = 16; off > 0; off >>= 1) v = max(v, __shfl_xor_sync(0xFFFFFFFFu, v, off));
      if (t == 0) gmax[g] = v;
    }
  };
  auto rescan = [&](int d) {
    unsigned long long best = 0;
    const uint32_t* row = s.W + (size_t)d * m;
    for (int e0 = t; e0 < m; e0 += kGreedyThreads * 4) {
      uint32_t v[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) v[q] = e0 + kGreedyThreads * q < m ? row[e0 + kGreedyThreads * q] : 0u;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int e = e0 + kGreedyThreads * q;
        if (v[q] != 0 && act[e]) best = max(best, pair_key((uint32_t)d, (uint32_t)e, v[q]));
      }
    }
    best = block_max_u64(best, red);
    if (t == 0) sb[d] = best;
    __syncthreads();
    refresh(d >> 5);
  };
  for (int d = t; d < m; d += kGreedyThreads) {
    act[d] = s.act[d];
    sb[d] = s.act[d] ? s.best[d] : 0ull;
  }
  __syncthreads();
  for (int g = warp; g < groups; g += kGreedyThreads / 32) {
    const int d = g * 32 + lane;
    unsigned long long v = d < m ? sb[d] : 0ull;
    for (int off = 16; off > 0; off >>= 1) v = max(v, __shfl_xor_sync(0xFFFFFFFFu, v, off));
    if (lane == 0) gmax[g] = v;
  }
  __syncthreads();
  int r = s.counts[0];
  for (int tries = 0; r < m - 1 && tries <= m;) {  // a rescan makes a row exact: at most m between two merges
    const unsigned long long top = block_max_u64(t < groups ? gmax[t] : 0ull, red);
    if (top == 0) break;  // no pair shares weight
    uint32_t a, b;
    key_pair(top, &a, &b);
    if (!act[a] || !act[b] || s.W[(size_t)a * m + b] != (uint32_t)(top >> 28)) {
      ++tries;
      if (act[a]) rescan((int)a);
      if (act[b]) rescan((int)b);
      __syncthreads();
      continue;
    }
    tries = 0;
    // merged signature: the chunks of a that b holds, in order
    const int la = s.len[a], lb = s.len[b];
    int32_t* sa = s.sig + s.off[a];
    const int32_t x = t < la ? sa[t] : 0;
    if (t < lb) s_b[t] = s.sig[s.off[b] + t];
    __syncthreads();
    const bool keep = t < la && find_in(s_b, lb, x) >= 0;
    const uint32_t bal = __ballot_sync(0xFFFFFFFFu, keep);
    if (lane == 0 && warp < kSigMax / 32) warp_n[warp] = __popc(bal);
    __syncthreads();
    int ln = 0;
    for (int q = 0; q < kSigMax / 32; ++q) ln += warp_n[q];
    if (keep) {
      int o = __popc(bal & ((1u << lane) - 1u));
      for (int q = 0; q < warp; ++q) o += warp_n[q];
      s_new[o] = x;
    }
    __syncthreads();
    if (t < ln) {
      sa[t] = s_new[t];
      s.rec_sig[(size_t)r * kSigMax + t] = s_new[t];
    }
    if (t == 0) {
      s.len[a] = ln;
      s.rec_len[r] = ln;
      s.rec_key[r] = top;
      s.rec_child[r] = make_int2(s.top[a], s.top[b]);
      s.top[a] = r;
      s.act[b] = act[b] = 0;
      sb[b] = 0;
    }
    __syncthreads();
    // its weights (zero where either slot's was), and its best pair on the way;
    // with long signatures, kShare threads per other slot
    unsigned long long best = 0;
    auto put = [&](int d, uint32_t wa, uint32_t v) {
      if (v != wa) {
        s.W[(size_t)a * m + d] = v;
        s.W[(size_t)d * m + a] = v;
      }
      if (v != 0) best = max(best, pair_key(a, (uint32_t)d, v));
    };
    auto shared_weight = [&](int d, int first, int step) {
      const int32_t* sd = s.sig + s.off[d];
      const int ld = s.len[d];
      uint32_t v = 0;
      for (int q = first; q < ld; q += step) {
        const int32_t x = sd[q];
        if (find_in(s_new, ln, x) >= 0) v += (uint32_t)w[x];
      }
      return v;
    };
    if (t == 0) live_n = 0;
    __syncthreads();
    for (int d = t; d < m; d += kGreedyThreads) {
      const uint32_t wa = s.W[(size_t)a * m + d];
      if (wa == 0 || !act[d]) continue;
      if (s.W[(size_t)b * m + d] == 0)
        put(d, wa, 0u);
      else if (ln <= kShare)
        put(d, wa, shared_weight(d, 0, 1));
      else
        live[atomicAdd(&live_n, 1)] = (uint16_t)d;
    }
    if (ln > kShare) {
      __syncthreads();
      for (int i0 = 0; i0 < live_n; i0 += kGreedyThreads / kShare) {
        const int i = i0 + t / kShare;
        uint32_t v = i < live_n ? shared_weight(live[i], t % kShare, kShare) : 0u;
        for (int off = 1; off < kShare; off <<= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
        if (i < live_n && t % kShare == 0) put(live[i], s.W[(size_t)a * m + live[i]], v);
      }
    }
    best = block_max_u64(best, red);
    if (t == 0) sb[a] = best;
    __syncthreads();
    refresh((int)a >> 5);
    if ((b >> 5) != (a >> 5)) {
      __syncthreads();
      refresh((int)b >> 5);
    }
    __syncthreads();
    ++r;
  }
  if (t == 0) s.counts[0] = r;
}

// ---------------------------------------------------------------------------
// The sequence and the tree.  Node of merge t: m + t.
// ---------------------------------------------------------------------------
struct Tree {
  int32_t* merges;    // [2 (m - 1)] slot pairs
  int64_t* values;    // [m - 1]
  int32_t* rank;      // position of each record in the sequence
  int32_t* rec_of;    // record of merge t, -1 for a forced one
  int32_t* children;  // [2 (m - 1)] nodes
  int32_t* parent;    // [2 m - 1]
  int32_t* leaves;    // [m - 1] leaves below a recorded merge
  int32_t* base;      // [m] leaves in front of a remaining slot's subtree
  int32_t* dfs;       // [m]
};

// Records in decreasing key order; warp per record.
__global__ void __launch_bounds__(256) k_rank(Slots s, Tree tr) {
  const int lane = threadIdx.x & 31, warps = (gridDim.x * blockDim.x) >> 5, n = s.counts[0];
  for (int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < n; r += warps) {
    const unsigned long long k = s.rec_key[r];
    int above = 0;
    for (int q = lane; q < n; q += 32) above += s.rec_key[q] > k;
    above = __reduce_add_sync(0xFFFFFFFFu, above);
    if (lane == 0) {
      uint32_t a, b;
      key_pair(k, &a, &b);
      tr.rank[r] = above;
      tr.rec_of[above] = r;
      tr.merges[2 * above] = (int32_t)a;
      tr.merges[2 * above + 1] = (int32_t)b;
      tr.values[above] = (int64_t)(k >> 28);
      tr.leaves[above] = 0;
    }
  }
}

__device__ __forceinline__ int node_of(const Slots& s, const Tree& tr, int top) {
  return top < 0 ? ~top : s.m + tr.rank[top];
}

// Children and parents of the recorded merges.
__global__ void k_link(Slots s, Tree tr) {
  const int n = s.counts[0];
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) {
    const int t = tr.rank[r];
    const int2 c = s.rec_child[r];
    const int x = node_of(s, tr, c.x), y = node_of(s, tr, c.y);
    tr.children[2 * t] = x;
    tr.children[2 * t + 1] = y;
    tr.parent[x] = s.m + t;
    tr.parent[y] = s.m + t;
  }
}

// Leaves below every recorded merge.
__global__ void k_count(Slots s, Tree tr) {
  const int top = s.m + s.counts[0];
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < s.m; i += gridDim.x * blockDim.x) {
    // a node whose slot is still active has no parent yet (k_tail's come later)
    for (int v = tr.parent[i]; v >= 0 && v < top; v = tr.parent[v]) atomicAdd(&tr.leaves[v - s.m], 1);
  }
}

// The forced merges, one block: the remaining slots s_0 < s_1 < .. in order,
// merge j joins s_0's cluster with s_j; and the leaves in front of each.
__global__ void __launch_bounds__(kGreedyThreads) k_tail(Slots s, Tree tr) {
  __shared__ int warp_n[kGreedyThreads / 32], warp_l[kGreedyThreads / 32], s_first;
  const int n = s.counts[0], t = threadIdx.x, lane = t & 31, warp = t >> 5;
  int found = 0, leaves = 0;
  for (int d0 = 0; d0 < s.m; d0 += kGreedyThreads) {
    const int d = d0 + t;
    const bool here = d < s.m && s.act[d];
    const int node = here ? node_of(s, tr, s.top[d]) : 0;
    const int mine = here ? (node < s.m ? 1 : tr.leaves[node - s.m]) : 0;
    const uint32_t bal = __ballot_sync(0xFFFFFFFFu, here);
    int in = mine;
    for (int off = 1; off < 32; off <<= 1) {
      const int o = __shfl_up_sync(0xFFFFFFFFu, in, off);
      if (lane >= off) in += o;
    }
    if (lane == 31) {
      warp_n[warp] = __popc(bal);
      warp_l[warp] = in;
    }
    __syncthreads();
    int at = found + __popc(bal & ((1u << lane) - 1u)), before = leaves + in - mine;
    for (int q = 0; q < kGreedyThreads / 32; ++q) {
      if (q < warp) {
        at += warp_n[q];
        before += warp_l[q];
      }
      found += warp_n[q];
      leaves += warp_l[q];
    }
    if (here) {
      tr.base[d] = before;
      if (at == 0) s_first = d;
    }
    __syncthreads();
    if (here && at > 0) {
      const int j = n + at - 1;  // merge number
      const int left = at == 1 ? node_of(s, tr, s.top[s_first]) : s.m + j - 1;
      tr.merges[2 * j] = s_first;
      tr.merges[2 * j + 1] = d;
      tr.values[j] = 0;
      tr.rec_of[j] = -1;
      tr.children[2 * j] = left;
      tr.children[2 * j + 1] = node;
      tr.parent[node] = s.m + j;
      tr.parent[left] = s.m + j;
    }
  }
}

// Left-to-right leaf order: leaves in front of leaf i inside the subtree of its
// remaining slot, plus that slot's base.
__global__ void k_leaf_order(Slots s, Tree tr) {
  const int top = s.m + s.counts[0];
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < s.m; i += gridDim.x * blockDim.x) {
    int v = i, pos = 0, slot = i;
    for (int p = tr.parent[v]; p >= 0 && p < top; p = tr.parent[v]) {
      const int left = tr.children[2 * (p - s.m)];
      if (left != v) pos += left < s.m ? 1 : tr.leaves[left - s.m];
      slot = tr.merges[2 * (p - s.m)];
      v = p;
    }
    tr.dfs[tr.base[slot] + pos] = i;
  }
}

// Emission key of every (request, chunk) occurrence: climb from the leaf
// while the parent's signature still holds the chunk.  On a path the later
// merges are nearer the root, so merges in decreasing number, then the leaf,
// are its nodes from the root down.
__global__ void k_greedy_emit(Slots s, Tree tr, const int32_t* __restrict__ chunks,
                              unsigned long long* __restrict__ keys) {
  const int64_t occ = s.off[s.m];
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < occ; j += (int64_t)gridDim.x * blockDim.x) {
    int lo = 0, hi = s.m - 1;  // request of occurrence j: the last i with off[i] <= j
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (s.off[mid] <= j) lo = mid; else hi = mid - 1;
    }
    const int32_t x = chunks[j];
    int v = lo;
    for (;;) {
      const int p = tr.parent[v];
      if (p < 0) break;
      const int r = tr.rec_of[p - s.m];
      if (r < 0 || find_in(s.rec_sig + (size_t)r * kSigMax, s.rec_len[r], x) < 0) break;
      v = p;
    }
    const uint32_t from_root = v < s.m ? 2u * (uint32_t)s.m : 2u * (uint32_t)s.m - (uint32_t)v;
    keys[j] = ((unsigned long long)from_root << 32) | (unsigned long long)(uint32_t)x;
  }
}

// Each request's chunks in the order of their keys: warp per request.
__global__ void k_greedy_rank(int m, const int64_t* __restrict__ req_off, const unsigned long long* __restrict__ keys,
                              int64_t* __restrict__ perm) {
  const int lane = threadIdx.x & 31;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < m; i += warps) {
    const int64_t base = req_off[i];
    const int len = (int)(req_off[i + 1] - base);
    for (int q = lane; q < len; q += 32) {
      const unsigned long long kq = keys[base + q];
      int rank = 0;
      for (int r = 0; r < len; ++r) rank += keys[base + r] < kq;
      perm[base + rank] = (int64_t)(kq & 0xFFFFFFFFull);
    }
  }
}

}  // namespace
}  // namespace mpt

extern "C" mpt_status mpt_greedy(const int64_t* weights, int64_t n_chunks, int32_t m, const int64_t* req_offsets,
                                 const int64_t* chunk_ids, void* stream_ptr, int64_t* cost, int64_t* savings,
                                 int64_t* lower_bound, int32_t* merges, int64_t* merge_values, int64_t* perm_chunks,
                                 int32_t* dfs_order) {
  using namespace mpt;
  if (!weights || !req_offsets || n_chunks < 1 || n_chunks > INT32_MAX || m < 1) return MPT_ERR_INVALID_ARG;
  if (m > kMaxGreedyM) return MPT_ERR_TOO_LARGE;
  if (req_offsets[0] != 0) return MPT_ERR_INVALID_ARG;
  const int64_t occ = req_offsets[m];
  if (occ > 0 && !chunk_ids) return MPT_ERR_INVALID_ARG;
  for (int64_t x = 0; x < n_chunks; ++x)
    if (weights[x] <= 0) return MPT_ERR_INVALID_ARG;
  // sorted, de-duplicated-checked signatures; per-request weight < 2^32
  std::vector<int32_t> sig;
  int64_t total = 0;
  try {
    int64_t ids[kSigMax];
    for (int i = 0; i < m; ++i) {
      const int64_t a = req_offsets[i], b = req_offsets[i + 1];
      if (b < a) return MPT_ERR_INVALID_ARG;
      if (b - a > kSigMax) return MPT_ERR_TOO_LARGE;
      std::copy(chunk_ids + a, chunk_ids + b, ids);
      std::sort(ids, ids + (b - a));
      int64_t rw = 0;
      for (int64_t q = 0; q < b - a; ++q) {
        if (ids[q] < 0 || ids[q] >= n_chunks || (q > 0 && ids[q] == ids[q - 1])) return MPT_ERR_INVALID_ARG;
        sig.push_back((int32_t)ids[q]);
        rw += weights[ids[q]];
        if (rw >= ((int64_t)1 << 32)) return MPT_ERR_OVERFLOW;
      }
      total += rw;
    }
  } catch (...) {
    return MPT_ERR_OUT_OF_MEMORY;
  }
  cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_ptr);
  // device buffers (this call allocates and frees its own)
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off += (bytes + 255) & ~(size_t)255;
    return o;
  };
  const size_t M = (size_t)m;
  const size_t O = (size_t)std::max<int64_t>(occ, 1);
  const size_t o_w = take((size_t)n_chunks * 8), o_off = take((M + 1) * 8), o_sig = take(O * 4), o_chunks = take(O * 4),
               o_len = take(M * 4), o_W = take(M * M * 4), o_best = take(M * 8), o_act = take(M), o_mark = take(M * 4),
               o_top = take(M * 4), o_key = take(M * 8), o_child = take(M * 8), o_rsig = take(M * kSigMax * 4),
               o_rlen = take(M * 4), o_merges = take(M * 8), o_val = take(M * 8), o_rank = take(M * 4),
               o_rec = take(M * 4), o_children = take(M * 8), o_par = take(2 * M * 4), o_leaves = take(M * 4),
               o_base = take(M * 4), o_dfs = take(M * 4), o_keys = take(O * 8), o_perm = take(O * 8),
               o_comp = take(M * 4), o_bpar = take(M * 4), o_cbest = take(M * 8), o_ctl = take(32);
  char* d = nullptr;
  if (device_alloc(reinterpret_cast<void**>(&d), off) != cudaSuccess) return MPT_ERR_OUT_OF_MEMORY;
  const int64_t sms = sm_count();
  mpt_status st = MPT_OK;
  cudaError_t e = cudaSuccess;
  auto h2d = [&](size_t o, const void* h, size_t bytes) {
    if (e == cudaSuccess && bytes) e = cudaMemcpyAsync(d + o, h, bytes, cudaMemcpyHostToDevice, stream);
  };
  auto d2h = [&](void* h, size_t o, size_t bytes) {
    if (e == cudaSuccess && bytes && h) e = cudaMemcpyAsync(h, d + o, bytes, cudaMemcpyDeviceToHost, stream);
  };
  auto I64 = [&](size_t o) { return reinterpret_cast<int64_t*>(d + o); };
  auto I32 = [&](size_t o) { return reinterpret_cast<int32_t*>(d + o); };
  auto U32 = [&](size_t o) { return reinterpret_cast<uint32_t*>(d + o); };
  auto U64 = [&](size_t o) { return reinterpret_cast<unsigned long long*>(d + o); };
  // control words: 0-2 the counts of the rounds, 3 the state of Borůvka's, 4-5 the tree weight
  int32_t* ctl = I32(o_ctl);
  const Slots sl{m, I64(o_off), I32(o_sig), I32(o_len), U32(o_W), U64(o_best), reinterpret_cast<uint8_t*>(d + o_act),
                 I32(o_mark), I32(o_top), U64(o_key), reinterpret_cast<int2*>(d + o_child), I32(o_rsig), I32(o_rlen),
                 ctl};
  const Tree tr{I32(o_merges), I64(o_val), I32(o_rank), I32(o_rec), I32(o_children), I32(o_par), I32(o_leaves),
                I32(o_base), I32(o_dfs)};
  h2d(o_w, weights, (size_t)n_chunks * 8);
  h2d(o_off, req_offsets, (M + 1) * 8);
  h2d(o_sig, sig.data(), (size_t)occ * 4);
  if (e == cudaSuccess && occ)
    e = cudaMemcpyAsync(d + o_chunks, d + o_sig, (size_t)occ * 4, cudaMemcpyDeviceToDevice, stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(d + o_ctl, 0, 32, stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(d + o_par, 0xFF, 2 * M * 4, stream);
  const unsigned wb = (unsigned)std::min<int64_t>(((int64_t)m * 32 + 255) / 256, sms * 8);  // a warp per slot
  const unsigned tb = (unsigned)std::min<int64_t>((m + 255) / 256, sms * 8);               // a thread per slot
  if (e == cudaSuccess) {
    k_slots_init<<<tb, 256, 0, stream>>>(sl, I32(o_comp), U64(o_cbest));
    e = cudaFuncSetAttribute(k_pair_weights, cudaFuncAttributeMaxDynamicSharedMemorySize, kPwSmem);
  }
  if (e == cudaSuccess) {
    const dim3 grid((unsigned)((m + kPwCols - 1) / kPwCols), (unsigned)((m + kPwRows - 1) / kPwRows));
    k_pair_weights<<<grid, kPwCols, kPwSmem, stream>>>(m, I64(o_off), I32(o_sig), I64(o_w), U32(o_W));
    // maximum spanning tree by Borůvka rounds (each at least halves the
    // components that still have an edge)
    int rounds = 1;
    while ((1 << rounds) < m) ++rounds;
    for (int r = 0; r < rounds; ++r) {
      k_bv_vertex_best<<<wb, 256, 0, stream>>>(m, U32(o_W), I32(o_comp), U64(o_cbest), ctl + 3);
      k_bv_step<<<1, kGreedyThreads, 0, stream>>>(m, I32(o_comp), U64(o_cbest), I32(o_bpar),
                                                  reinterpret_cast<unsigned long long*>(ctl + 4), ctl + 3);
    }
    e = cudaGetLastError();
  }
  // Rounds of merges, `ahead` enqueued between two looks at what they merged
  // (nothing, once no pair shares weight; later rounds return at once).  Where
  // keys tie or wait for one another a round merges a pair or two, and the rest
  // goes to one block (2 to 5 us a merge with signatures of 8 chunks, a round 9
  // us).  Few requests go there at once, or after a few rounds without a look.
  int ahead = 2;
  while (ahead < 12 && (1 << ahead) < 4 * m) ++ahead;  // 2 + log2(m), rounded up
  if (m <= kFewRounds) ahead = m <= kNoRounds ? 0 : 4;
  int32_t counts[3] = {0, 0, 0};
  bool rest = m <= kFewRounds;
  for (int round = 0, merged = 0; e == cudaSuccess && m > 1; merged = counts[0]) {
    for (int k = 0; k < ahead; ++k, ++round) {
      k_row_best<<<(unsigned)m, kBestThreads, 0, stream>>>(sl, round);
      k_match<<<wb, 256, 0, stream>>>(sl, round);
      k_reweigh<<<(unsigned)std::min<int64_t>(m, sms * 4), 256, 0, stream>>>(sl, I64(o_w), round);
    }
    if (ahead == 0) k_row_best<<<(unsigned)m, kBestThreads, 0, stream>>>(sl, 0);
    e = cudaGetLastError();
    if (rest) break;
    if (e == cudaSuccess) e = cudaMemcpyAsync(counts, ctl, 12, cudaMemcpyDeviceToHost, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess || counts[0] == counts[1 + ((round - 1) & 1)]) break;
    rest = 2 * (counts[0] - merged) < 5 * ahead;
    if (rest) break;
  }
  if (e == cudaSuccess && rest && m > 1) {
    e = cudaFuncSetAttribute(k_merge_rest, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rest_smem_bytes(m));
    if (e == cudaSuccess) {
      k_merge_rest<<<1, kGreedyThreads, rest_smem_bytes(m), stream>>>(sl, I64(o_w));
      e = cudaGetLastError();
    }
  }
  if (e == cudaSuccess && st == MPT_OK) {
    k_rank<<<wb, 256, 0, stream>>>(sl, tr);
    k_link<<<tb, 256, 0, stream>>>(sl, tr);
    k_count<<<tb, 256, 0, stream>>>(sl, tr);
    k_tail<<<1, kGreedyThreads, 0, stream>>>(sl, tr);
    k_leaf_order<<<tb, 256, 0, stream>>>(sl, tr);
    const int64_t eblocks = std::min<int64_t>(((int64_t)O + 255) / 256, sms * 16);
    k_greedy_emit<<<(unsigned)eblocks, 256, 0, stream>>>(sl, tr, I32(o_chunks), U64(o_keys));
    k_greedy_rank<<<wb, 256, 0, stream>>>(m, I64(o_off), U64(o_keys), I64(o_perm));
    e = cudaGetLastError();
  }
  std::vector<int64_t> vals;
  unsigned long long mst = 0;
  try {
    vals.assign(M > 1 ? M - 1 : 1, 0);
  } catch (...) {
    if (st == MPT_OK) st = MPT_ERR_OUT_OF_MEMORY;
  }
  if (st == MPT_OK) {
    d2h(vals.data(), o_val, (M - 1) * 8);
    d2h(&mst, o_ctl + 16, 8);
    d2h(merges, o_merges, (M - 1) * 2 * 4);
    d2h(perm_chunks, o_perm, (size_t)occ * 8);
    d2h(dfs_order, o_dfs, M * 4);
  }
  const cudaError_t es = cudaStreamSynchronize(stream);
  if (e == cudaSuccess) e = es;
  if (e != cudaSuccess) st = MPT_ERR_CUDA;
  cudaFree(d);
  if (st != MPT_OK) return st;
  int64_t sav = 0;
  for (size_t t = 0; t + 1 < M; ++t) sav += vals[t];
  if (merge_values && M > 1) std::copy(vals.begin(), vals.begin() + (M - 1), merge_values);
  if (savings) *savings = sav;
  if (cost) *cost = total - sav;
  if (lower_bound) *lower_bound = total - (int64_t)mst;
  return MPT_OK;
}
