// Serving order and finite radix cache (Sec. 8, Thm 7), and eq. (1) for many
// strings.
//
// Strings are laid-out requests (chunk ids).  Everything here starts from
// their lexicographic order (a string before its extensions), built by a
// merge sort whose keys are the strings' first chunks:
//   * Thm 7's serving order is that order (the DFS order of the trie), or,
//     with a bounded reorder window, that order inside each window;
//   * the trie of eq. (1): in lexicographic order, string x shares exactly
//     lcp[x] = lcp(string x-1, string x) nodes with all earlier strings, so
//     the trie weight is sum_x w(suffix of x after lcp[x]), and the node of
//     (x, depth s) is the one created by the last y <= x with lcp[y] <= s;
//   * the radix cache with LRU leaf eviction (Sec. 8).  Serving a request
//     touches every node on its root path; a node's last touch is never older
//     than its descendants', so the least recently used leaf is the least
//     recently used node, deepest first among a request's own path.  Evicting
//     in that order keeps the cache equal to the longest prefix of the
//     recency order (last touch descending, depth ascending) whose weight fits
//     the capacity C.  A node on request t's path is therefore a hit iff the
//     weight of the recency order up to and including it, d, is <= C -- one
//     number per access serves every capacity at once.  For the node v at
//     depth q of request t, last touched by request j < t,
//         d = sum over r in (j, t) of w(nodes of r's path not touched again before t)
//           + w(ancestors-or-self of v whose last touch before t is j).
#include <algorithm>
#include <climits>
#include <cstring>
#include <memory>
#include <utility>
#include <vector>

#include "../../include/mpt.h"
#include "mpt_internal.cuh"

namespace mpt {
namespace {

// Exclusive prefix sum of uint32 values in place (n <= 2048 * 16384).
constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;
constexpr int kScanSumThreads = 1024;
constexpr int kScanSumItems = 16;

template <int kThreads>
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* total) {
  __shared__ uint32_t warp_sums[kThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, off);
    if (lane >= off) x += y;
  }
  if (lane == 31) warp_sums[warp] = x;
  __syncthreads();
  if (warp == 0) {
    uint32_t s = lane < kThreads / 32 ? warp_sums[lane] : 0u;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, s, off);
      if (lane >= off) s += y;
    }
    if (lane < kThreads / 32) warp_sums[lane] = s;
  }
  __syncthreads();
  const uint32_t before = (warp > 0 ? warp_sums[warp - 1] : 0u) + x - v;
  *total = warp_sums[kThreads / 32 - 1];
  __syncthreads();
  return before;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_tiles(uint32_t* __restrict__ a, int64_t n, uint32_t* __restrict__ sums) {
  const int64_t first = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
  uint32_t v[kScanItems];
  uint32_t local = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    v[i] = first + i < n ? a[first + i] : 0u;
    local += v[i];
  }
  uint32_t total;
  uint32_t run = block_exclusive_scan<kScanThreads>(local, &total);
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    if (first + i < n) a[first + i] = run;
    run += v[i];
  }
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

__global__ void __launch_bounds__(kScanSumThreads) k_scan_sums(uint32_t* __restrict__ sums, int count) {
  const int first = threadIdx.x * kScanSumItems;
  uint32_t v[kScanSumItems];
  uint32_t local = 0;
#pragma unroll
  for (int i = 0; i < kScanSumItems; ++i) {
    v[i] = first + i < count ? sums[first + i] : 0u;
    local += v[i];
  }
  uint32_t total;
  uint32_t run = block_exclusive_scan<kScanSumThreads>(local, &total);
#pragma unroll
  for (int i = 0; i < kScanSumItems; ++i) {
    if (first + i < count) sums[first + i] = run;
    run += v[i];
  }
}

__global__ void __launch_bounds__(kScanThreads) k_scan_add(uint32_t* __restrict__ a, int64_t n, const uint32_t* __restrict__ sums) {
  const int64_t first = (int64_t)blockIdx.x * kScanTile;
  const uint32_t add = sums[blockIdx.x];
  for (int i = threadIdx.x; i < kScanTile; i += kScanThreads) {
    const int64_t idx = first + i;
    if (idx < n) a[idx] += add;
  }
}

constexpr int64_t kScanMax = (int64_t)kScanTile * kScanSumThreads * kScanSumItems;

int64_t scan_tiles(int64_t n) { return (n + kScanTile - 1) / kScanTile; }

cudaError_t exclusive_scan(uint32_t* a, int64_t n, uint32_t* sums, cudaStream_t st, int* launches) {
  if (n <= 0) return cudaSuccess;
  if (n > kScanMax) return cudaErrorInvalidValue;
  const int tiles = (int)scan_tiles(n);
  k_scan_tiles<<<tiles, kScanThreads, 0, st>>>(a, n, sums);
  k_scan_sums<<<1, kScanSumThreads, 0, st>>>(sums, tiles);
  k_scan_add<<<tiles, kScanThreads, 0, st>>>(a, n, sums);
  *launches += 3;
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Merge sort of (uint64 key, uint32 id) by key, then by a rule on the ids that
// leaves no two equal.  Tiles of kSortTile pairs are sorted in shared memory
// (bitonic); a pass then joins four runs at a time, every pair finding its
// place by a binary search in the other three.  It replaces a stable radix sort
// per 8 key bits and string position, 88 launches of 2 to 8 us for 2,921
// strings of 8 chunks and 128 for 100,000: two launches here up to 4,096 pairs,
// five up to 262,144.  Tiles of 4,096 took 52 us each, 78 steps of one block,
// where four smaller ones and a pass take 21 us.  The searches of a pass are its time (a chain of
// log2(run) reads from L2), so four runs a pass: two would double the passes,
// eight more than double the reads of each.
// ---------------------------------------------------------------------------
constexpr int kSortTile = 1024;
constexpr int kSortThreads = 512;

// Keys that are all different, or hold whole strings: equal ones by index.
struct ByKey {
  __device__ __forceinline__ bool less_tie(uint32_t a, uint32_t b) const { return a < b; }
};

// Strings whose first `packed` chunks are equal (they are the key): by the
// rest, a string before its extensions, then by index.
struct ByString {
  const int64_t* off;
  const int32_t* chunk;
  int64_t packed;
  __device__ __forceinline__ bool less_tie(uint32_t a, uint32_t b) const {
    if (a == b || a == 0xFFFFFFFFu || b == 0xFFFFFFFFu) return a < b;  // the last: padding of a tile
    const int64_t ba = off[a], la = off[a + 1] - ba, bb = off[b], lb = off[b + 1] - bb;
    const int64_t lim = la < lb ? la : lb;
    for (int64_t s = packed; s < lim; ++s) {
      const int32_t x = chunk[ba + s], y = chunk[bb + s];
      if (x != y) return x < y;
    }
    return la != lb && (la > packed || lb > packed) ? la < lb : a < b;
  }
};

template <typename Rule>
__device__ __forceinline__ bool pair_less(unsigned long long ka, uint32_t a, unsigned long long kb, uint32_t b,
                                          const Rule& rule) {
  return ka != kb ? ka < kb : rule.less_tie(a, b);
}

template <typename Rule>
__global__ void __launch_bounds__(kSortThreads)
k_sort_tiles(unsigned long long* __restrict__ keys, uint32_t* __restrict__ ids, int64_t n, Rule rule) {
  extern __shared__ __align__(16) unsigned long long sk[];
  uint32_t* si = reinterpret_cast<uint32_t*>(sk + kSortTile);
  const int64_t start = (int64_t)blockIdx.x * kSortTile;
  const int count = (int)(n - start < kSortTile ? n - start : kSortTile);
  int size = 64;  // power of two that holds the tile
  while (size < count) size <<= 1;
  for (int i = threadIdx.x; i < size; i += kSortThreads) {
    sk[i] = i < count ? keys[start + i] : ~0ull;
    si[i] = i < count ? ids[start + i] : 0xFFFFFFFFu;
  }
  for (int width = 2; width <= size; width <<= 1) {
    for (int step = width >> 1; step > 0; step >>= 1) {
      __syncthreads();
      for (int p = threadIdx.x; p < size / 2; p += kSortThreads) {
        const int i = ((p & ~(step - 1)) << 1) | (p & (step - 1)), j = i | step;
        const unsigned long long ki = sk[i], kj = sk[j];
        const uint32_t a = si[i], c = si[j];
        const bool up = (i & width) == 0;
        if (pair_less(kj, c, ki, a, rule) == up) {
          sk[i] = kj;
          sk[j] = ki;
          si[i] = c;
          si[j] = a;
        }
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < count; i += kSortThreads) {
    keys[start + i] = sk[i];
    ids[start + i] = si[i];
  }
}

// Joins runs 4g .. 4g + 3 of `run` sorted pairs into one.
template <typename Rule>
__global__ void __launch_bounds__(256)
k_sort_merge(const unsigned long long* __restrict__ keys, const uint32_t* __restrict__ ids,
             unsigned long long* __restrict__ kout, uint32_t* __restrict__ iout, int64_t n, int64_t run, Rule rule) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const unsigned long long k = keys[i];
    const uint32_t id = ids[i];
    const int64_t own = i / run, first = own & ~(int64_t)3;
    int64_t lo[3], hi[3], rank = i - own * run;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const int64_t other = first + (q < (int)(own - first) ? q : q + 1);
      lo[q] = other * run < n ? other * run : n;
      hi[q] = (other + 1) * run < n ? (other + 1) * run : n;
      rank -= lo[q];
    }
    // pairs of the other runs that come before this one, the three searches in step
    while (lo[0] < hi[0] || lo[1] < hi[1] || lo[2] < hi[2]) {
      int64_t mid[3];
      unsigned long long km[3];
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        mid[q] = (lo[q] + hi[q]) >> 1;
        km[q] = lo[q] < hi[q] ? keys[mid[q]] : 0ull;
      }
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        if (lo[q] < hi[q]) {
          if (km[q] != k ? km[q] < k : rule.less_tie(ids[mid[q]], id))
            lo[q] = mid[q] + 1;
          else
            hi[q] = mid[q];
        }
      }
    }
    const int64_t to = first * run + rank + lo[0] + lo[1] + lo[2];
    kout[to] = k;
    iout[to] = id;
  }
}

// Sorts (*keys, *ids); the sorted arrays end up in *keys / *ids (the pointers
// may be swapped with the second buffers).
template <typename Rule>
cudaError_t merge_sort(unsigned long long** keys, uint32_t** ids, unsigned long long** k2, uint32_t** i2, int64_t n,
                       const Rule& rule, cudaStream_t st, int* launches) {
  if (n <= 1) return cudaSuccess;
  constexpr int kBytes = kSortTile * 12;
  auto tiles = k_sort_tiles<Rule>;
  cudaError_t e = cudaFuncSetAttribute(tiles, cudaFuncAttributeMaxDynamicSharedMemorySize, kBytes);
  if (e != cudaSuccess) return e;
  tiles<<<(unsigned)((n + kSortTile - 1) / kSortTile), kSortThreads, kBytes, st>>>(*keys, *ids, n, rule);
  ++*launches;
  for (int64_t run = kSortTile; run < n; run *= 4) {
    int64_t blocks = (n + 255) / 256;
    const int64_t cap = sm_count() * 64;
    if (blocks > cap) blocks = cap;
    k_sort_merge<<<(unsigned)blocks, 256, 0, st>>>(*keys, *ids, *k2, *i2, n, run, rule);
    ++*launches;
    std::swap(*keys, *k2);
    std::swap(*ids, *i2);
  }
  return cudaGetLastError();
}

int bits_for(uint64_t max_value) {
  int b = 0;
  while (b < 64 && (max_value >> b) != 0) ++b;
  return b;
}

// ---------------------------------------------------------------------------
// Lexicographic order of the strings.
// ---------------------------------------------------------------------------
constexpr int kThreads = 256;

// blocks of kThreads for n items, at most per_sm per SM (grid-stride loops)
unsigned grid_for(int64_t n, int64_t per_sm = 32) {
  int64_t b = (n + kThreads - 1) / kThreads;
  const int64_t cap = sm_count() * per_sm;
  if (b > cap) b = cap;
  return (unsigned)(b < 1 ? 1 : b);
}

// Sort key of every string: its window (arrival position / window; window 0:
// none), then its first `packed` chunks + 1 at `bits` bits each, 0 past its
// end.  arrival (may be null: 0, 1, ..) lists the requests as they arrive.
__global__ void k_lex_keys(int64_t m, const int64_t* __restrict__ off, const int32_t* __restrict__ chunk,
                           const int32_t* __restrict__ arrival, int64_t window, int packed, int bits,
                           unsigned long long* __restrict__ keys, uint32_t* __restrict__ ids) {
  for (int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; a < m; a += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = arrival ? arrival[a] : a;
    const int64_t b = off[r], len = off[r + 1] - b;
    unsigned long long k = window > 0 ? (unsigned long long)(a / window) : 0ull;
    for (int s = 0; s < packed; ++s) k = (k << bits) | (s < len ? (unsigned long long)chunk[b + s] + 1ull : 0ull);
    keys[a] = k;
    ids[a] = (uint32_t)r;
  }
}

__global__ void k_inverse(const uint32_t* __restrict__ ord, int64_t m, int32_t* __restrict__ pos) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
    pos[ord[i]] = (int32_t)i;
}

// lcp[x] = common prefix length of the strings at sorted positions x - 1 and x
// (lcp[0] = 0); trie weight = sum_x w(suffix of string x after lcp[x]).
__global__ void __launch_bounds__(kThreads)
k_lcp_cost(const uint32_t* __restrict__ ord, int64_t m, const int64_t* __restrict__ off,
           const int32_t* __restrict__ chunk, const int64_t* __restrict__ w, int32_t* __restrict__ lcp,
           unsigned long long* __restrict__ cost) {
  unsigned long long local = 0;
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < m; x += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t r = ord[x];
    const int64_t b = off[r], len = off[r + 1] - b;
    int64_t l = 0;
    if (x > 0) {
      const uint32_t p = ord[x - 1];
      const int64_t pb = off[p], plen = off[p + 1] - pb;
      const int64_t lim = len < plen ? len : plen;
      while (l < lim && chunk[b + l] == chunk[pb + l]) ++l;
    }
    lcp[x] = (int32_t)l;
    for (int64_t s = l; s < len; ++s) local += (unsigned long long)w[chunk[b + s]];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) local += __shfl_xor_sync(0xFFFFFFFFu, local, o);
  if ((threadIdx.x & 31) == 0 && local) atomicAdd(cost, local);
}

// ---------------------------------------------------------------------------
// Trie nodes and the per-access recency distance.
// ---------------------------------------------------------------------------
// st[k][i] = min lcp[i - 8^k + 1 .. i] (k = 1 .. K-1; level 0 is lcp itself)
__global__ void k_sparse_level(int32_t* __restrict__ st, int64_t m, int k) {
  const int64_t part = (int64_t)1 << (3 * (k - 1));
  const int32_t* prev = st + (int64_t)(k - 1) * m;
  int32_t* cur = st + (int64_t)k * m;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    int32_t v = prev[i];
#pragma unroll
    for (int q = 1; q < 8; ++q)
      if (i >= q * part) v = min(v, prev[i - q * part]);
    cur[i] = v;
  }
}

// the last sorted position y <= x with lcp[y] <= s (exists: lcp[0] = 0)
__device__ __forceinline__ int64_t node_owner(const int32_t* __restrict__ st, int64_t m, int K, int64_t x, int s) {
  if (st[x] <= s) return x;
  int64_t p = x;  // every lcp in [p, x] is > s
  for (int k = K - 1; k >= 0; --k) {
    const int64_t len = (int64_t)1 << (3 * k);
    while (p - len >= 0 && st[(int64_t)k * m + (p - 1)] > s) p -= len;  // at most seven times
  }
  return p - 1;
}

// new[x] = nodes first created by the string at sorted position x
__global__ void k_new_nodes(const uint32_t* __restrict__ ord, int64_t m, const int64_t* __restrict__ off,
                            const int32_t* __restrict__ lcp, uint32_t* __restrict__ fresh) {
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < m; x += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t r = ord[x];
    fresh[x] = (uint32_t)(off[r + 1] - off[r] - lcp[x]);
  }
}

// order[t] = t without a given one, and len[t] = length of the string served
// at t (len[m] = 0): scanned, the accesses' first positions.
__global__ void k_served(bool given, int64_t m, const int64_t* __restrict__ off, int32_t* __restrict__ order,
                         uint32_t* __restrict__ len) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t <= m; t += (int64_t)gridDim.x * blockDim.x) {
    if (t < m && !given) order[t] = (int32_t)t;
    const int64_t r = t < m && given ? order[t] : t;
    len[t] = t < m ? (uint32_t)(off[r + 1] - off[r]) : 0u;
  }
}

// Per access (served position t, depth s), laid out at aoff[t] + s: its trie
// node (with its own number, as a sort key), its chunk weight, its request's
// served position.
__global__ void __launch_bounds__(kThreads)
k_accesses(const int32_t* __restrict__ order, int64_t m, const int64_t* __restrict__ off,
           const int32_t* __restrict__ chunk, const int64_t* __restrict__ w, const int32_t* __restrict__ lexpos,
           const int32_t* __restrict__ st, int K, const uint32_t* __restrict__ node_base,
           const uint32_t* __restrict__ aoff, unsigned long long* __restrict__ node, uint32_t* __restrict__ acc_id,
           int64_t* __restrict__ aw, int64_t* __restrict__ asuf, int32_t* __restrict__ aowner) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < m; t += (int64_t)gridDim.x * blockDim.x) {
    const int32_t r = order[t];
    const int64_t b = off[r], len = off[r + 1] - b;
    const int64_t x = lexpos[r];
    const int64_t a0 = aoff[t];
    for (int64_t s = 0; s < len; ++s) {
      const int64_t y = node_owner(st, m, K, x, (int)s);
      node[a0 + s] = node_base[y] + (uint32_t)(s - st[y]);
      acc_id[a0 + s] = (uint32_t)(a0 + s);
      aw[a0 + s] = w[chunk[b + s]];
      aowner[a0 + s] = (int32_t)t;
    }
    int64_t suf = 0;
    for (int64_t s = len - 1; s >= 0; --s) {
      suf += aw[a0 + s];
      asuf[a0 + s] = suf;
    }
  }
}

// After a sort of the accesses by node, then number (served order), neighbours
// with the same node are consecutive touches of it.
__global__ void k_prev_next(const unsigned long long* __restrict__ skey, const uint32_t* __restrict__ sacc, int64_t N,
                            const int32_t* __restrict__ aowner, int32_t* __restrict__ prev_t,
                            int32_t* __restrict__ next_t) {
  for (int64_t z = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; z < N; z += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t a = sacc[z];
    const unsigned long long k = skey[z];
    prev_t[a] = (z > 0 && skey[z - 1] == k) ? aowner[sacc[z - 1]] : -1;
    next_t[a] = (z + 1 < N && skey[z + 1] == k) ? aowner[sacc[z + 1]] : INT_MAX;
  }
}

// the largest capacity below the trie weight (every distance is at most the
// trie weight, so larger capacities see only compulsory misses)
__global__ void k_scan_limit(const int64_t* __restrict__ caps, int n_caps, const unsigned long long* __restrict__ trie,
                             int64_t* __restrict__ limit) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    int64_t best = -1;
    const int64_t tw = (int64_t)*trie;
    for (int i = 0; i < n_caps; ++i)
      if (caps[i] < tw && caps[i] > best) best = caps[i];
    *limit = best;
  }
}

// weight of the nodes of served request r's path not touched again before t
__device__ __forceinline__ int64_t untouched_suffix(const uint32_t* __restrict__ aoff, const int32_t* __restrict__ next_t,
                                                    const int64_t* __restrict__ asuf, int64_t r, int64_t t) {
  const int64_t b = aoff[r];
  int64_t lo = 0, hi = (int64_t)aoff[r + 1] - b;  // next_t is nondecreasing along a path
  const int64_t len = hi;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if ((int64_t)next_t[b + mid] >= t)
      hi = mid;
    else
      lo = mid + 1;
  }
  return lo < len ? asuf[b + lo] : 0;
}

constexpr int kDistThreads = 256;

// One warp per served request t: the recency distance of each access on its
// path.  dist = INT64_MAX for a first touch (a miss at every capacity),
// limit + 1 when it exceeds the largest capacity of interest.
__global__ void __launch_bounds__(kDistThreads)
k_distance(int64_t m, const uint32_t* __restrict__ aoff, const int32_t* __restrict__ prev_t,
           const int32_t* __restrict__ next_t, const int64_t* __restrict__ aw, const int64_t* __restrict__ asuf,
           const int64_t* __restrict__ limit_p, int64_t* __restrict__ dist) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (kDistThreads / 32);
  const int64_t limit = *limit_p;
  for (int64_t t = (int64_t)blockIdx.x * (kDistThreads / 32) + (threadIdx.x >> 5); t < m; t += warps) {
    const int64_t b = aoff[t], len = (int64_t)aoff[t + 1] - b;
    int64_t scanned = t;  // requests [scanned, t) are summed
    int64_t sum = 0;
    bool over = limit < 0;
    int64_t run_j = -2, run_w = 0;
    for (int64_t q = 0; q < len; ++q) {
      const int64_t j = prev_t[b + q];
      int64_t d;
      if (j < 0) {
        d = LLONG_MAX;
      } else {
        const int64_t wq = aw[b + q];
        if (j == run_j) {
          run_w += wq;
        } else {
          run_j = j;
          run_w = wq;
        }
        while (!over && scanned > j + 1) {
          const int64_t lo = scanned - 32 > j + 1 ? scanned - 32 : j + 1;
          const int64_t r = scanned - 1 - lane;
          int64_t c = r >= lo ? untouched_suffix(aoff, next_t, asuf, r, t) : 0;
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xFFFFFFFFu, c, o);
          sum += c;
          scanned = lo;
          if (sum > limit) over = true;
        }
        d = over ? limit + 1 : sum + run_w;
        if (d > limit) d = limit + 1;
      }
      if (lane == 0) dist[b + q] = d;
    }
  }
}

constexpr int kMaxCaps = 1024;

// Weight of the accesses by how many of the sorted capacities they miss at:
// bins[j] = sum of w over accesses with caps[j - 1] < dist <= caps[j].  Each
// block keeps `copies` bins per value, a lane's own where they fit, so that
// lanes do not queue for one; an add per capacity and access on one counter each
// took 41 us at 23,368 accesses and 10 capacities, 165 us at 800,000.
constexpr int kBinWords = 4096;  // uint64 bins of a block

__global__ void __launch_bounds__(kThreads)
k_cache_costs(const int64_t* __restrict__ dist, const int64_t* __restrict__ aw, int64_t N,
              const int64_t* __restrict__ caps, int n_caps, int copies, unsigned long long* __restrict__ bins,
              unsigned long long* __restrict__ compulsory) {
  __shared__ unsigned long long acc[kBinWords];
  __shared__ int64_t cap_s[kMaxCaps];
  for (int i = threadIdx.x; i < n_caps; i += blockDim.x) cap_s[i] = caps[i];
  for (int i = threadIdx.x; i < (n_caps + 1) * copies; i += blockDim.x) acc[i] = 0;
  __syncthreads();
  const int copy = (int)threadIdx.x & (copies - 1);
  unsigned long long first = 0;
  for (int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; a < N; a += (int64_t)gridDim.x * blockDim.x) {
    const int64_t d = dist[a];
    const unsigned long long wa = (unsigned long long)aw[a];
    if (d == LLONG_MAX) first += wa;
    int lo = 0, hi = n_caps;  // capacities below d
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (cap_s[mid] < d) lo = mid + 1; else hi = mid;
    }
    atomicAdd(&acc[lo * copies + copy], wa);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) first += __shfl_xor_sync(0xFFFFFFFFu, first, o);
  if ((threadIdx.x & 31) == 0 && first) atomicAdd(compulsory, first);
  __syncthreads();
  for (int i = threadIdx.x; i <= n_caps; i += blockDim.x) {
    unsigned long long v = 0;
    for (int q = 0; q < copies; ++q) v += acc[i * copies + q];
    if (v) atomicAdd(&bins[i], v);
  }
}

// ---------------------------------------------------------------------------
// Host side.
// ---------------------------------------------------------------------------
constexpr int64_t kMaxStrings = (int64_t)1 << 22;
constexpr int64_t kMaxAccesses = (int64_t)1 << 27;
constexpr int64_t kMaxLength = 4096;

struct Arena {
  char* base = nullptr;
  size_t off = 0;
  template <typename T>
  T* take(int64_t count) {
    T* p = reinterpret_cast<T*>(base ? base + off : nullptr);
    off += ((size_t)(count > 0 ? count : 1) * sizeof(T) + 255) & ~(size_t)255;
    return p;
  }
};

struct Strings {
  int64_t m = 0, total = 0, maxlen = 0;
  std::unique_ptr<int32_t[]> chunk;  // not initialised first
};

mpt_status check_strings(int64_t n_chunks, int64_t m, const int64_t* offsets, const int64_t* chunks, Strings* out) {
  if (!offsets || n_chunks < 1 || n_chunks >= INT32_MAX || m < 1) return MPT_ERR_INVALID_ARG;
  if (m > kMaxStrings) return MPT_ERR_TOO_LARGE;
  if (offsets[0] != 0) return MPT_ERR_INVALID_ARG;
  int64_t maxlen = 0;
  for (int64_t i = 0; i < m; ++i) {
    const int64_t len = offsets[i + 1] - offsets[i];
    if (len < 0) return MPT_ERR_INVALID_ARG;
    if (len > maxlen) maxlen = len;
  }
  const int64_t total = offsets[m];
  if (total > 0 && !chunks) return MPT_ERR_INVALID_ARG;
  if (total > kMaxAccesses || maxlen > kMaxLength) return MPT_ERR_TOO_LARGE;
  out->m = m;
  out->total = total;
  out->maxlen = maxlen;
  try {
    out->chunk.reset(new int32_t[(size_t)(total > 0 ? total : 1)]);
  } catch (...) {
    return MPT_ERR_OUT_OF_MEMORY;
  }
  // one pass without branches: an id in range is below n_chunks as an unsigned number
  int32_t* to = out->chunk.get();
  uint64_t outside = 0;
  for (int64_t p = 0; p < total; ++p) {
    outside |= (uint64_t)chunks[p] >= (uint64_t)n_chunks;
    to[p] = (int32_t)chunks[p];
  }
  return outside ? MPT_ERR_INVALID_ARG : MPT_OK;
}

mpt_status check_weights(const int64_t* weights, int64_t n_chunks) {
  if (!weights) return MPT_ERR_INVALID_ARG;
  for (int64_t x = 0; x < n_chunks; ++x)
    if (weights[x] <= 0) return MPT_ERR_INVALID_ARG;
  return MPT_OK;
}

mpt_status check_permutation(const int32_t* p, int64_t m) {
  std::vector<char> seen;
  try {
    seen.assign((size_t)m, 0);
  } catch (...) {
    return MPT_ERR_OUT_OF_MEMORY;
  }
  for (int64_t i = 0; i < m; ++i) {
    if (p[i] < 0 || p[i] >= m || seen[(size_t)p[i]]) return MPT_ERR_INVALID_ARG;
    seen[(size_t)p[i]] = 1;
  }
  return MPT_OK;
}

// Device copies of the strings and the buffers of their lexicographic sort.
struct LexBuffers {
  int64_t* off;
  int32_t* chunk;
  int64_t* w;
  unsigned long long *keys, *keys2;
  uint32_t *ord, *ord2;
  int32_t* lexpos;
  int32_t* lcp;  // level 0 of the sparse table when the cache is simulated
  unsigned long long* trie;
};

void carve_lex(Arena& a, const Strings& s, int64_t n_chunks, int64_t sparse_levels, bool weights, LexBuffers* b) {
  const int64_t m = s.m;
  b->off = a.take<int64_t>(m + 1);
  b->chunk = a.take<int32_t>(s.total);
  b->w = weights ? a.take<int64_t>(n_chunks) : nullptr;
  b->keys = a.take<unsigned long long>(m);
  b->keys2 = a.take<unsigned long long>(m);
  b->ord = a.take<uint32_t>(m);
  b->ord2 = a.take<uint32_t>(m);
  b->lexpos = a.take<int32_t>(m);
  b->lcp = a.take<int32_t>(m * (sparse_levels > 0 ? sparse_levels : 1));
  b->trie = a.take<unsigned long long>(1);
}

// Sorts the strings (b->ord = string at each sorted position), first by window
// when there are any (window > 0; arrival on the device or null).  With
// `with_cost`, also the inverse b->lexpos, lcp and the trie weight.
cudaError_t run_lex(const Strings& s, LexBuffers* b, int64_t n_chunks, const int32_t* d_arrival, int64_t window,
                    bool with_cost, cudaStream_t st, int* launches) {
  const int64_t m = s.m;
  // chunk + 1 takes at most 31 bits and a window number 22, so at least one chunk is packed
  const int bits = bits_for((uint64_t)n_chunks), wbits = window > 0 ? bits_for((uint64_t)((m - 1) / window)) : 0;
  const int fit = (64 - wbits) / bits;
  const int packed = (int)(s.maxlen < fit ? s.maxlen : fit);
  k_lex_keys<<<grid_for(m), kThreads, 0, st>>>(m, b->off, b->chunk, d_arrival, window, packed, bits, b->keys, b->ord);
  ++*launches;
  cudaError_t e = packed == s.maxlen
                      ? merge_sort(&b->keys, &b->ord, &b->keys2, &b->ord2, m, ByKey{}, st, launches)
                      : merge_sort(&b->keys, &b->ord, &b->keys2, &b->ord2, m, ByString{b->off, b->chunk, packed}, st,
                                   launches);
  if (e != cudaSuccess || !with_cost) return e;
  k_inverse<<<grid_for(m), kThreads, 0, st>>>(b->ord, m, b->lexpos);
  ++*launches;
  if ((e = cudaMemsetAsync(b->trie, 0, sizeof(unsigned long long), st)) != cudaSuccess) return e;
  k_lcp_cost<<<grid_for(m), kThreads, 0, st>>>(b->ord, m, b->off, b->chunk, b->w, b->lcp, b->trie);
  ++*launches;
  return cudaGetLastError();
}

cudaError_t upload_strings(const Strings& s, const int64_t* offsets, const int64_t* weights, int64_t n_chunks,
                           LexBuffers* b, cudaStream_t st) {
  cudaError_t e = cudaMemcpyAsync(b->off, offsets, (size_t)(s.m + 1) * 8, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess && s.total > 0)
    e = cudaMemcpyAsync(b->chunk, s.chunk.get(), (size_t)s.total * 4, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess && b->w) e = cudaMemcpyAsync(b->w, weights, (size_t)n_chunks * 8, cudaMemcpyHostToDevice, st);
  return e;
}

mpt_status cuda_status(cudaError_t e) {
  if (e == cudaSuccess) return MPT_OK;
  return e == cudaErrorMemoryAllocation ? MPT_ERR_OUT_OF_MEMORY : MPT_ERR_CUDA;
}

int sparse_levels_for(int64_t m) {
  int K = 1;
  while (((int64_t)1 << (3 * K)) <= m) ++K;
  return K;  // 8^K > m
}

}  // namespace

// Eq. (1) for any number of strings (used by mpt_trie_cost beyond 32 strings).
mpt_status trie_cost_lex(const int64_t* weights, int64_t n_chunks, int64_t m, const int64_t* offsets,
                         const int64_t* chunks, cudaStream_t st, int64_t* cost) {
  Strings s;
  mpt_status ms = check_strings(n_chunks, m, offsets, chunks, &s);
  if (ms != MPT_OK) return ms;
  if ((ms = check_weights(weights, n_chunks)) != MPT_OK) return ms;
  Arena a;
  LexBuffers b{};
  carve_lex(a, s, n_chunks, 1, true, &b);
  char* mem = nullptr;
  cudaError_t e = device_alloc(reinterpret_cast<void**>(&mem), a.off);
  if (e != cudaSuccess) return cuda_status(e);
  Arena a2{mem, 0};
  carve_lex(a2, s, n_chunks, 1, true, &b);
  int launches = 0;
  unsigned long long h = 0;
  e = upload_strings(s, offsets, weights, n_chunks, &b, st);
  if (e == cudaSuccess) e = run_lex(s, &b, n_chunks, nullptr, 0, true, st, &launches);
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h, b.trie, 8, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFree(mem);
  if (e != cudaSuccess) return cuda_status(e);
  *cost = (int64_t)h;
  return MPT_OK;
}

}  // namespace mpt

extern "C" {

mpt_status mpt_serve_order(int64_t n_chunks, int32_t m, const int64_t* seq_offsets, const int64_t* seq_chunks,
                           const int32_t* arrival, int32_t window, void* stream, int32_t* order) {
  using namespace mpt;
  if (!order) return MPT_ERR_INVALID_ARG;
  Strings s;
  mpt_status ms = check_strings(n_chunks, m, seq_offsets, seq_chunks, &s);
  if (ms != MPT_OK) return ms;
  if (arrival && (ms = check_permutation(arrival, m)) != MPT_OK) return ms;
  if (window < 0) return MPT_ERR_INVALID_ARG;
  const bool windowed = window > 0 && window < m;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);

  Arena a;
  LexBuffers b{};
  carve_lex(a, s, n_chunks, 1, false, &b);
  // arrival positions matter only to windows
  int32_t* d_arrival = windowed && arrival ? a.take<int32_t>(m) : nullptr;
  char* mem = nullptr;
  cudaError_t e = device_alloc(reinterpret_cast<void**>(&mem), a.off);
  if (e != cudaSuccess) return cuda_status(e);
  Arena a2{mem, 0};
  carve_lex(a2, s, n_chunks, 1, false, &b);
  if (windowed && arrival) d_arrival = a2.take<int32_t>(m);

  int launches = 0;
  e = upload_strings(s, seq_offsets, nullptr, n_chunks, &b, st);
  if (e == cudaSuccess && d_arrival) e = cudaMemcpyAsync(d_arrival, arrival, (size_t)m * 4, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = run_lex(s, &b, n_chunks, d_arrival, windowed ? window : 0, false, st, &launches);
  if (e == cudaSuccess) e = cudaMemcpyAsync(order, b.ord, (size_t)m * 4, cudaMemcpyDeviceToHost, st);
  const cudaError_t es = cudaStreamSynchronize(st);
  if (e == cudaSuccess) e = es;
  cudaFree(mem);
  return cuda_status(e);
}

mpt_status mpt_cache_costs(const int64_t* weights, int64_t n_chunks, int32_t m, const int64_t* seq_offsets,
                           const int64_t* seq_chunks, const int32_t* order, const int64_t* capacities,
                           int32_t n_caps, void* stream, int64_t* costs, int64_t* unbounded) {
  using namespace mpt;
  if (n_caps < 0 || n_caps > kMaxCaps || (n_caps > 0 && (!capacities || !costs))) return MPT_ERR_INVALID_ARG;
  for (int32_t i = 0; i < n_caps; ++i)
    if (capacities[i] < 0) return MPT_ERR_INVALID_ARG;
  Strings s;
  mpt_status ms = check_strings(n_chunks, m, seq_offsets, seq_chunks, &s);
  if (ms != MPT_OK) return ms;
  if ((ms = check_weights(weights, n_chunks)) != MPT_OK) return ms;
  if (order && (ms = check_permutation(order, m)) != MPT_OK) return ms;
  int64_t heaviest = 0;
  for (int64_t x = 0; x < n_chunks; ++x) heaviest = weights[x] > heaviest ? weights[x] : heaviest;
  if (heaviest > ((int64_t)1 << 62) / (s.total > 0 ? s.total : 1)) {
    // distances and costs are sums of distinct node weights: bounded by the
    // total string weight
    int64_t total_w = 0;
    for (int64_t p = 0; p < s.total; ++p) {
      const int64_t wx = weights[s.chunk[(size_t)p]];
      if (total_w > ((int64_t)1 << 62) - wx) return MPT_ERR_OVERFLOW;
      total_w += wx;
    }
  }
  std::vector<unsigned long long> h_bins;
  std::vector<int32_t> by_cap;
  std::vector<int64_t> h_caps;
  try {
    h_bins.resize((size_t)n_caps + 1);
    by_cap.resize((size_t)n_caps);
    h_caps.resize((size_t)n_caps);
  } catch (...) {
    return MPT_ERR_OUT_OF_MEMORY;
  }
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int64_t N = s.total;
  const int K = sparse_levels_for(m);

  auto carve = [&](Arena& a, LexBuffers* b, int32_t** d_order, uint32_t** d_aoff, uint32_t** node_base,
                   unsigned long long** node, unsigned long long** node2, uint32_t** acc_id, uint32_t** acc2,
                   uint32_t** sums, int64_t** aw, int64_t** asuf,
                   int32_t** aowner, int32_t** prev_t, int32_t** next_t, int64_t** dist, int64_t** d_caps,
                   int64_t** limit, unsigned long long** d_bins, unsigned long long** compulsory) {
    carve_lex(a, s, n_chunks, K, true, b);
    *d_order = a.take<int32_t>(m);
    *d_aoff = a.take<uint32_t>(m + 1);
    *node_base = a.take<uint32_t>(m);
    *node = a.take<unsigned long long>(N);
    *node2 = a.take<unsigned long long>(N);
    *acc_id = a.take<uint32_t>(N);
    *acc2 = a.take<uint32_t>(N);
    *sums = a.take<uint32_t>(scan_tiles((int64_t)m + 1));
    *aw = a.take<int64_t>(N);
    *asuf = a.take<int64_t>(N);
    *aowner = a.take<int32_t>(N);
    *prev_t = a.take<int32_t>(N);
    *next_t = a.take<int32_t>(N);
    *dist = a.take<int64_t>(N);
    *d_caps = a.take<int64_t>(n_caps);
    *limit = a.take<int64_t>(1);
    *d_bins = a.take<unsigned long long>(n_caps + 1);
    *compulsory = a.take<unsigned long long>(1);
  };
  LexBuffers b{};
  int32_t* d_order;
  int64_t *aw, *asuf, *dist, *d_caps, *limit;
  uint32_t *d_aoff, *node_base, *acc_id, *acc2, *sums;
  int32_t *aowner, *prev_t, *next_t;
  unsigned long long *node, *node2, *d_bins, *compulsory;
  Arena a;
  carve(a, &b, &d_order, &d_aoff, &node_base, &node, &node2, &acc_id, &acc2, &sums, &aw, &asuf, &aowner, &prev_t,
        &next_t, &dist, &d_caps, &limit, &d_bins, &compulsory);
  char* mem = nullptr;
  cudaError_t e = device_alloc(reinterpret_cast<void**>(&mem), a.off);
  if (e != cudaSuccess) return cuda_status(e);
  Arena a2{mem, 0};
  carve(a2, &b, &d_order, &d_aoff, &node_base, &node, &node2, &acc_id, &acc2, &sums, &aw, &asuf, &aowner, &prev_t,
        &next_t, &dist, &d_caps, &limit, &d_bins, &compulsory);

  int launches = 0;
  unsigned long long h_trie = 0, h_first = 0;
  // the capacities in increasing order
  for (int32_t i = 0; i < n_caps; ++i) by_cap[(size_t)i] = i;
  std::sort(by_cap.begin(), by_cap.end(), [&](int32_t x, int32_t y) { return capacities[x] < capacities[y]; });
  for (int32_t i = 0; i < n_caps; ++i) h_caps[(size_t)i] = capacities[by_cap[(size_t)i]];
  int copies = 32;
  while (copies > 1 && copies * (n_caps + 1) > kBinWords) copies >>= 1;
  e = upload_strings(s, seq_offsets, weights, n_chunks, &b, st);
  if (e == cudaSuccess && order) e = cudaMemcpyAsync(d_order, order, (size_t)m * 4, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) {
    // served position -> first access: the lengths in served order, summed
    k_served<<<grid_for(m + 1), kThreads, 0, st>>>(order != nullptr, m, b.off, d_order, d_aoff);
    ++launches;
    e = exclusive_scan(d_aoff, m + 1, sums, st, &launches);
  }
  if (e == cudaSuccess && n_caps > 0)
    e = cudaMemcpyAsync(d_caps, h_caps.data(), (size_t)n_caps * 8, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(d_bins, 0, ((size_t)n_caps + 1) * 8, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(compulsory, 0, 8, st);
  if (e == cudaSuccess) e = run_lex(s, &b, n_chunks, nullptr, 0, true, st, &launches);
  if (e == cudaSuccess && N > 0) {
    for (int k = 1; k < K; ++k) k_sparse_level<<<grid_for(m), kThreads, 0, st>>>(b.lcp, m, k);
    k_new_nodes<<<grid_for(m), kThreads, 0, st>>>(b.ord, m, b.off, b.lcp, node_base);
    launches += K;
    e = exclusive_scan(node_base, m, sums, st, &launches);
    if (e == cudaSuccess) {
      k_accesses<<<grid_for(m), kThreads, 0, st>>>(d_order, m, b.off, b.chunk, b.w, b.lexpos, b.lcp, K, node_base,
                                                   d_aoff, node, acc_id, aw, asuf, aowner);
      ++launches;
      e = merge_sort(&node, &acc_id, &node2, &acc2, N, ByKey{}, st, &launches);
      if (e == cudaSuccess) {
        k_prev_next<<<grid_for(N), kThreads, 0, st>>>(node, acc_id, N, aowner, prev_t, next_t);
        k_scan_limit<<<1, 32, 0, st>>>(d_caps, n_caps, b.trie, limit);
        k_distance<<<grid_for(m * 32, 64), kDistThreads, 0, st>>>(m, d_aoff, prev_t, next_t, aw, asuf, limit,
                                                                         dist);
        k_cache_costs<<<grid_for(N, 4), kThreads, 0, st>>>(dist, aw, N, d_caps, n_caps, copies, d_bins, compulsory);
        launches += 4;
        e = cudaGetLastError();
      }
    }
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h_trie, b.trie, 8, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h_first, compulsory, 8, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(h_bins.data(), d_bins, ((size_t)n_caps + 1) * 8, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFree(mem);
  if (e != cudaSuccess) return cuda_status(e);
  // every trie node is first touched exactly once
  if (h_first != h_trie) return MPT_ERR_INTERNAL;
  unsigned long long missed = 0;  // by the accesses beyond the i-th capacity
  for (int32_t i = n_caps - 1; i >= 0; --i) {
    missed += h_bins[(size_t)i + 1];
    costs[by_cap[(size_t)i]] = (int64_t)missed;
  }
  if (unbounded) *unbounded = (int64_t)h_trie;
  return MPT_OK;
}

mpt_status mpt_layout_pinned(const int64_t* weights, int64_t n_chunks, int32_t m, const int64_t* ranked_offsets,
                             const int64_t* ranked_chunks, int32_t t, int32_t method, void* stream,
                             int64_t* perm_chunks, int32_t* serve_order, int64_t* cost) {
  using namespace mpt;
  if (!weights || !ranked_offsets || n_chunks < 1 || n_chunks >= INT32_MAX || m < 1 || t < 0) return MPT_ERR_INVALID_ARG;
  if (method != MPT_PIN_EXACT && method != MPT_PIN_GREEDY) return MPT_ERR_INVALID_ARG;
  if (method == MPT_PIN_EXACT && m > 32) return MPT_ERR_TOO_LARGE;
  if (ranked_offsets[0] != 0) return MPT_ERR_INVALID_ARG;
  const int64_t total = ranked_offsets[m];
  if (total > 0 && !ranked_chunks) return MPT_ERR_INVALID_ARG;
  for (int32_t i = 0; i < m; ++i)
    if (ranked_offsets[i + 1] < ranked_offsets[i]) return MPT_ERR_INVALID_ARG;
  for (int64_t p = 0; p < total; ++p)
    if (ranked_chunks[p] < 0 || ranked_chunks[p] >= n_chunks) return MPT_ERR_INVALID_ARG;
  // free part of request i: its ranked list after the first t entries
  std::vector<int64_t> foff, fchunks, seq, fperm, poff;
  std::vector<uint64_t> bits;
  const int64_t words = (n_chunks + 63) / 64;
  try {
    foff.assign((size_t)m + 1, 0);
    seq.resize((size_t)(total > 0 ? total : 1));
    for (int32_t i = 0; i < m; ++i) {
      const int64_t a = ranked_offsets[i], b = ranked_offsets[i + 1];
      const int64_t pin = b - a < t ? b - a : t;
      for (int64_t p = a + pin; p < b; ++p) fchunks.push_back(ranked_chunks[p]);
      foff[(size_t)i + 1] = (int64_t)fchunks.size();
    }
    fperm.resize(fchunks.size() > 0 ? fchunks.size() : 1);
    if (method == MPT_PIN_EXACT) {
      bits.assign((size_t)m * (size_t)words, 0);
      poff.resize((size_t)m + 1);
    }
  } catch (...) {
    return MPT_ERR_OUT_OF_MEMORY;
  }
  mpt_status ms;
  if (method == MPT_PIN_EXACT) {
    for (int32_t i = 0; i < m; ++i)
      for (int64_t p = foff[(size_t)i]; p < foff[(size_t)i + 1]; ++p) {
        const int64_t x = fchunks[(size_t)p];
        uint64_t& wd = bits[(size_t)i * (size_t)words + (size_t)(x >> 6)];
        if (wd >> (x & 63) & 1ull) return MPT_ERR_INVALID_ARG;  // repeated chunk
        wd |= 1ull << (x & 63);
      }
    mpt_ctx* ctx = nullptr;
    if ((ms = mpt_create(weights, n_chunks, bits.data(), m, &ctx)) != MPT_OK) return ms;
    int64_t opt = 0;
    ms = mpt_solve(ctx, nullptr, 0, stream, &opt);
    if (ms == MPT_OK) ms = mpt_layout(ctx, poff.data(), fperm.data(), nullptr);
    mpt_destroy(ctx);
    if (ms != MPT_OK) return ms;
    // mpt_layout's request ranges coincide with the free CSR (same sizes)
    for (int32_t i = 0; i <= m; ++i)
      if (poff[(size_t)i] != foff[(size_t)i]) return MPT_ERR_INTERNAL;
  } else {
    ms = mpt_greedy(weights, n_chunks, m, foff.data(), fchunks.empty() ? nullptr : fchunks.data(), stream, nullptr,
                    nullptr, nullptr, nullptr, nullptr, fperm.data(), nullptr);
    if (ms != MPT_OK) return ms;
  }
  // strings: free layout, then the pinned passages in relevance order
  for (int32_t i = 0; i < m; ++i) {
    const int64_t a = ranked_offsets[i], b = ranked_offsets[i + 1];
    const int64_t pin = b - a < t ? b - a : t;
    int64_t o = a;
    for (int64_t p = foff[(size_t)i]; p < foff[(size_t)i + 1]; ++p) seq[(size_t)o++] = fperm[(size_t)p];
    for (int64_t p = a; p < a + pin; ++p) seq[(size_t)o++] = ranked_chunks[p];
  }
  if (perm_chunks && total > 0) std::memcpy(perm_chunks, seq.data(), (size_t)total * 8);
  if (serve_order) {
    ms = mpt_serve_order(n_chunks, m, ranked_offsets, seq.data(), nullptr, 0, stream, serve_order);
    if (ms != MPT_OK) return ms;
  }
  if (cost) {
    ms = trie_cost_lex(weights, n_chunks, m, ranked_offsets, seq.data(), reinterpret_cast<cudaStream_t>(stream), cost);
    if (ms != MPT_OK) return ms;
  }
  return MPT_OK;
}

}  // extern "C"
