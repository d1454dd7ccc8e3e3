// K4: hierarchy walk -> layout, and the trie-cost check (Sec. 2, eq. 1).
//
// Layout (Thm 1 proof, "<=" direction): the hierarchy has root {0..m-1};
// node S with |S| >= 2 has children A = split[S] (left) and S \ A (right).
// At node B the chunks of I(B) \ I(parent(B)) are emitted, in increasing chunk
// id, with I(parent(root)) empty.  A chunk x is therefore emitted for request
// i at the highest node B on i's root-to-leaf path with B inside N_x (the
// request set of x), and request i's permutation is R_i sorted by
// (depth of that node, chunk id).  The left-to-right leaf order is the trie
// DFS order that Thm 7 (Sec. 8) serves requests in.  After a blocked solve
// split is read at the rotated position of each node and OPT = F(full) =
// F'(full) + sum_i pi_i + u from Gp = F' << b (uint32, or uint64 on the wide
// path) and the offsets pi, u (k_scatter_zeta.cu); after a general one both
// are in natural order.
//
// Trie cost: a string's node at depth p is new exactly when no earlier
// string shares its first p+1 symbols, so the trie weight is
//     sum_i sum over positions p >= max_{j<i} lcp(i, j) of w(seq_i[p]).
#include "mpt_internal.cuh"

namespace mpt {
namespace {

constexpr int kWalkThreads = 256;
constexpr int kMaxM = 32;

// One block, bound by its chains: the walk's splits, one dependent read per
// level of the hierarchy instead of one per node (m = 28: 45 -> 27 us).
// opt: OPT, then the eight counters as int32.
__global__ void __launch_bounds__(kWalkThreads)
k_walk(int m, const uint32_t* __restrict__ split, const int64_t* __restrict__ F, const int32_t* __restrict__ F32,
       const uint32_t* __restrict__ Gp, const unsigned long long* __restrict__ Gp64,
       const unsigned long long* __restrict__ priv, int L, int b, InnerPerm perm, const uint32_t* __restrict__ used_N,
       const int32_t* __restrict__ used_x, int32_t* __restrict__ counters, int64_t slots,
       unsigned long long* __restrict__ keys, int64_t* __restrict__ perm_offsets, int64_t* __restrict__ perm_chunks,
       int32_t* __restrict__ dfs, int64_t* __restrict__ opt) {
  __shared__ uint32_t anc[kMaxM][kMaxM];  // anc[i][d]: the depth-d node on request i's path
  __shared__ uint32_t nodes[2][kMaxM];    // a level's nodes, and where their leaves start in dfs order
  __shared__ int starts[2][kMaxM];
  __shared__ int leaf_depth[kMaxM];
  __shared__ int cnt[kMaxM];
  __shared__ int fill[kMaxM];
  __shared__ long long offs[kMaxM + 1];
  __shared__ int bad;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t full = (m >= 32) ? 0xFFFFFFFFu : ((1u << m) - 1u);
  if (tid < kMaxM) {
    cnt[tid] = 0;
    fill[tid] = 0;
    leaf_depth[tid] = 0;
  }
  if (tid == 0) bad = 0;
  __syncthreads();
  if (warp == 0) {
    // level by level, a lane per node: a level's nodes are disjoint, so there
    // are at most m of them, and those at a level are looked up together
    if (lane == 0) {
      nodes[0][0] = full;
      starts[0][0] = 0;
    }
    int live = 1;
    bool wrong = false;
    for (int d = 0; live > 0; ++d) {
      __syncwarp();
      const bool has = lane < live;
      const uint32_t S = has ? nodes[d & 1][lane] : 0u;
      const int at = has ? starts[d & 1][lane] : 0;
      const bool inner = (S & (S - 1)) != 0;
      for (uint32_t r = S; r; r &= r - 1) anc[__ffs(r) - 1][d] = S;
      if (has && !inner) {
        const int i = __ffs(S) - 1;
        leaf_depth[i] = d;
        dfs[at] = i;
      }
      // blocked path: split and F (as F << b in Gp) in rotated order
      uint32_t A = 0;
      if (inner) A = (Gp || Gp64) ? split[rot_index(S, L, b, perm)] : split[S];
      wrong = __any_sync(0xFFFFFFFFu, inner && (A == 0 || (A & ~S) != 0 || A == S));
      if (wrong) break;
      const uint32_t inners = __ballot_sync(0xFFFFFFFFu, inner);
      if (inner) {
        const int to = 2 * __popc(inners & ((1u << lane) - 1u));
        nodes[(d + 1) & 1][to] = A;
        starts[(d + 1) & 1][to] = at;
        nodes[(d + 1) & 1][to + 1] = S ^ A;  // right child, its leaves after the left subtree's
        starts[(d + 1) & 1][to + 1] = at + __popc(A);
      }
      live = 2 * __popc(inners);
    }
    if (wrong && lane == 0) {
      bad = 1;
      atomicOr(&counters[1], kErrBadSplit);
    }
  } else if (warp == 1) {
    int64_t pi_all = 0;
    if (priv) {
      pi_all = lane < m ? (int64_t)priv[lane] : 0;
      for (int off = 16; off > 0; off >>= 1) pi_all += __shfl_xor_sync(0xFFFFFFFFu, pi_all, off);
      pi_all += (int64_t)priv[kUniversalSlot];
    }
    if (lane == 0)
      *opt = Gp64 ? (int64_t)(Gp64[rot_index(full, L, b, perm)] >> b) + pi_all
             : Gp ? (int64_t)(Gp[rot_index(full, L, b, perm)] >> b) + pi_all
                  : (F ? F[full] : (int64_t)F32[full]);
  }
  int used = counters[0];
  if (used > slots) used = (int)slots;
  if (warp >= 2)
    for (int t = tid - 64; t < used; t += kWalkThreads - 64)
      for (uint32_t r = used_N[t]; r; r &= r - 1) atomicAdd(&cnt[__ffs(r) - 1], 1);
  __syncthreads();
  if (warp == 0) {
    const int own = lane < m ? cnt[lane] : 0;
    long long acc = own;
    for (int off = 1; off < 32; off <<= 1) {
      const long long o = __shfl_up_sync(0xFFFFFFFFu, acc, off);
      if (lane >= off) acc += o;
    }
    if (lane < m) {
      offs[lane] = acc - own;
      perm_offsets[lane] = acc - own;
    }
    if (lane == m - 1) {
      offs[m] = acc;
      perm_offsets[m] = acc;
      if (acc != slots) atomicOr(&counters[1], kErrLayoutCount);
    }
    __syncwarp();
    // the counters leave with the results, in one copy (they changed in this
    // kernel, so they are read past L1)
    if (lane < 8) reinterpret_cast<int32_t*>(opt)[2 + lane] = __ldcg(counters + lane);
  }
  __syncthreads();
  if (bad) return;

  for (int t = tid; t < used; t += kWalkThreads) {
    const uint32_t N = used_N[t];
    const unsigned long long x = (unsigned long long)(uint32_t)used_x[t];
    for (uint32_t r = N; r; r &= r - 1) {
      const int i = __ffs(r) - 1;
      int d = 0;
      while (d < leaf_depth[i] && (anc[i][d] & ~N) != 0) ++d;
      const int slot = atomicAdd(&fill[i], 1);
      if (offs[i] + slot < slots) keys[offs[i] + slot] = ((unsigned long long)d << 32) | x;
    }
  }
  __syncthreads();

  for (int i = warp; i < m; i += kWalkThreads / 32) {
    const long long base = offs[i];
    const int len = cnt[i];
    for (int j = lane; j < len; j += 32) {
      const unsigned long long kj = keys[base + j];
      int rank = 0;
      for (int t = 0; t < len; ++t) rank += keys[base + t] < kj;
      perm_chunks[base + rank] = (int64_t)(kj & 0xFFFFFFFFull);
    }
  }
}

__global__ void __launch_bounds__(kWalkThreads)
k_trie_cost(int m, const int64_t* __restrict__ w, const int64_t* __restrict__ offs, const int64_t* __restrict__ seq,
            int64_t* __restrict__ cost) {
  __shared__ int maxlcp[kMaxM];
  __shared__ unsigned long long total;
  const int tid = threadIdx.x;
  if (tid < kMaxM) maxlcp[tid] = 0;
  if (tid == 0) total = 0;
  __syncthreads();
  for (int p = tid; p < m * m; p += kWalkThreads) {
    const int i = p / m, j = p % m;
    if (j >= i) continue;
    const int64_t li = offs[i + 1] - offs[i], lj = offs[j + 1] - offs[j];
    const int64_t lim = li < lj ? li : lj;
    int64_t l = 0;
    while (l < lim && seq[offs[i] + l] == seq[offs[j] + l]) ++l;
    atomicMax(&maxlcp[i], (int)l);
  }
  __syncthreads();
  for (int i = tid; i < m; i += kWalkThreads) {
    unsigned long long s = 0;
    for (int64_t p = offs[i] + maxlcp[i]; p < offs[i + 1]; ++p) s += (unsigned long long)w[seq[p]];
    atomicAdd(&total, s);
  }
  __syncthreads();
  if (tid == 0) *cost = (int64_t)total;
}

}  // namespace

cudaError_t launch_walk(const Shape& s, const Workspace& ws, cudaStream_t stream, int* launches) {
  k_walk<<<1, kWalkThreads, 0, stream>>>(s.m, s.blocked ? ws.split_rot : ws.split, s.lean ? nullptr : ws.F,
                                         s.lean ? ws.fw : nullptr, s.blocked && !s.wide ? ws.Gp : nullptr,
                                         s.blocked && s.wide ? ws.Gp64 : nullptr, s.blocked ? ws.priv : nullptr,
                                         s.L, s.b, s.perm, ws.used_N,
                                         ws.used_x, ws.counters, s.slots, ws.keys,
                                         ws.perm_offsets, ws.perm_chunks, ws.dfs, ws.opt);
  ++*launches;
  return cudaGetLastError();
}

cudaError_t launch_trie_cost(int m, const int64_t* d_weights, const int64_t* d_offsets, const int64_t* d_chunks,
                             int64_t* d_cost, cudaStream_t stream) {
  k_trie_cost<<<1, kWalkThreads, 0, stream>>>(m, d_weights, d_offsets, d_chunks, d_cost);
  return cudaGetLastError();
}

}  // namespace mpt
