// K3 (pruned form): the Sec. 3.1 recurrence on the tiles of k_dp_blocked.cu,
// over the splits that can be reported instead of all of them.
//
// Which splits can be reported.  Let A | B be the reported split of S (the
// smallest optimal A among those holding S's lowest request) and |A| >= 2,
// with A1 | A2 the split of A, A1 holding that request.  A1 | (A2 + B) is a
// split of S too, A1 is a proper subset of A and so the smaller integer, and
//     F(A1) + F(A2 + B) <= F(A1) + F(A2) + F(B) - w(I(A2 + B))
//                        = F(A) + F(B) + w(I(A)) - w(I(A2 + B)).
// If w(I(A)) <= w(I(A2 + B)) it would be at least as good, against the choice
// of A.  So w(I(A)) > w(I(A2 + B)) >= w(I(S)): on the tables less the
// universal weight u (k_scatter_zeta.cu), where every w(I(.)) >= 0,
//     the reported A is a single request or has w(I(A)) > 0.
// Leaving every other A out changes no F(S) and no split(S).  Requests that
// share few chunks leave few such A ("members").
//
// Members are downward closed (A' within A keeps I(A)), so a member
// A = (Ta, Ua) has (Ta, {}) a member or a single request.  With the inner bits
// Ua = (a1, a2), a2 the low kRB bits, the members of one Ta are a list of
// rows (a1, mask of the a2's):
//   k_prune_tiles    w(I), and per Ta the row list and whether it is short (at
//                    most kPruneRows rows);
//   k_prune_members  per lowest request the Ta's with a short and those with
//                    a long list, each in increasing order;
//   k_dp_pruned      per tile T every short Ta within T, then, where T's own
//                    list is short too, the self pair and the tile's final
//                    entries.  Where T has no list, w(I(T, U)) = 0 for all U.
// Long lists go through the pair kernel of the full recurrence on just those
// Ta, and tiles with a long list through its row kernel (k_dp_blocked.cu).
//
// 64-bit keys have no pair kernel for long lists: their rows beyond the first
// kPruneRows are read from the table as they come.
//
// Measured on one GB300 (create, solve, layout and tables; full recurrence before,
// pruned after, by seed): 28 requests of 20 passages 673 -> 3.9 .. 17 ms (a passage
// held by 12 to 17 of the 28 decides it), 24 requests of 10 passages 11.1 -> 0.7 .. 0.8
// ms and with 64-bit keys 80 -> 0.7 .. 1.0 ms, 26 requests of 40 passages, lean tables,
// 81 -> 5 .. 58 ms.
// k_dp_pruned is bound by the integer ALU pipe where a popular passage gives
// long a1 lists: 83 % of the pipe busy over the heaviest layers of 26 requests of
// 40 passages, 57 to 75 % with 20 passages, the rest of the time lost to the
// barrier per pair (the warps of a group have 1, 2 or 4 rows of work each).  Also
// measured (tile stage at m = 28, seed 1, when the kernel took 13.1 ms): a block
// per tile, four to an SM, with the row groups dealt by a hash of the block 15.5
// ms, in turn per SM 16.2; three such blocks with three slots 16.8, with two slots
// 16.7, two blocks with four 21.9; the members evaluated one by one instead of by
// rows 242 ms; the inner bits in natural order 69.9 ms.
#include "mpt_internal.cuh"

#include <algorithm>

namespace mpt {
namespace {

constexpr int kPB = 12;  // inner bits of a tile
constexpr uint32_t kPMask = (1u << kPB) - 1u;
constexpr int kPQueue = 512;     // pairs queued between two rounds of evaluation
constexpr int kQueueShift = 20;  // queue entries: Ta below (L <= 20), rows above
static_assert(kPruneClasses <= 256, "classes are kept in bytes");
static_assert(256 < 1 << (32 - kQueueShift), "queue entries hold the row count");
constexpr int kRowBytes = 128;
constexpr int kMembersShift = 9;  // info: rows below, members above
constexpr uint32_t kRowsMask = (1u << kMembersShift) - 1u;
constexpr uint32_t kUnitSteps = 60;
// A pair of the full recurrence is 2,187 units of 243 steps, a thread each: 16,600
// steps of a warp.  Lists dearer than this go there.  26 requests of 40
// passages, seeds 9, 11, 12, 13 and 14: with 9,000 42.7, 17.5, 43.0, 55.6 and 43.7
// ms, with 12,000 31.0, 9.9, 29.1, 34.9, 43.7, with 14,000 26.0, 9.4, 24.2, 34.9,
// 43.6, with 17,000 25.7, 9.4, 24.2, 34.1, 50.0.  Over 60 instances of 21 to 28
// requests (pooled passages, random sets, few large sets, uniform requests) 10,000
// takes 3.5 % longer on the average and up to 1.9 times, 20,000 as long (0.91 to 1.05).
constexpr uint32_t kLongSteps = 14000;
constexpr double kFullPairSteps = 16600.0;
constexpr int kPruneMinPairs = 16;     // pairs that a further block of a tile has to have

// Shape of the kernel for 32-bit keys (rows of 32) and 64-bit keys (rows of
// 16): one thread per row.
template <typename Key, int kSlots_ = 2>
struct PrunedCfg {
  static constexpr int kRB = sizeof(Key) == 4 ? 5 : 4;
  static constexpr int kRow = 1 << kRB;
  static constexpr int kRows = 1 << (kPB - kRB);  // = threads per block
  static constexpr int kLogWarps = kPB - kRB - 5;
  // rows kept per Ta: those of a short list, or all (64-bit keys have no other kernel for a long one)
  static constexpr int kKept = sizeof(Key) == 4 ? kPruneRows : kRows;
  static constexpr int kSlots = kSlots_;  // windows of pairs: one in use, the others being copied
  static constexpr int kGroups = sizeof(Key) == 8 ? 1 : kSlots == 2 ? 4 : kSlots <= 4 ? 2 : 1;  // per block, at most
  static constexpr int kSlotBytes = (kRows + kPruneRows) * kRowBytes;  // Y window, X rows
  static constexpr int kTileBytes = kRows * (kRow + 1) * (int)sizeof(Key);  // a tile's keys, rows kRow + 1 apart
  static constexpr int kSeqStride = kRows + 2;  // so that a row's entries lie in different banks
  static constexpr int kSeqBytes = kRow * kSeqStride * 2;
  static constexpr int kSharedAt = kSlots * kSlotBytes + kSeqBytes + kPQueue * 4;
  static_assert(kSlotBytes >= kTileBytes, "a tile's keys fit a slot");
  static constexpr int kSharedBytes = 3072 + kSlots * 512;
  static constexpr int kGroupBytes = (kSharedAt + kSharedBytes + 127) / 128 * 128;
  static_assert(kGroupBytes * kGroups <= 227 * 1024, "one block fits an SM");
};

// What a group of k_dp_pruned shares beside its windows and queue.
template <typename Key, int kSlots_>
struct PrunedShared {
  // listed entries of the tile T: F << b, split, Ua, row of the list; by level, levels' sizes
  Key f[kPruneSelf];
  uint2 rows[2 * kSlots_][kPruneRows];  // lists of the pairs in use, staged and to be staged next: (a1, mask)
  uint32_t sp[kPruneSelf], start[kPB + 2], warp_n[PrunedCfg<Key>::kRows / 32];
  uint32_t last, any, unit;
  uint16_t u[kPruneSelf];
  uint8_t k[kPruneSelf], order[kPruneSelf];
};

// w(I(T, .)) and the row list of every T, one block per tile at a time, from
// the sets N_x of the chunks that some but not all requests share (N: stored
// rotated index, w: weight; K1's list): w(I(S)) = sum of w over N containing
// S.  Few tiles lie within any N_x; they are a superset sum over the 2^12
// inner sets in shared memory, and the others are left unwritten: their readers
// know from info that they are 0.  The general transform (K2) reads and writes
// the table once per 8 to 12 request bits after a clear.  m = 28: 0.29 + 2.0 ms
// of clear and transform (HBM-bound) -> 0.06 ms (0.29 with the zeros written).
// The row list: threads = rows, the mask of a row from its non-zero entries.
// info: 0 when T has no member, else rows | members << kMembersShift |
// kListLong (32-bit keys) when they are more than kPruneRows or, where the pair
// kernel runs (long_ok), cost more than a pair there | kTileLong when the tile
// is left to the row kernel (a long list, or more than kPruneRows rows or
// kPruneSelf members).  Cost: a row takes as many
// warps as have a lane whose row holds a1, each for its steps and the loads,
// here kUnitSteps steps' worth.
template <typename Key, typename G>
__global__ void __launch_bounds__(256)
k_prune_tiles(int L, bool long_ok, int n_shared, const uint32_t* __restrict__ N, const unsigned long long* __restrict__ w,
              G* __restrict__ wIr, uint32_t* __restrict__ info, uint2* __restrict__ rows,
              int32_t* __restrict__ counters) {
  using C = PrunedCfg<Key>;
  constexpr int kThreads = 256, kPer = 16 / (int)sizeof(G);
  __shared__ __align__(16) G s[1 << kPB];
  __shared__ uint32_t warp_n[8], warp_m[8], warp_c[8];
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  const int n = min(counters[3], n_shared);
  for (uint32_t T = blockIdx.x; T < (1u << L); T += gridDim.x) {
    const bool single = T != 0 && (T & (T - 1u)) == 0;
    bool clear = false;  // s holds the tile
    for (int base = 0; base < n; base += kThreads) {
      const int i = base + (int)tid;
      const uint32_t Ni = i < n ? N[i] : 0u;
      const bool hit = i < n && (T & ~(Ni >> kPB)) == 0;
      if (!__syncthreads_or(hit)) continue;
      if (!clear) {
        for (uint32_t v = tid; v <= kPMask; v += kThreads) s[v] = 0;
        clear = true;
        __syncthreads();
      }
      if (hit) atomicAdd(&s[Ni & kPMask], (G)w[i]);
    }
    G* out = wIr + ((size_t)T << kPB);
    if (!clear) {
      // no member: 0 to every reader, which goes by info, but in tile 0 and
      // beside a single request's listed entry
      if (T == 0 || single)
        for (uint32_t v = tid; v < (1u << kPB) / kPer; v += kThreads) reinterpret_cast<uint4*>(out)[v] = make_uint4(0, 0, 0, 0);
      if (tid == 0) {
        info[T] = single ? 1u | (1u << kMembersShift) : 0u;  // a single request is always listed
        if (single) rows[(size_t)T * C::kKept] = make_uint2(0u, 1u);
      }
      continue;
    }
#pragma unroll
    for (int j = 0; j < kPB; ++j) {
      __syncthreads();
#pragma unroll
      for (int q = 0; q < (1 << (kPB - 1)) / kThreads; ++q) {
        const uint32_t p = tid + (uint32_t)(q * kThreads);
        const uint32_t v = ((p >> j) << (j + 1)) | (p & ((1u << j) - 1u));
        s[v] += s[v | (1u << j)];
      }
    }
    __syncthreads();
    for (uint32_t v = tid; v < (1u << kPB) / kPer; v += kThreads)
      reinterpret_cast<uint4*>(out)[v] = reinterpret_cast<const uint4*>(s)[v];
    uint32_t mask = 0;
    if (T != 0 && tid < (uint32_t)C::kRows) {
      // entry i + row of the row at a time, so that a warp reads different banks
      for (uint32_t i = 0; i < (uint32_t)C::kRow; ++i) {
        const uint32_t a2 = (i + tid) & (C::kRow - 1);
        if (s[tid * C::kRow + a2] != 0) mask |= 1u << a2;
      }
      if (single && tid == 0) mask |= 1u;
    }
    uint32_t steps = 0;
    for (uint32_t r = mask; r; r &= r - 1) steps += (uint32_t)C::kRow >> __popc(__ffs(r) - 1);
    const uint32_t cost = mask ? (steps + kUnitSteps) << (C::kLogWarps - __popc(tid >> 5)) : 0u;
    const uint32_t bal = __ballot_sync(0xFFFFFFFFu, mask != 0);
    const uint32_t members = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)__popc(mask));
    const uint32_t costs = __reduce_add_sync(0xFFFFFFFFu, cost);
    if (lane == 0) {
      warp_n[warp] = (uint32_t)__popc(bal);
      warp_m[warp] = members;
      warp_c[warp] = costs;
    }
    __syncthreads();
    uint32_t at = (uint32_t)__popc(bal & ((1u << lane) - 1u)), nr = 0, nm = 0, nc = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      at += (uint32_t)q < warp ? warp_n[q] : 0u;
      nr += warp_n[q];
      nm += warp_m[q];
      nc += warp_c[q];
    }
    if (mask && at < (uint32_t)C::kKept) rows[(size_t)T * C::kKept + at] = make_uint2(tid, mask);
    if (tid == 0) {
      const bool many = nr > (uint32_t)kPruneRows;
      const bool is_long = sizeof(Key) == 4 && (many || (long_ok && nc > kLongSteps));
      if (is_long && !long_ok) atomicOr(counters + 1, kErrWorkspace);  // against the host's bound
      info[T] = nr == 0 ? 0u
                        : nr | (nm << kMembersShift) | (is_long ? kListLong : 0u) |
                              (is_long || many || nm > (uint32_t)kPruneSelf ? kTileLong : 0u);
    }
  }
}

// Ta's with lowest request l: 2^(L-1-l) of them, kept in this region of the
// two member arrays.
__host__ __device__ __forceinline__ uint32_t member_base(int L, int l) { return (1u << L) - (1u << (L - l)); }

// One block per lowest request: the Ta's with short and with long lists, each
// in increasing order (kPer consecutive candidates per thread and round).
__global__ void __launch_bounds__(1024)
k_prune_members(int L, const uint32_t* __restrict__ info, uint32_t* __restrict__ short_ta,
                uint32_t* __restrict__ long_ta, uint32_t* __restrict__ member_n) {
  constexpr int kPer = 8;
  __shared__ uint32_t ws[32], wl[32];
  const int l = blockIdx.x;
  const uint32_t total = 1u << (L - 1 - l);
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  uint32_t* so = short_ta + member_base(L, l);
  uint32_t* lo = long_ta + member_base(L, l);
  uint32_t ns = 0, nl = 0;
  for (uint32_t base = 0; base < total; base += 1024 * kPer) {
    uint32_t c[kPer];
    uint32_t ks = 0, kl = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const uint32_t h = base + threadIdx.x * kPer + (uint32_t)k;
      c[k] = h < total ? info[(h << (l + 1)) | (1u << l)] : 0u;
    }
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      ks += c[k] != 0 && !(c[k] & kListLong);
      kl += (c[k] & kListLong) != 0;
    }
    uint32_t is = ks, il = kl;
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t a = __shfl_up_sync(0xFFFFFFFFu, is, off), b = __shfl_up_sync(0xFFFFFFFFu, il, off);
      if (lane >= (uint32_t)off) {
        is += a;
        il += b;
      }
    }
    if (lane == 31) {
      ws[warp] = is;
      wl[warp] = il;
    }
    __syncthreads();
    uint32_t ts = 0, tl = 0, bs = 0, bl = 0;
    for (uint32_t q = 0; q < 32; ++q) {
      bs += q < warp ? ws[q] : 0u;
      bl += q < warp ? wl[q] : 0u;
      ts += ws[q];
      tl += wl[q];
    }
    uint32_t ps = ns + bs + is - ks, pl = nl + bl + il - kl;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const uint32_t Ta = ((base + threadIdx.x * kPer + (uint32_t)k) << (l + 1)) | (1u << l);
      if (c[k] & kListLong)
        lo[pl++] = Ta;
      else if (c[k] != 0)
        so[ps++] = Ta;
    }
    ns += ts;
    nl += tl;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    member_n[l] = ns;
    member_n[kMaxMembersL + l] = nl;
  }
}

// The tiles of a layer differ in work by two orders of magnitude (those within
// a popular passage's N_x have all their parts for members), and a heavy one
// taken last leaves the other SMs waiting: SMs were busy for 80 % of the heavy
// layers' time.  Tiles are dealt from the most work to the least, by classes of
// sqrt(2) of an estimate: over the N_x that hold T's lowest request, their
// common parts with T times the inner splits.  m = 28: solves
// of 3.05, 3.61, 8.47 and 14.41 ms by seed -> 2.85, 3.38, 8.34 and 14.11 ms, with
// two launches of 13 us each; so only where the host's estimate of the pairs is
// above kPruneSortPairs (some 0.5 ms).
__device__ __forceinline__ int work_class(uint32_t T, int n, const uint32_t* __restrict__ N) {
  float work = 1.0f;
  const uint32_t low = T & (~T + 1u);
  for (int i = 0; i < n; ++i) {
    const uint32_t Ni = N[i], NT = Ni >> kPB;
    if (NT & low) work += exp2f((float)(__popc(NT & T) - 1) + 0.585f * (float)__popc(Ni & kPMask));
  }
  const int c = (int)(2.0f * log2f(work));
  return kPruneClasses - 1 - min(c, kPruneClasses - 1);  // the most work first
}

__global__ void __launch_bounds__(256)
k_prune_classes(int L, int n_shared, const uint32_t* __restrict__ N, const int32_t* __restrict__ counters,
                uint32_t* __restrict__ hist, uint8_t* __restrict__ cls) {
  const int n = min(counters[3], n_shared);
  for (uint32_t T = 1 + blockIdx.x * blockDim.x + threadIdx.x; T < (1u << L); T += gridDim.x * blockDim.x) {
    const int c = work_class(T, n, N);
    cls[T] = (uint8_t)c;
    atomicAdd(&hist[__popc(T) * kPruneClasses + c], 1u);
  }
}

__global__ void __launch_bounds__(256)
k_prune_order(int L, const uint8_t* __restrict__ cls, const uint32_t* __restrict__ hist,
              uint32_t* __restrict__ placed, uint32_t* __restrict__ order) {
  for (uint32_t T = 1 + blockIdx.x * blockDim.x + threadIdx.x; T < (1u << L); T += gridDim.x * blockDim.x) {
    const int kh = __popc(T), c = cls[T];  // as counted: the order is a permutation whatever the estimate
    uint32_t at = 0;
    for (int k = 0; k < kh; ++k) at += (uint32_t)c_binom.v[L][k];
    for (int q = 0; q < c; ++q) at += hist[kh * kPruneClasses + q];
    at += atomicAdd(&placed[kh * kPruneClasses + c], 1u);
    order[at] = colex_rank(T);
  }
}

__device__ __forceinline__ uint32_t min_keep(uint32_t a, uint32_t b, bool* keep) { return __vibmin_u32(a, b, keep); }
__device__ __forceinline__ unsigned long long min_keep(unsigned long long a, unsigned long long b, bool* keep) {
  *keep = a <= b;
  return *keep ? a : b;
}
__device__ __forceinline__ void pcopy16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

// One 128-byte window row; `swz` (a multiple of 16) is XOR-ed into the offsets of
// its 16-byte chunks.  Window rows are kept with swz = (row mod 8) * 16, so
// that lanes reading the same chunk of consecutive rows hit different banks.
template <typename Key, int kRow>
__device__ __forceinline__ void pload_row(Key (&v)[kRow], const char* p, uint32_t swz) {
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const uint4 t = *reinterpret_cast<const uint4*>(p + (((uint32_t)c << 4) ^ swz));
    if constexpr (sizeof(Key) == 4) {
      v[4 * c] = t.x;
      v[4 * c + 1] = t.y;
      v[4 * c + 2] = t.z;
      v[4 * c + 3] = t.w;
    } else {
      v[2 * c] = ((Key)t.y << 32) | t.x;
      v[2 * c + 1] = ((Key)t.w << 32) | t.z;
    }
  }
}

// acc[s2] = min over the a2 of `mask` within s2 of x[a2] + y[s2 ^ a2]; with
// kAll the mask is full.  The mask is the same in every lane: each a2, and
// each 16 bytes of x, is one uniform branch around its steps.  x is read as it
// is needed, which keeps the kernel within 128 registers.
template <typename Key, int kRow, bool kAll>
__device__ __forceinline__ void pconv(Key (&acc)[kRow], const char* x, const Key (&y)[kRow], uint32_t mask) {
  constexpr int kPer = 16 / (int)sizeof(Key);
#pragma unroll
  for (int g = 0; g < kRow; g += kPer) {
    if (kAll || (mask >> g & ((1u << kPer) - 1u))) {
      const uint4 t = *reinterpret_cast<const uint4*>(x + g * (int)sizeof(Key));
      Key v[kPer];
      if constexpr (sizeof(Key) == 4) {
        v[0] = t.x;
        v[1] = t.y;
        v[2] = t.z;
        v[3] = t.w;
      } else {
        v[0] = ((Key)t.y << 32) | t.x;
        v[1] = ((Key)t.w << 32) | t.z;
      }
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        const int a2 = g + q;
        if (kAll || (mask >> a2 & 1u)) {
#pragma unroll
          for (int s2 = 0; s2 < kRow; ++s2) {
            if ((a2 & s2) == a2) {
              const Key k = v[q] + y[s2 ^ a2];
              acc[s2] = k < acc[s2] ? k : acc[s2];
            }
          }
        }
      }
    }
  }
}

// One tile T with |T| = kh >= 1 per group of threads, or `items` groups per tile
// that each take every items-th pair; a block of up to kGroups groups stays on
// an SM and its groups take the next unit of the layer as they finish (*next).
// Thread = row s1 of the tile, with its
// kRow outputs' best keys in registers and, in shared memory, the numbers of
// their pairs in the queue (written only on a strict improvement, the pairs
// coming in increasing Ta).  Per pair the complement window Y and the listed
// rows of X are copied to shared memory, kSlots - 1 pairs ahead of the steps
// and the lists as far ahead of those (read into registers one pair ahead
// instead: 1 % slower where all four groups run);
// one barrier per pair.  Every lane of a warp runs the same (a1, mask) at a
// time, with those lanes idle whose row does not hold a1, so that X is read
// by broadcast.
// The inner bits are stored in an order (perm) that puts those of the request
// sets that cost most first into a2, where a listed row is then one register
// convolution without idle lanes, and next into the bits that tell the warps
// apart.  Rows with more of a list's a1 bits take longer (1, 2, 2 and 4 rows of
// work for the four warps of a group, say), so the groups deal their warps the
// row groups in rotated orders and each sub-partition has one of each kind.
// Groups of one tile, rounds of one group beyond the queue and, with
// long_lists, the pair kernel's minima meet in `partial` ((key << 32 | Ta); for
// 64-bit keys, one block per tile and no pair kernel, the key, and Ta in
// partial_ta).  The group that finishes last (done[]) goes on to the tile's
// entries.
template <typename Key, typename Tab, int kSlots_>
__global__ void __launch_bounds__(PrunedCfg<Key, kSlots_>::kRows * PrunedCfg<Key, kSlots_>::kGroups,
                                  sizeof(Key) == 8 && kSlots_ == 2 ? 2 : 1)
k_dp_pruned(int L, int kh, uint32_t items, bool long_tiles, bool long_lists, InnerPerm perm,
            const uint32_t* __restrict__ order, const Tab* __restrict__ wIr,
            const uint32_t* __restrict__ info, const uint2* __restrict__ rows, const uint32_t* __restrict__ short_ta,
            const uint32_t* __restrict__ long_ta, const uint32_t* __restrict__ member_n, unsigned long long* partial, uint32_t* partial_ta,
            uint32_t* __restrict__ done, uint32_t* __restrict__ next, Key* Gp,
            Key* Gc, uint32_t* __restrict__ split_rot, int32_t* __restrict__ flags) {
  using C = PrunedCfg<Key, kSlots_>;
  constexpr int kRB = C::kRB, kRow = C::kRow, NT = C::kRows, kWarps = NT / 32;
  constexpr uint32_t kFull = 0xFFFFFFFFu >> (32 - kRow);
  constexpr Key kNone = ~(Key)0;
  constexpr uint32_t kSelf = 0xFFFFu, kListed = 0x8000u;  // pair numbers of the self pair and of listed entries
  constexpr int kMeet = 8;
  static_assert(kPQueue <= 0x8000, "pair numbers fit beside the two marks");
  extern __shared__ __align__(16) char block_sm[];
  const uint32_t group = threadIdx.x / NT, tid = threadIdx.x % NT, lane = tid & 31u, warp = tid >> 5;
  char* psm = block_sm + group * C::kGroupBytes;
  Key* skey = reinterpret_cast<Key*>(psm + C::kSlotBytes);  // after the pairs: keys, rows kRow + 1 apart
  uint16_t* seq = reinterpret_cast<uint16_t*>(psm + C::kSlots * C::kSlotBytes);  // [in-row entry][thread]
  uint32_t* queue = reinterpret_cast<uint32_t*>(psm + C::kSlots * C::kSlotBytes + C::kSeqBytes);
  auto& sh = *reinterpret_cast<PrunedShared<Key, kSlots_>*>(psm + C::kSharedAt);
  auto sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1u + group), "n"(NT) : "memory"); };  // of this group
  // The warps of one sub-partition (number mod 4) get row groups of every kind:
  // those of the groups rotated, or of a group of eight warps mirrored.
  auto rows_of = [&](uint32_t w) { return kWarps == 4 ? (w + group) & 3u : (w < 4 ? w : 11u - w); };
  auto warp_of = [&](uint32_t rg) { return kWarps == 4 ? (rg - group) & 3u : (rg < 4 ? rg : 11u - rg); };
  const uint32_t s1 = lane | (rows_of(warp) << 5);
  auto key_at = [&](uint32_t U) -> Key& { return skey[U + (U >> kRB)]; };
  auto seq_at = [&](uint32_t U) -> uint16_t& {  // in the column of the thread that has the row
    const uint32_t r = U >> kRB;
    return seq[(U & (kRow - 1)) * C::kSeqStride + ((r & 31u) | (warp_of(r >> 5) << 5))];
  };
  const uint32_t tiles = (uint32_t)c_binom.v[L][kh];

  // The layer before may still run (launch_layer): what it and earlier ones
  // wrote is read only behind earlier().
  bool waited = false;
  auto earlier = [&]() {
    if (!waited) asm volatile("griddepcontrol.wait;" ::: "memory");
    waited = true;
  };
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // One unit: a tile, or one of `items` parts of it.  Every thread of the
  // group takes the same way out.
  auto run = [&](uint32_t unit) {
  // sorted: the parts of one tile one after the other, the heavy tiles' first
  // (all tiles' first parts, then all second ones: 2 to 8 % longer solves)
  const uint32_t item = order ? unit % items : unit / tiles, tile = order ? order[unit / items] : unit % tiles;
  if (MPT_BAD(flags, tile < tiles)) return;
  const uint32_t T = colex_unrank((unsigned long long)tile, kh, L);
  if (MPT_BAD(flags, T < (1u << L) && __popc(T) == kh)) return;
  const uint32_t iT = info[T];
  const bool long_tile = (iT & kTileLong) != 0;
  if (long_tile && kh == 1) {  // no pairs: the row kernel does it all
    if (!long_tiles && tid == 0) atomicOr(flags, kErrWorkspace);
    return;
  }
  const uint32_t cT = (iT >> kMembersShift) & 0x1FFFu;
  const int l = __ffs(T) - 1;
  const uint32_t low = 1u << l, rest = T ^ low;
  Key bk[kRow];
#pragma unroll
  for (int i = 0; i < kRow; ++i) {
    bk[i] = kNone;
    seq[i * C::kSeqStride + tid] = 0;
  }

  auto stage_window = [&](char* slot, const Key* win) {
    const char* y = reinterpret_cast<const char*>(win);
    const uint32_t c0 = tid >> 3, col = (tid & 7u) * 16u, swz = col ^ ((c0 & 7u) * 16u);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t r = c0 + (uint32_t)(j * (NT / 8));
      pcopy16(slot + r * kRowBytes + swz, y + r * kRowBytes + col);
    }
  };
  // The row list of queued pair p, copied kSlots - 1 pairs ahead of its windows.
  constexpr int kRing = 2 * C::kSlots;
  auto stage_list = [&](uint32_t p) {
    const uint32_t Tp = queue[p] & ((1u << kQueueShift) - 1u), n = min(queue[p] >> kQueueShift, (uint32_t)kPruneRows);
    if (2 * tid < n) pcopy16(&sh.rows[p % kRing][2 * tid], rows + (size_t)Tp * C::kKept + 2 * tid);
  };
  auto stage = [&](uint32_t p, uint32_t s) {
    const uint32_t Tp = queue[p] & ((1u << kQueueShift) - 1u), n = min(queue[p] >> kQueueShift, (uint32_t)kPruneRows);
    char* slot = psm + s * C::kSlotBytes;
    const uint32_t col = (tid & 7u) * 16u;
    const char* x = reinterpret_cast<const char*>(Gp + ((size_t)Tp << kPB));
    stage_window(slot, Gc + ((size_t)(T ^ Tp) << kPB));
    for (uint32_t r = tid >> 3; r < n; r += NT / 8)
      pcopy16(slot + (NT + r) * kRowBytes + col, x + sh.rows[p % kRing][r].x * kRowBytes + col);
  };
  // Candidates: the short lists of lowest request l, or the proper parts of T
  // holding it when those are fewer; both in increasing order.  A queue entry,
  // or 0.
  const uint32_t nm = member_n[l], np = (1u << (kh - 1)) - 1u;
  const bool by_parts = np < nm;
  const uint32_t total = by_parts ? np : nm;
  const uint32_t* mem = short_ta + member_base(L, l);
  auto candidate = [&](uint32_t i) -> uint32_t {
    if (i >= total) return 0u;
    const uint32_t Ta = by_parts ? (low | deposit_bits(i, rest)) : mem[i];
    if ((Ta & ~T) != 0 || Ta == T) return 0u;
    const uint32_t c = info[Ta];
    return c == 0 || (c & kListLong) ? 0u : Ta | ((c & kRowsMask) << kQueueShift);
  };
  // Blocks of this tile that take part: as many as there are kPruneMinPairs
  // pairs for (the same number in each of them).
  constexpr int kScan = kPQueue / NT;  // runs of 32 candidates that a warp looks at together: one round's finds fit
  uint32_t parts = 1;
  if (items > 1) {
    uint32_t n = 0;
    for (uint32_t base = tid; base < total; base += kScan * NT) {
#pragma unroll
      for (int k = 0; k < kScan; ++k) n += candidate(base + (uint32_t)(k * NT)) != 0;
    }
    n = __reduce_add_sync(0xFFFFFFFFu, n);
    if (lane == 0) sh.warp_n[warp] = n;
    sync();
    n = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) n += sh.warp_n[w];
    parts = min(items, max(1u, n / (uint32_t)kPruneMinPairs));
    if (item >= parts) return;
    sync();
  }

  // Keys and Ta's of the round to shared memory; from here thread tid has the
  // outputs tid, tid + NT, ..
  auto dump = [&]() {
    sync();
#pragma unroll
    for (int i = 0; i < kRow; ++i) skey[s1 * (kRow + 1) + i] = bk[i];
    sync();
  };
  unsigned long long* pt = partial + ((size_t)tile << kPB);
  uint32_t* pt_ta = partial_ta + ((size_t)tile << kPB);  // 64-bit keys
  // the Ta of an output's best pair, before the self pair: from the queue, or
  // where the minima have met
  bool met = parts > 1;  // minima in `partial`
  auto ta_at = [&](uint32_t U) -> uint32_t {
    if (!met) return queue[seq_at(U)] & ((1u << kQueueShift) - 1u);
    return sizeof(Key) == 4 ? (uint32_t)__ldcg(&pt[U]) : pt_ta[U];
  };
  auto to_partial = [&]() {
    // kMeet reads in flight at a time, here, where the minima are read back and
    // in the last pass over the tile: one at a time, each of a thread's 32 waited
    // for L2 (m = 28 by seed: 2.59, 3.34, 8.08 and 13.68 -> 2.34, 3.08, 7.49 and
    // 12.91 ms per solve)
    for (uint32_t U0 = tid; U0 <= kPMask; U0 += kMeet * NT) {
      unsigned long long there[kMeet];
#pragma unroll
      for (int q = 0; q < kMeet; ++q) there[q] = __ldcg(&pt[U0 + (uint32_t)(q * NT)]);
#pragma unroll
      for (int q = 0; q < kMeet; ++q) {
        const uint32_t U = U0 + (uint32_t)(q * NT);
        const unsigned long long own =
            ((unsigned long long)key_at(U) << 32) | (queue[seq_at(U)] & ((1u << kQueueShift) - 1u));
        if (own < there[q]) atomicMin(&pt[U], own);
      }
    }
  };

  // The pairs, a queue of them at a time.
  uint32_t found = 0, base = 0;
  if (sizeof(Key) == 4 && long_lists && kh >= 2) {
    // has T a part with a long list?
    const uint32_t nl = member_n[kMaxMembersL + l];
    bool any = false;
    if (np < nl) {
      for (uint32_t i = tid; i < np; i += NT) any = any || (info[low | deposit_bits(i, rest)] & kListLong) != 0;
    } else {
      for (uint32_t i = tid; i < nl; i += NT) {
        const uint32_t Ta = long_ta[member_base(L, l) + i];
        any = any || ((Ta & ~T) == 0 && Ta != T);
      }
    }
    if (tid == 0) sh.any = 0;
    sync();
    if (any) sh.any = 1;
    sync();
    met = met || sh.any != 0;
  }
  if (sizeof(Key) == 4 && kh >= 2) met = met || long_tile;
  // phase 0: the pairs; phase 1: the self pair, Ta = T over the tile's own
  // members, B = (0, U \ Ua) in tile 0
  for (int phase = kh >= 2 ? 0 : 1; phase < 2;) {
    uint32_t qn = 1;
    if (phase == 0) {
      for (qn = 0; base < total; base += kScan * NT) {
        uint32_t Ta[kScan], bal[kScan], mine = 0;
#pragma unroll
        for (int k = 0; k < kScan; ++k) Ta[k] = candidate(base + (warp * kScan + (uint32_t)k) * 32u + lane);
#pragma unroll
        for (int k = 0; k < kScan; ++k) {
          bal[k] = __ballot_sync(0xFFFFFFFFu, Ta[k] != 0);
          mine += (uint32_t)__popc(bal[k]);
        }
        sync();
        if (lane == 0) sh.warp_n[warp] = mine;
        sync();
        uint32_t at = found, sum = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
          at += (uint32_t)w < warp ? sh.warp_n[w] : 0u;
          sum += sh.warp_n[w];
        }
        // this block's pairs are the found ones numbered item, item + parts, ..
        const uint32_t q0 = (found + parts - 1 - item) / parts, q1 = (found + sum + parts - 1 - item) / parts;
        if (qn + q1 - q0 > (uint32_t)kPQueue) break;  // next round
#pragma unroll
        for (int k = 0; k < kScan; ++k) {
          const uint32_t o = at + __popc(bal[k] & ((1u << lane) - 1u));
          if (Ta[k] != 0 && o % parts == item) queue[qn + o / parts - q0] = Ta[k];
          at += (uint32_t)__popc(bal[k]);
        }
        found += sum;
        qn += q1 - q0;
      }
      sync();
      // the first lists, then the first kSlots - 1 pairs; a group is committed
      // for each slot, also without a pair, so that the waits below can count them
#pragma unroll
      for (uint32_t p = 0; p < (uint32_t)kRing - 2; ++p)
        if (p < qn) stage_list(p);
      asm volatile("cp.async.commit_group;" ::: "memory");
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      sync();
      earlier();
#pragma unroll
      for (int p = 0; p < C::kSlots - 1; ++p) {
        if ((uint32_t)p < qn) stage(p, p);
        asm volatile("cp.async.commit_group;" ::: "memory");
      }
    } else {
      earlier();
      if (cT == 0) break;
      // The listed entries themselves first, one thread each, level by level
      // in |Ua| (a member Ua' within Ua has a lower level): a level's entries
      // are finished, then offered to the later ones.  Then X = their rows.
      stage_window(psm, Gc);
      asm volatile("cp.async.commit_group;" ::: "memory");
      const uint32_t n = iT & kRowsMask;  // at most kPruneRows
      if (tid <= (uint32_t)kPB + 1) sh.start[tid] = 0;
      if (warp == 0) {
        static_assert(kPruneRows <= 32, "one list row per lane");
        const uint2 own = lane < n ? rows[(size_t)T * C::kKept + lane] : make_uint2(0u, 0u);
        uint32_t at = 0;
        for (uint32_t k = 0; k < n; ++k) {
          const uint2 e = make_uint2(__shfl_sync(0xFFFFFFFFu, own.x, k), __shfl_sync(0xFFFFFFFFu, own.y, k));
          if (e.y >> lane & 1u) {
            const uint32_t i = at + __popc(e.y & ((1u << lane) - 1u));
            sh.u[i] = (uint16_t)((e.x << kRB) | lane);
            sh.k[i] = (uint8_t)k;
          }
          if (lane == 0) sh.rows[0][k] = e;
          at += __popc(e.y);
        }
      }
      sync();
      static_assert(kPruneSelf <= NT, "one thread per listed entry");
      const bool mine = tid < cT;
      const uint32_t u = mine ? sh.u[tid] : 0u;
      const uint32_t level = mine ? (uint32_t)__popc(u) : 32u;
      const Key w = mine ? (Key)wIr[((size_t)T << kPB) | u] : (Key)0;
      uint32_t rank = 0;
      for (uint32_t j = 0; j < cT; ++j) {
        const uint32_t lj = (uint32_t)__popc(sh.u[j]);
        rank += lj < level || (lj == level && j < tid);
      }
      if (mine) {
        sh.order[rank] = (uint8_t)tid;
        atomicAdd(&sh.start[level + 1], 1u);
      }
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      Key best = mine && kh >= 2 ? key_at(u) : kNone;
      uint32_t ta = mine && kh >= 2 ? ta_at(u) : 0u;
      for (uint32_t lv = 0, k = 0; k < cT; ++lv) {
        if (level == lv) {
          Key f = w;
          uint32_t A = 0;
          if (!(kh == 1 && u == 0)) {
            f = (best >> kPB) - w;
            A = (((uint32_t)(best & kPMask) + perm.nat(u) - kPMask) << L) | ta;
          }
          sh.f[tid] = f << kPB;
          sh.sp[tid] = A;
          *reinterpret_cast<Key*>(psm + (NT + sh.k[tid]) * kRowBytes + (u & (kRow - 1)) * sizeof(Key)) = f << kPB;
        }
        sync();
        for (const uint32_t end = k + sh.start[lv + 1]; k < end; ++k) {
          const uint32_t j = sh.order[k], uj = sh.u[j], v = u ^ uj;
          if (mine && level > lv && (uj & ~u) == 0) {
            const uint32_t r = v >> kRB, off = (v & (kRow - 1)) * (uint32_t)sizeof(Key);
            const Key c = sh.f[j] + *reinterpret_cast<const Key*>(psm + r * kRowBytes + (off ^ ((r & 7u) * 16u)));
            if (c < best) {  // equal: the smaller Ta stays
              best = c;
              ta = T;
            }
          }
        }
      }
    }
    for (uint32_t p = 0, s = 0; p < qn; ++p, s = s + 1 == (uint32_t)C::kSlots ? 0 : s + 1) {
      // pair p's copies have landed; behind the barrier every thread is done
      // with pair p - 1, whose slot takes the next pair to be copied
      asm volatile("cp.async.wait_group %0;" ::"n"(C::kSlots - 2) : "memory");
      sync();
      if (phase == 0) {
        const uint32_t q = p + (uint32_t)(C::kSlots - 1);
        if (q < qn) stage(q, s == 0 ? C::kSlots - 1 : s - 1);
        if (q + C::kSlots - 1 < qn) stage_list(q + C::kSlots - 1);
        asm volatile("cp.async.commit_group;" ::: "memory");
      }
      const char* slot = psm + s * C::kSlotBytes;
      const uint2* list = sh.rows[p % kRing];
      const uint32_t n = phase == 0 ? queue[p] >> kQueueShift : iT & kRowsMask;
      Key acc[kRow];
#pragma unroll
      for (int i = 0; i < kRow; ++i) acc[i] = kNone;
      for (uint32_t k = 0; k < min(n, (uint32_t)kPruneRows); ++k) {
        const uint32_t a1 = list[k].x, mask = list[k].y;
        if ((a1 & ~s1) != 0) continue;
        Key y[kRow];
        const uint32_t r = s1 ^ a1;
        const char* x = slot + (NT + k) * kRowBytes;
        pload_row<Key, kRow>(y, slot + r * kRowBytes, (r & 7u) * 16u);
        if (mask == kFull)
          pconv<Key, kRow, true>(acc, x, y, mask);
        else
          pconv<Key, kRow, false>(acc, x, y, mask);
      }
      if constexpr (C::kKept > kPruneRows) {
        // the rest of a long list, its rows of X straight from the table
        const uint32_t Tp = queue[p] & ((1u << kQueueShift) - 1u);
        for (uint32_t k = kPruneRows; k < n; ++k) {
          const uint2 e = rows[(size_t)Tp * C::kKept + k];
          if ((e.x & ~s1) != 0) continue;
          Key y[kRow];
          const uint32_t r = s1 ^ e.x;
          pload_row<Key, kRow>(y, slot + r * kRowBytes, (r & 7u) * 16u);
          pconv<Key, kRow, false>(acc, reinterpret_cast<const char*>(Gp + (((size_t)Tp << kPB) | (e.x << kRB))), y, e.y);
        }
      }
      __syncwarp();
      const uint16_t number = (uint16_t)(phase == 0 ? p : kSelf);
#pragma unroll
      for (int i = 0; i < kRow; ++i) {
        bool keep;  // true when the running best is <= this pair's minimum
        bk[i] = min_keep(bk[i], acc[i], &keep);
        if (!keep) seq[i * C::kSeqStride + tid] = number;
      }
    }
    dump();
    if (phase == 1) break;
    if constexpr (sizeof(Key) == 4) {
      if (met || base < total) {
        to_partial();
        if (base < total) {  // a further round
          met = true;
          sync();
#pragma unroll
          for (int i = 0; i < kRow; ++i) {
            bk[i] = kNone;
            seq[i * C::kSeqStride + tid] = 0;
          }
          continue;
        }
        if (long_tile) return;  // the row kernel goes on from there
        __threadfence();
        sync();
        if (parts > 1) {
          if (tid == 0) {
            const uint32_t before = atomicAdd(&done[tile], 1u);
            sh.last = before == parts - 1;
            if (sh.last) done[tile] = 0;  // for the next layer
          }
          sync();
          if (!sh.last) return;
          __threadfence();
        }
        for (uint32_t U0 = tid; U0 <= kPMask; U0 += kMeet * NT) {
          unsigned long long there[kMeet];
#pragma unroll
          for (int q = 0; q < kMeet; ++q) there[q] = __ldcg(&pt[U0 + (uint32_t)(q * NT)]);
#pragma unroll
          for (int q = 0; q < kMeet; ++q) key_at(U0 + (uint32_t)(q * NT)) = (Key)(there[q] >> 32);
        }
        sync();
#pragma unroll
        for (int i = 0; i < kRow; ++i) bk[i] = skey[s1 * (kRow + 1) + i];
      }
    }
    if constexpr (sizeof(Key) == 8) {
      // one block per tile, its rounds one after the other: plain merges; a
      // tile left to the row kernel has its minima in its slot there
      if (met || base < total || long_tile) {
        for (uint32_t U = tid; U <= kPMask; U += NT) {
          const Key k = key_at(U);
          const uint32_t ta = queue[seq_at(U)] & ((1u << kQueueShift) - 1u);
          if (!met || k < pt[U] || (k == pt[U] && ta < pt_ta[U])) {
            pt[U] = k;
            pt_ta[U] = ta;
          }
        }
        met = true;
        sync();
        if (base < total) {
#pragma unroll
          for (int i = 0; i < kRow; ++i) {
            bk[i] = kNone;
            seq[i * C::kSeqStride + tid] = 0;
          }
          continue;
        }
        if (long_tile && long_tiles) return;
        for (uint32_t U = tid; U <= kPMask; U += NT) key_at(U) = pt[U];
        sync();
#pragma unroll
        for (int i = 0; i < kRow; ++i) bk[i] = skey[s1 * (kRow + 1) + i];
      }
    }
    if (long_tile) {
      // only with the row kernel around (the host's bound)
      if (tid == 0) atomicOr(flags, kErrWorkspace);
      return;
    }
    phase = 1;
  }

  // w(I(T, U)) = 0 outside the tile's list; the listed entries replace theirs
  if (cT != 0) {
    for (uint32_t i = tid; i < cT; i += NT) {
      key_at(sh.u[i]) = sh.f[i];
      seq_at(sh.u[i]) = (uint16_t)(kListed | i);
    }
    sync();
  }
  const size_t tbase = (size_t)T << kPB;
  const uint32_t nat_lo = perm.nat(tid);
  for (uint32_t UB = 0; UB <= kPMask; UB += kMeet * NT) {
  uint32_t ta_of[kMeet];
#pragma unroll
  for (int q = 0; q < kMeet; ++q) {
    const uint32_t U = (UB + (uint32_t)(q * NT)) | tid;
    ta_of[q] = !met && (seq_at(U) & kListed) ? 0u : ta_at(U);  // kListed, kSelf: no number of a queued pair
  }
#pragma unroll
  for (int q = 0; q < kMeet; ++q) {
    const uint32_t U0 = UB + (uint32_t)(q * NT);
    const uint32_t U = U0 | tid, nat = nat_lo | perm.nat(U0);
    Key key = key_at(U);
    const uint32_t number = cT != 0 ? seq_at(U) : 0u;
    uint32_t A;
    if ((number & kListed) && number != kSelf) {
      A = sh.sp[number & ~kListed];
    } else {
      A = (((uint32_t)(key & kPMask) + nat - kPMask) << L) | (number == kSelf ? T : ta_of[q]);
      key &= ~(Key)kPMask;  // F << b
    }
    if (MPT_BAD(flags, valid_split(T | (nat << L), A))) continue;
    Gp[tbase | U] = key;
    Gc[tbase | U] = key | (Key)(~nat & kPMask);
    split_rot[tbase | U] = A;
  }
  }
  };
  // the first unit of a group is its own number, the others come from *next
  const uint32_t units = tiles * items, own = gridDim.x * (blockDim.x / NT);
  for (uint32_t unit = blockIdx.x + gridDim.x * group; unit < units;) {
    run(unit);
    if (own >= units) break;
    sync();  // every thread is done with the unit's shared memory
    if (tid == 0) sh.unit = own + atomicAdd(next, 1u);
    sync();
    unit = sh.unit;
  }
  earlier();  // a layer is finished only behind the one before
}

template <typename Key, typename G>
cudaError_t tables(const Shape& s, const Workspace& ws, G* wIr, cudaStream_t stream, int* launches) {
  const int64_t tiles = (int64_t)1 << s.L, most = sm_count() * 8 * 8;
  k_prune_tiles<Key><<<(unsigned)(tiles < most ? tiles : most), 256, 0, stream>>>(
      s.L, s.prune_pairs, s.n_shared, ws.shared_N, ws.shared_w, wIr, ws.prune_info, ws.prune_rows, ws.counters);
  k_prune_members<<<(unsigned)s.L, 1024, 0, stream>>>(s.L, ws.prune_info, ws.prune_short, ws.prune_long, ws.prune_n);
  *launches += 2;
  if (s.prune_sort) {
    const unsigned blocks = (unsigned)(tiles / 256 + 1 < sm_count() * 4 ? tiles / 256 + 1 : sm_count() * 4);
    uint32_t* placed = ws.prune_hist + kMaxMembersL * kPruneClasses;
    k_prune_classes<<<blocks, 256, 0, stream>>>(s.L, s.n_shared, ws.shared_N, ws.counters, ws.prune_hist,
                                                ws.prune_class);
    k_prune_order<<<blocks, 256, 0, stream>>>(s.L, ws.prune_class, ws.prune_hist, placed, ws.prune_order);
    *launches += 2;
  }
  return cudaGetLastError();
}

template <typename Key, typename Tab, int kSlots_>
cudaError_t launch_layer(const Shape& s, const Workspace& ws, const Tab* wIr, int kh, uint32_t items, int groups,
                         unsigned long long units, unsigned long long* partial, Key* Gp, Key* Gc, cudaStream_t stream) {
  using C = PrunedCfg<Key, kSlots_>;
  static_assert(sizeof(PrunedShared<Key, kSlots_>) <= C::kSharedBytes, "a group's shared values");
  auto k = k_dp_pruned<Key, Tab, kSlots_>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kGroupBytes * C::kGroups);
  if (e != cudaSuccess) return e;
  const unsigned long long sms = (unsigned long long)sm_count();
  const uint32_t* order = nullptr;
  if (s.prune_sort) {
    unsigned long long before = 0;
    for (int q = 0; q < kh; ++q) before += h_binom.v[s.L][q];
    order = ws.prune_order + before;
  }
  // The layer may start while the one before runs out of blocks: its first
  // units' candidates, queues and lists do not depend on it.  24 requests of 10
  // passages, 12 layers: 0.40 -> 0.33 ms per solve; 23 of 40: 0.73 -> 0.67 ms.
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(sizeof(Key) == 8 || units < sms ? units : sms));
  cfg.blockDim = dim3((unsigned)(C::kRows * groups));
  cfg.dynamicSmemBytes = (size_t)(C::kGroupBytes * groups);
  cfg.stream = stream;
  cudaLaunchAttribute early{};
  early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &early;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, s.L, kh, items, s.prune_long, s.prune_pairs, s.perm, order, wIr,
                            (const uint32_t*)ws.prune_info, (const uint2*)ws.prune_rows, (const uint32_t*)ws.prune_short,
                            (const uint32_t*)ws.prune_long, (const uint32_t*)ws.prune_n, partial, ws.partial_ta,
                            ws.prune_done, ws.prune_done + kPruneSplitTiles + kh, Gp, Gc, ws.split_rot,
                            ws.counters + 1);
}

template <typename Key, typename Tab>
cudaError_t layer(const Shape& s, const Workspace& ws, const Tab* wIr, int kh, uint32_t items,
                  unsigned long long* partial, Key* Gp, Key* Gc, cudaStream_t stream, int* launches) {
  // a block per SM, and in it as many groups as there are units for; 64-bit
  // groups, whose eight warps are balanced by themselves, as blocks of one
  // (m = 24, weights x 4096: 0.41 ms of tile stage, 0.44 with two to a block).
  // Where a group has an SM, or half of one, to itself, nothing but copies
  // further ahead hides their latency: 23 requests of 40 passages, six of whose
  // eleven steps are of that size, 1.01 -> 0.93 ms from create to tables.
  const unsigned long long units = h_binom.v[s.L][kh] * items, sms = (unsigned long long)sm_count();
  ++*launches;
  if (units <= sms)
    return launch_layer<Key, Tab, sizeof(Key) == 8 ? 4 : 6>(s, ws, wIr, kh, items, 1, units, partial, Gp, Gc, stream);
  if constexpr (sizeof(Key) == 8) {
    return launch_layer<Key, Tab, 2>(s, ws, wIr, kh, items, 1, units, partial, Gp, Gc, stream);
  } else {
    if (units <= 2 * sms) return launch_layer<Key, Tab, 4>(s, ws, wIr, kh, items, 2, units, partial, Gp, Gc, stream);
    const int groups = units >= sms * 4 ? 4 : (int)((units + sms - 1) / sms);
    return launch_layer<Key, Tab, 2>(s, ws, wIr, kh, items, groups, units, partial, Gp, Gc, stream);
  }
}

// The members of each single request's list by k_prune_tiles' rules: the
// listed rows, members and cost of {l} bound those of every T that holds l.
struct ByteSums {
  uint8_t bits[256] = {}, eighths[256] = {};  // set bits; sum over them of 8 >> bits of their number
};
constexpr ByteSums make_byte_sums() {
  ByteSums t{};
  for (int v = 1; v < 256; ++v) t.bits[v] = (uint8_t)(t.bits[v >> 1] + (v & 1));
  for (int v = 0; v < 256; ++v)
    for (int i = 0; i < 8; ++i)
      if (v >> i & 1) t.eighths[v] = (uint8_t)(t.eighths[v] + (8 >> t.bits[i]));
  return t;
}

template <typename Key>
void singles(int L, const InnerPerm& perm, const uint32_t* sets, size_t n, bool* tiles, bool* pairs, double* costs) {
  using C = PrunedCfg<Key>;
  static constexpr ByteSums kByte = make_byte_sums();
  *tiles = *pairs = false;
  for (int l = 0; l < L; ++l) {
    uint32_t row[C::kRows] = {1u};
    for (size_t i = 0; i < n; ++i)
      if (sets[i] >> l & 1u) {
        const uint32_t v = perm.stored(sets[i] >> L);
        row[v >> C::kRB] |= 1u << (v & (C::kRow - 1));
      }
    static constexpr uint32_t kWithout[5] = {0x55555555u, 0x33333333u, 0x0F0F0F0Fu, 0x00FF00FFu, 0x0000FFFFu};
    for (int j = 0; j < C::kRB; ++j)
      for (uint32_t& r : row) r |= r >> (1 << j) & kWithout[j];
    for (uint32_t bit = 1; bit < (uint32_t)C::kRows; bit <<= 1)
      for (uint32_t r = 0; r < (uint32_t)C::kRows; ++r)
        if (!(r & bit)) row[r] |= row[r | bit];
    uint32_t rows = 0, members = 0, cost = 0;
    for (uint32_t r = 0; r < (uint32_t)C::kRows; ++r) {
      if (row[r] == 0) continue;
      uint32_t steps = 0;
      for (int q = 0; q < C::kRow / 8; ++q) {
        const uint32_t v = row[r] >> (8 * q) & 255u;
        steps += kByte.eighths[v] * ((uint32_t)C::kRow / 8) >> kByte.bits[q];  // q: the members' bits above the byte
        members += kByte.bits[v];
      }
      ++rows;
      cost += (steps + kUnitSteps) << (C::kLogWarps - kByte.bits[r >> 5]);
    }
    const bool many = rows > (uint32_t)kPruneRows, is_long = sizeof(Key) == 4 && (many || cost > kLongSteps);
    *pairs = *pairs || is_long;
    *tiles = *tiles || is_long || many || members > (uint32_t)kPruneSelf;
    costs[l] = is_long ? kFullPairSteps : (double)cost;
  }
}

// Blocks per tile of a layer with 32-bit keys.  The pairs of a tile vary from
// one to the bound, so a layer is cut so that its longest tile gives blocks of
// about kPartPairs pairs, as far as kMostBlocks blocks go round; blocks that
// find no part of theirs leave after counting the tile's pairs.
uint32_t pruned_items(const Shape& s, int kh) {
  constexpr double kPartPairs = 48, kMostBlocks = 16384;
  const double tiles = (double)h_binom.v[s.L][kh];
  if (s.wide || kh < 2 || tiles > kPruneSplitTiles) return 1;
  const double P = (double)((1ull << (kh - 1)) - 1ull), most = P < s.prune_most ? P : s.prune_most;
  const double items = most / kPartPairs < kMostBlocks / tiles ? most / kPartPairs : kMostBlocks / tiles;
  return items < 1.0 ? 1u : (uint32_t)items;
}

// Whether the pruned recurrence is the faster one where some list or tile is
// left to the pair and row kernels.  Each layer takes as long as its work over
// all SMs or a block's part of its heaviest tile, whichever is more, in this
// kernel and in the pair kernel, besides what the kernels of a layer take with
// nothing to do; work in warp steps of the lists, on the 152 SMs of a GB300 (no
// CUDA call is made here).  The lists of one Ta are the sum over the sets N with
// Ta within N_T of the list of N alone (a product over its bits, as
// k_prune_tiles counts it), less what the sets have in common: the singles'
// lists are known, and with sum S and union e of those of {l}, and C such that
// e = S / (1 + S / C), the n larger Ta's with lowest request l and sum t over all
// of them are taken as t / (1 + t / (n C)).
//
// Constants (ms): fitted to solves of 2,300 instances of 13 to 28 requests whose
// estimate matters (random sets of one density or size, few large ones, pooled
// passages, uniform requests; both key widths): median error 0 to 6 %, 5 % to
// 95 % of them within -24 .. +50 %.  Full solves: fitted to the same, from
// below (m = 13 to 27: 0.13 .. 229 ms, 64-bit keys m = 13 to 24: 0.17 .. 62 ms).
// Of the 801 of them that the pairs' estimate alone (Overlap in mpt_api.cu) would
// send here, 240 were slower than the full form by more than 5 %, by up to 2.9
// times and, with 64-bit keys, which have no pair kernel for a heavy list, 14
// times.  This rule takes 466 of them, one of which is (by 9 %), and leaves 41
// out that would be faster by more than 10 % (by up to 1.7 times).
template <typename Key>
bool pruned_pays(const Shape& s, const InnerPerm& perm, const uint32_t* sets, size_t n, const double* single,
                 bool pairs) {
  using C = PrunedCfg<Key>;
  constexpr bool kWide = sizeof(Key) == 8;
  // a warp step over all SMs and in one block, of a short list and in the pair kernel
  constexpr double kStep[2] = {kWide ? 5e-9 : 2.4e-9, 2.4e-9}, kOwnStep[2] = {kWide ? 1.7e-6 : 7e-7, 3e-7};
  const double per_solve = kWide ? 0.157 : pairs ? 0.077 : 0.112, per_layer = kWide ? 0.0247 : pairs ? 0.063 : 0.0302,
               per_tile = kWide ? 1e-5 : pairs ? 2e-4 : 2.8e-5;
  const int L = s.L;
  double three = 1.0;
  for (int l = 0; l < L; ++l) three *= 3.0;
  const double full = kWide ? 0.06 + 0.11 * L + 1.08e-4 * three : 0.06 + 0.066 * L + 1.55e-5 * three;
  auto choose = [](int a, int i) { return i < 0 || i > a ? 0.0 : (double)h_binom.v[a][i]; };
  // sums of the sets' lists (short, long), by lowest request l of a Ta and requests of N_T above l
  double sum[2][kMaxMembersL][kMaxMembersL] = {};
  for (size_t q = 0; q < n; ++q) {
    const uint32_t v = perm.stored(sets[q] >> L), row = v >> C::kRB;
    const int in_row = __builtin_popcount(v & (C::kRow - 1)), lanes = __builtin_popcount(row & 31u),
              warps = __builtin_popcount(row >> 5);
    double cost = (double)C::kRow;
    for (int i = 0; i < in_row; ++i) cost *= 1.5;
    cost = (cost + kUnitSteps) * (double)(1u << lanes) * (double)(1u << C::kLogWarps);
    for (int i = 0; i < warps; ++i) cost *= 1.5;
    const bool is_long = !kWide && (lanes + warps > 5 || cost > kLongSteps);
    int above = 0;
    for (int l = L - 1; l >= 0; --l)
      if (sets[q] >> l & 1u) sum[is_long][l][above++] += is_long ? kFullPairSteps : cost;
  }
  double layer[2][kMaxMembersL + 1] = {}, heaviest[2][kMaxMembersL + 1] = {};
  for (int l = 0; l < L; ++l) {
    const int A = L - 1 - l;
    double S = 0.0;
    int used[kMaxMembersL], n_used = 0;  // the a that occur
    for (int a = 0; a < L; ++a) {
      const double here = sum[0][l][a] + sum[1][l][a];
      S += here;
      if (here > 0.0) used[n_used++] = a;
    }
    const double e = single[l];
    const bool e_long = !kWide && e >= kFullPairSteps;
    const double Cs = S > 0.0 && e < 0.999 * S ? e * S / (S - e) : 0.0;  // 0: nothing in common
    // the lists (t[0] short, t[1] long) of `count` Ta's of i + 1 requests, at most `cap` of them above l
    auto lists = [&](int i, int cap, double count, double* t) {
      t[0] = t[1] = 0.0;
      for (int q = n_used - 1; q >= 0 && used[q] >= i; --q) {
        const double c = choose(used[q] < cap ? used[q] : cap, i);
        t[0] += sum[0][l][used[q]] * c;
        t[1] += sum[1][l][used[q]] * c;
      }
      const double all = t[0] + t[1];
      if (all == 0.0) return false;
      if (Cs > 0.0 && count > 0.0) {
        const double f = count * Cs / (count * Cs + all);
        t[0] *= f;
        t[1] *= f;
      }
      return true;
    };
    double t[2];
    for (int i = 0; i <= A; ++i) {  // Ta = l and i more
      if (i == 0) {
        t[e_long] = e;
        t[!e_long] = 0.0;
      } else if (!lists(i, L, choose(A, i), t)) {
        break;
      }
      for (int kh = i + 2; kh <= L && kh - 1 <= A; ++kh)
        for (int q = 0; q < 2; ++q) layer[q][kh] += t[q] * choose(A - i, kh - 1 - i);
    }
    for (int kh = 2; kh - 1 <= A; ++kh) {
      double v[2] = {e_long ? 0.0 : e, e_long ? e : 0.0};
      for (int i = 1; i < kh - 1 && lists(i, kh - 1, choose(kh - 1, i), t); ++i) {
        v[0] += t[0];
        v[1] += t[1];
      }
      for (int q = 0; q < 2; ++q) heaviest[q][kh] = std::max(heaviest[q][kh], v[q]);
    }
  }
  double ms = per_solve + per_layer * L + per_tile * (double)(1ull << L);
  for (int kh = 2; kh <= L; ++kh) {
    const double parts[2] = {(double)pruned_items(s, kh), (double)listed_items(L, kh, 152)};
    for (int q = 0; q < 2; ++q) ms += std::max(kStep[q] * layer[q][kh], kOwnStep[q] * heaviest[q][kh] / parts[q]);
  }
  return (pairs ? 1.15 : 1.1) * ms < full;
}

}  // namespace

bool prune_singles(const Shape& s, const InnerPerm& perm, const uint32_t* sets, size_t n, bool* tiles, bool* pairs) {
  double costs[kMaxMembersL];
  if (s.wide) {
    singles<unsigned long long>(s.L, perm, sets, n, tiles, pairs, costs);
    return !*tiles || pruned_pays<unsigned long long>(s, perm, sets, n, costs, *pairs);
  }
  singles<uint32_t>(s.L, perm, sets, n, tiles, pairs, costs);
  return !*tiles || pruned_pays<uint32_t>(s, perm, sets, n, costs, *pairs);
}

cudaError_t launch_prune_tables(const Shape& s, const Workspace& ws, cudaStream_t stream, int* launches) {
  const size_t cleared = kPruneSplitTiles + kMaxMembersL + 2 * kMaxMembersL * kPruneClasses;
  cudaError_t e = cudaMemsetAsync(ws.prune_done, 0, cleared * 4, stream);
  if (e != cudaSuccess) return e;
  auto* lean = reinterpret_cast<unsigned int*>(ws.fw_rot);
  auto* full = reinterpret_cast<unsigned long long*>(ws.wI_rot);
  if (s.wide)
    return s.lean ? tables<unsigned long long>(s, ws, lean, stream, launches)
                  : tables<unsigned long long>(s, ws, full, stream, launches);
  return s.lean ? tables<uint32_t>(s, ws, lean, stream, launches) : tables<uint32_t>(s, ws, full, stream, launches);
}

// Whether the blocks of a layer meet in `partial`.
bool pruned_meet(const Shape& s, int kh, uint32_t items) {
  if (s.wide || kh < 2) return false;
  const double P = (double)((1ull << (kh - 1)) - 1ull);
  return s.prune_long || items > 1 || (P < s.prune_most ? P : s.prune_most) > (double)kPQueue;
}

cudaError_t launch_dp_pruned(const Shape& s, const Workspace& ws, cudaStream_t stream, int* launches,
                             BlockedTiming* timing) {
  cudaError_t e = cudaSuccess;
  auto mark = [&](cudaEvent_t* ev, int i) {
    if (timing && ev) cudaEventRecord(ev[i], stream);
  };
  for (int kh = 0; kh <= s.L && e == cudaSuccess; ++kh) {
    const uint32_t items = pruned_items(s, kh);
    if (pruned_meet(s, kh, items))
      e = cudaMemsetAsync(ws.partial, 0xFF, (size_t)(h_binom.v[s.L][kh] << kPB) * sizeof(unsigned long long), stream);
    if (e == cudaSuccess && kh >= 2 && s.prune_pairs) {
      if (timing) mark(timing->pair_ev, 2 * timing->pair_launches);
      e = launch_listed_pairs(s, ws, kh, stream, launches);
      if (timing) mark(timing->pair_ev, 2 * timing->pair_launches++ + 1);
    }
    if (timing) mark(timing->tile_ev, 2 * timing->tile_launches);
    if (e == cudaSuccess && kh == 0) {
      e = launch_tile0(s, ws, stream);
      ++*launches;
    } else if (e == cudaSuccess) {
      if (s.wide)
        e = s.lean ? layer(s, ws, ws.fw_rot, kh, items, ws.partial, ws.Gp64, ws.Gc64, stream, launches)
                   : layer(s, ws, ws.wI_rot, kh, items, ws.partial, ws.Gp64, ws.Gc64, stream, launches);
      else
        e = s.lean ? layer(s, ws, ws.fw_rot, kh, items, ws.partial, ws.Gp, ws.Gc, stream, launches)
                   : layer(s, ws, ws.wI_rot, kh, items, ws.partial, ws.Gp, ws.Gc, stream, launches);
      if (e == cudaSuccess && s.prune_long)
        e = s.wide ? launch_wide_listed_tiles(s, ws, kh, stream, launches)
                   : launch_listed_tiles(s, ws, kh, stream, launches);
    }
    if (timing) mark(timing->tile_ev, 2 * timing->tile_launches++ + 1);
  }
  return e;
}

}  // namespace mpt
