// K3, wide blocked form: the Sec. 3.1 recurrence
//     F({i}) = w(R_i),   F(S) = min over S = A (+) B of F(A) + F(B) - w(I(S)),
// with the tiling of k_dp_blocked.cu (rotated tables, tile T and inner U,
// proper pairs per window pair, the self pair inside the tile) and 64-bit
// packed keys, for instances whose candidate sums do not fit the 32-bit keys
// (shared weight sum_i w(R_i) - sum_i pi_i - m u >= 2^(32-b), F and w(I) less
// the offsets of k_scatter_zeta.cu) but stay below 2^51:
//     key = Gp[A] + Gc[B] = ((F(A) + F(B)) << b) | (2^b - 1 - U + Ua),
// Gp = F << b and Gc = Gp | (~u & (2^b - 1)) as uint64.  The candidates and
// the tie order (value, Ua, Ta) are those of the 32-bit path, so the argmin is
// the same: the least A as an integer among the optimal splits.
//
// Pair kernel.  Windows of 4096 uint64 entries are 256 rows of 16, padded to
// 18 words and XOR-placed.  A unit (s1, a1) is one 4-bit register
// convolution (81 add-min steps) of row a1 of X with row s1 ^ a1 of Y into
// the 16 outputs of row s1.  The 3^8 = 6561 units of a window pair come in
// 1645 chunks (the units of one row with fixed low bits: 4, or 1-2 for the
// rows with fewer than 2 bits), cut into 256 ranges of 7 or 6 consecutive
// chunks; warps 0..3 run the 7-chunk ranges and warps 4..7 the others, so
// each sub-partition issues 13 chunk-times per pair for 12.85 of work.  A thread
// keeps one row's 16 minima in registers while its chunks stay in that row,
// and merges them into a per-pair shared array (64-bit atomicMin) when the
// row changes.  Owners fold the array into running (key, Ta) bests after
// every pair (pairs in increasing Ta, strict improvement), and each block
// writes its 4096 bests to a slot of its own: no atomics in global memory.
//
// Tile kernel (|T| >= 1; tile 0 is k_dp_tile0.cu's).  One block per tile
// finishes all 4096 entries by rows of 16, level by level in the row bits: the
// self pair (A = (T, Ua), B = (0, U \ Ua)) and the lexicographic (key, Ta)
// minimum with the tile's pair slots.
#include "mpt_internal.cuh"

namespace mpt {
namespace {

using u64 = unsigned long long;

constexpr int kWB = 12;                   // inner bits
constexpr int kWB2 = 4;                   // inner bits held in registers
constexpr int kWB1 = kWB - kWB2;          // 8 row bits
constexpr int kWRow = 1 << kWB2;          // 16 entries per row
constexpr int kWRowStride = kWRow + 2;    // 18 words (144 bytes): XOR-placed rows start in distinct bank groups
constexpr int kWRows = 1 << kWB1;         // 256 rows
constexpr int kWWin = kWRows * kWRowStride;
constexpr int kWThreads = 256;
constexpr int kWOwned = (1 << kWB) / kWThreads;  // 16 outputs folded per thread
constexpr int kWSmemBytes = (2 * 2 * kWWin + 2 * (1 << kWB)) * (int)sizeof(u64);
constexpr int kWTileThreads = 288;
constexpr int kWBestWords = (1 << kWB) + kWRows;  // per-output arrays, rows 17 words apart
constexpr int kWTileSmemBytes = (2 * kWWin + kWBestWords) * (int)sizeof(u64) + kWBestWords * (int)sizeof(uint32_t);
constexpr int kWChunks = 1645;
constexpr int kWLong = 109;               // threads with 7 chunks; the others take 6

static_assert(kWLong * 7 + (kWThreads - kWLong) * 6 == kWChunks, "chunk split");
static_assert(kWSmemBytes <= 227 * 1024 && kWTileSmemBytes <= 227 * 1024, "shared memory");

constexpr int popc8(uint32_t v) {
  int c = 0;
  while (v) {
    v &= v - 1;
    ++c;
  }
  return c;
}

constexpr uint32_t deposit8(uint32_t q, uint32_t mask) {
  uint32_t out = 0;
  while (mask) {
    const uint32_t lowb = mask & (~mask + 1u);
    if (q & 1u) out |= lowb;
    q >>= 1;
    mask ^= lowb;
  }
  return out;
}

struct WidePlan {
  uint32_t chunk[kWChunks];          // s1 | fixed << 8 | free << 16
  uint16_t first[kWThreads];         // thread t runs chunks first[t] .. first[t] + count[t] - 1
  uint16_t count[kWThreads];
  int nchunk, total;
};

// Chunks in increasing row order.  Rows with >= 2 bits: the two highest bits
// are free (4 units in Gray order), the others fixed; a 1-bit row is one
// chunk of 2 units, row 0 one chunk of 1 unit.
constexpr WidePlan make_wide_plan() {
  WidePlan pl{};
  int n = 0;
  for (uint32_t s1 = 0; s1 < (uint32_t)kWRows; ++s1) {
    const int p = popc8(s1);
    if (p < 2) {
      pl.chunk[n++] = s1 | (s1 << 16);
      continue;
    }
    uint32_t top = 0, r = s1;
    for (int t = 0; t < 2; ++t) {
      uint32_t hb = 0;
      for (int bit = kWB1 - 1; bit >= 0; --bit)
        if ((r >> bit) & 1u) {
          hb = 1u << bit;
          break;
        }
      top |= hb;
      r ^= hb;
    }
    const uint32_t lowm = s1 ^ top;
    for (uint32_t v = 0; v < (1u << (p - 2)); ++v) pl.chunk[n++] = s1 | (deposit8(v, lowm) << 8) | (top << 16);
  }
  pl.nchunk = n;
  // Ranges r = 0..255 of consecutive chunks, 7 for r < 109 and 6 after.  Lane
  // l of warp w runs range 4 l + w (warps 0..3) or 128 + 4 l + (w - 4): the
  // 7-chunk ranges stay on warps 0..3, and neighbouring lanes work 4 ranges
  // (about 26 chunks) apart, mostly in different rows, so their flushes do
  // not hit the same words.
  int firsts[kWThreads] = {};
  int c = 0;
  for (int r = 0; r < kWThreads; ++r) {
    firsts[r] = c;
    c += r < kWLong ? 7 : 6;
  }
  pl.total = c;
  for (int t = 0; t < kWThreads; ++t) {
    const int w = t / 32, l = t % 32;
    const int r = w < 4 ? 4 * l + w : 128 + 4 * l + (w - 4);
    pl.first[t] = (uint16_t)firsts[r];
    pl.count[t] = (uint16_t)(r < kWLong ? 7 : 6);
  }
  return pl;
}

constexpr WidePlan kWidePlanHost = make_wide_plan();
static_assert(kWidePlanHost.nchunk == kWChunks && kWidePlanHost.total == kWChunks, "chunk plan");
static __constant__ WidePlan c_wplan = make_wide_plan();

// Row placement: the low 3 row bits XOR-ed with higher ones; linear over GF(2).
__device__ __forceinline__ uint32_t row_pos_w(uint32_t r) { return r ^ (((r >> 3) ^ (r >> 6)) & 7u); }

__device__ __forceinline__ void cp_async16_w(void* smem_dst, const void* gmem_src) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_commit_w() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait_w() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Copy the two windows of a pair: thread t moves the 16-byte chunks t + 256 j
// (j < 8) of each window, i.e. rows (t >> 3) + 32 j, column t & 7.
__device__ __forceinline__ void stage_pair_w(u64* X, u64* Y, const u64* __restrict__ gx, const u64* __restrict__ gy) {
  const uint32_t t = threadIdx.x;
  const uint32_t rp0 = row_pos_w(t >> 3);
  const uint32_t col = (t & 7u) * 2u;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint32_t d = (rp0 ^ row_pos_w((uint32_t)(32 * j))) * kWRowStride + col;
    cp_async16_w(X + d, gx + 2 * (t + (uint32_t)(kWThreads * j)));
    cp_async16_w(Y + d, gy + 2 * (t + (uint32_t)(kWThreads * j)));
  }
}

__device__ __forceinline__ void load_row_w(u64 (&v)[kWRow], const u64* p) {
  const ulonglong2* q = reinterpret_cast<const ulonglong2*>(p);
#pragma unroll
  for (int c = 0; c < kWRow / 2; ++c) {
    const ulonglong2 t = q[c];
    v[2 * c] = t.x;
    v[2 * c + 1] = t.y;
  }
}

// acc[s2] = min(acc[s2], min over a2 in s2 of x[a2] + y[s2 ^ a2])  (81 steps)
__device__ __forceinline__ void conv16(u64 (&acc)[kWRow], const u64 (&x)[kWRow], const u64 (&y)[kWRow]) {
#pragma unroll
  for (int a2 = 0; a2 < kWRow; ++a2) {
#pragma unroll
    for (int s2 = 0; s2 < kWRow; ++s2) {
      if ((a2 & s2) == a2) {
        const u64 c = x[a2] + y[s2 ^ a2];
        acc[s2] = c < acc[s2] ? c : acc[s2];
      }
    }
  }
}

__global__ void __launch_bounds__(kWThreads, 1)
k_dp_pairs_w(const u64* __restrict__ Gp, const u64* __restrict__ Gc, u64* __restrict__ pkey, uint32_t* __restrict__ pta,
             int L, int kh, uint32_t pairs_per_tile, uint32_t items_per_tile, uint32_t pairs_per_item,
             int32_t* __restrict__ flags) {
  extern __shared__ __align__(16) u64 wsm[];
  u64* pmin = wsm + 4 * kWWin;  // two per-pair minimum arrays of 4096

  const uint32_t tile = blockIdx.x / items_per_tile;
  const uint32_t item = blockIdx.x % items_per_tile;
  const uint32_t T = colex_unrank(tile, kh, L);
  const uint32_t low = T & (~T + 1u);
  const uint32_t R = T ^ low;
  const uint32_t q0 = item * pairs_per_item;
  const uint32_t q1 = min(q0 + pairs_per_item, pairs_per_tile);
#ifdef MPT_BOUNDS
  {
    // the tile, and every pair's Ta: a proper part of T holding its lowest
    // request, so both windows lie inside the tables
    bool good = tile < c_binom.v[L][kh] && T < (1u << L) && __popc(T) == kh && q1 <= pairs_per_tile;
    uint32_t sb = deposit_bits(q0, R);
    for (uint32_t q = q0; q < q1 && good; ++q) {
      const uint32_t Ta = low | sb;
      good = (Ta & ~T) == 0 && Ta != T;
      sb = (sb - R) & R;
    }
    if (MPT_BAD(flags, good)) return;  // the same decision in every thread
  }
#endif
  // this thread's chunks, read from constant memory once (lanes read
  // different entries, which the constant cache serves one at a time)
  const uint32_t c0 = c_wplan.first[threadIdx.x];
  const int nch = (int)c_wplan.count[threadIdx.x];
  uint32_t chunks[7];
#pragma unroll
  for (int i = 0; i < 7; ++i) chunks[i] = i < nch ? c_wplan.chunk[c0 + i] : 0u;

  for (int i = threadIdx.x; i < 2 * (1 << kWB); i += kWThreads) pmin[i] = ~0ull;
  u64 bk[kWOwned];
  uint32_t bt[kWOwned];
#pragma unroll
  for (int j = 0; j < kWOwned; ++j) {
    bk[j] = ~0ull;
    bt[j] = 0;
  }

  uint32_t sub = deposit_bits(q0, R);
  {
    const uint32_t Ta = low | sub;
    stage_pair_w(wsm, wsm + kWWin, Gp + ((size_t)Ta << kWB), Gc + ((size_t)(T ^ Ta) << kWB));
    cp_async_commit_w();
  }
  for (uint32_t q = q0; q < q1; ++q) {
    const int cur = (int)((q - q0) & 1u);
    const uint32_t Ta = low | sub;
    const uint32_t next = (sub - R) & R;
    if (q + 1 < q1) {
      const uint32_t Tn = low | next;
      u64* nb = wsm + 2 * (cur ^ 1) * kWWin;
      stage_pair_w(nb, nb + kWWin, Gp + ((size_t)Tn << kWB), Gc + ((size_t)(T ^ Tn) << kWB));
      cp_async_commit_w();
      cp_async_wait_w<1>();
    } else {
      cp_async_wait_w<0>();
    }
    __syncthreads();
    const u64* X = wsm + 2 * cur * kWWin;
    const u64* Y = X + kWWin;
    u64* pm = pmin + cur * (1 << kWB);
    {
      uint32_t row = 0xFFFFFFFFu;
      u64 acc[kWRow];
#pragma unroll
      for (int i = 0; i < kWRow; ++i) acc[i] = ~0ull;
#pragma unroll
      for (int c = 0; c < 7; ++c) {
        if (c >= nch) break;
        const uint32_t ch = chunks[c];
        const uint32_t s1 = ch & 0xFFu, fixed = (ch >> 8) & 0xFFu, freem = (ch >> 16) & 0xFFu;
        if (s1 != row) {
          if (row != 0xFFFFFFFFu) {
#pragma unroll
            for (int i = 0; i < kWRow; ++i) atomicMin(&pm[(row << kWB2) | (uint32_t)i], acc[i]);
          }
          row = s1;
#pragma unroll
          for (int i = 0; i < kWRow; ++i) acc[i] = ~0ull;
        }
        const uint32_t ps1 = row_pos_w(s1);
        const uint32_t b0 = freem & (~freem + 1u), b1 = freem ^ b0;
        const int nunits = freem == 0 ? 1 : (b1 == 0 ? 2 : 4);
        uint32_t pa = row_pos_w(fixed);
#pragma unroll 1
        for (int k = 0; k < nunits; ++k) {
          // Gray order over the free bits: fixed, ^b0, ^b1, ^b0
          if (k > 0) pa ^= row_pos_w((k & 1) ? b0 : b1);
          u64 x[kWRow], y[kWRow];
          load_row_w(x, X + pa * kWRowStride);
          load_row_w(y, Y + (pa ^ ps1) * kWRowStride);
          conv16(acc, x, y);
        }
      }
      if (row != 0xFFFFFFFFu) {
#pragma unroll
        for (int i = 0; i < kWRow; ++i) atomicMin(&pm[(row << kWB2) | (uint32_t)i], acc[i]);
      }
    }
    __syncthreads();
    // fold this pair's minima into the running bests; reset the array for the
    // pair after next
#pragma unroll
    for (int j = 0; j < kWOwned; ++j) {
      const uint32_t o = threadIdx.x + (uint32_t)(j * kWThreads);
      const u64 v = pm[o];
      pm[o] = ~0ull;
      if (v < bk[j]) {
        bk[j] = v;
        bt[j] = Ta;
      }
    }
    sub = next;
  }

  const size_t slot = (size_t)blockIdx.x << kWB;
#pragma unroll
  for (int j = 0; j < kWOwned; ++j) {
    const uint32_t o = threadIdx.x + (uint32_t)(j * kWThreads);
    pkey[slot + o] = bk[j];
    pta[slot + o] = bt[j];
  }
}

template <typename Tab>
__device__ __forceinline__ int64_t load_wI_w(const Tab* p) {
  return (int64_t)__ldg(p);
}

// Folds a tile's `items` slots into its first one: the lexicographic
// (key, Ta) minimum of each output.  A block takes 32 outputs with 8 warps
// that share the slots; it reads and writes only its own outputs.
__global__ void __launch_bounds__(256)
k_fold_slots_w(u64* __restrict__ pkey, uint32_t* __restrict__ pta, uint32_t items) {
  __shared__ u64 sk[8][32];
  __shared__ uint32_t st[8][32];
  const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5;
  const size_t first = ((size_t)(blockIdx.x >> (kWB - 5)) * items << kWB) | ((blockIdx.x & ((1u << (kWB - 5)) - 1u)) << 5) | lane;
  u64 best = ~0ull;
  uint32_t ta = ~0u;
#pragma unroll 4
  for (uint32_t it = w; it < items; it += 8) {
    const u64 k = pkey[first + ((size_t)it << kWB)];
    const uint32_t t = pta[first + ((size_t)it << kWB)];
    if (k < best || (k == best && t < ta)) {
      best = k;
      ta = t;
    }
  }
  sk[w][lane] = best;
  st[w][lane] = ta;
  __syncthreads();
  if (w == 0) {
#pragma unroll
    for (int i = 1; i < 8; ++i) {
      const u64 k = sk[i][lane];
      const uint32_t t = st[i][lane];
      if (k < best || (k == best && t < ta)) {
        best = k;
        ta = t;
      }
    }
    pkey[first] = best;
    pta[first] = ta;
  }
}

// Word of output U = (s1, s2) in a per-output array: rows are 17 words apart,
// so threads that hold different rows and the same s2 hit different banks.
__device__ __forceinline__ uint32_t best_word_w(uint32_t U) { return U + (U >> kWB2); }

// Tile kernel, |T| = kh >= 1, 12 inner bits: the tile's rows of 16 level by
// level in |s1|, as k_dp_tile_rows does with 32-bit keys.  Candidates of
// U = (s1, s2) with Ua = (a1, a2), a proper subset of U:
//   * a1 a proper subset of s1: rows of this tile finished at earlier levels
//     against whole rows of tile 0, by the pair kernel's register convolution;
//   * a1 = s1: a 4-bit recurrence inside the row, in registers.
// Layers are short where this kernel matters (the pair kernel's work grows
// with 2^|T|, this one's does not), so a tile gets a block of 9 warps, which
// bound its chain: at the widest level 70 rows by 4 lanes.  A lane per few
// submasks with two dependent shared loads each, and a block barrier per size
// of U, took 565 us for one tile (m = 13); this form takes 75 us.
template <typename Tab>
__global__ void __launch_bounds__(kWTileThreads)
k_dp_tile_w(int L, int kh, const Tab* __restrict__ wIr, const u64* __restrict__ pkey, const uint32_t* __restrict__ pta,
            uint32_t items, uint32_t stride, u64* __restrict__ Gp, u64* __restrict__ Gc, uint32_t* __restrict__ split_rot,
            int32_t* __restrict__ flags, const uint32_t* __restrict__ info, InnerPerm perm) {
  extern __shared__ __align__(16) u64 tsm[];
  u64* cur = tsm;              // this tile, F << 12, padded rows
  u64* zc = cur + kWWin;       // tile 0, complement form, padded rows
  u64* bkey = zc + kWWin;      // best key per output so far
  uint32_t* bsplit = reinterpret_cast<uint32_t*>(bkey + kWBestWords);  // its Ta; after finishing, the split A
  constexpr uint32_t kMask = (1u << kWB) - 1u;

  const uint32_t tile = blockIdx.x;
  const uint32_t T = colex_unrank(tile, kh, L);
  const size_t tbase = (size_t)T << kWB;
  if (MPT_BAD(flags, tile < c_binom.v[L][kh] && T < (1u << L) && __popc(T) == kh)) return;
  if (info && !(info[T] & kTileLong)) return;  // finished by k_dp_pruned

  for (int c = threadIdx.x; c < (1 << (kWB - 1)); c += kWTileThreads) {
    const int row = c >> (kWB2 - 1), k = c & ((1 << (kWB2 - 1)) - 1);
    *reinterpret_cast<ulonglong2*>(zc + row_pos_w((uint32_t)row) * kWRowStride + 2 * k) =
        *reinterpret_cast<const ulonglong2*>(Gc + 2 * c);
  }
  for (int u = threadIdx.x; u < (1 << kWB); u += kWTileThreads) {
    u64 best = ~0ull;
    uint32_t ta = T;
    if (kh >= 2) {
      const size_t slot = ((size_t)tile * stride << kWB) | (uint32_t)u;
      best = pkey[slot];
      ta = pta[slot];
      for (uint32_t it = 1; it < items; ++it) {
        const u64 k = pkey[slot + ((size_t)it << kWB)];
        const uint32_t t = pta[slot + ((size_t)it << kWB)];
        if (k < best || (k == best && t < ta)) {
          best = k;
          ta = t;
        }
      }
    }
    bkey[best_word_w((uint32_t)u)] = best;
    bsplit[best_word_w((uint32_t)u)] = ta;
  }
  __syncthreads();

  for (int p1 = 0; p1 <= kWB1; ++p1) {
    const int rows = (int)c_binom.v[kWB1][p1];
    // the threads that finish this level's rows fetch their w(I(S)) now
    int64_t wv[kWRow];
    const bool finisher = (int)threadIdx.x < rows;
    const uint32_t s1f = finisher ? colex_unrank((unsigned long long)threadIdx.x, p1, kWB1) : 0u;
    if (finisher) {
#pragma unroll
      for (int i = 0; i < kWRow; ++i) wv[i] = load_wI_w(wIr + (tbase | (s1f << kWB2) | (uint32_t)i));
    }
    if (p1 >= 1) {
      int g = p1 < 5 ? p1 : 5;  // log2(lanes per row)
      while ((rows << g) > kWTileThreads) --g;
      const int G = 1 << g;
      const int ri = (int)(threadIdx.x >> g);
      const uint32_t r = threadIdx.x & (uint32_t)(G - 1);
      const bool active = ri < rows;
      u64 acc[kWRow];
#pragma unroll
      for (int i = 0; i < kWRow; ++i) acc[i] = ~0ull;
      uint32_t s1 = 0;
      if (active) {
        s1 = colex_unrank((unsigned long long)ri, p1, kWB1);
        uint32_t hi = 0, rr = s1;
        for (int t = 0; t < g; ++t) {
          const uint32_t top = 1u << (31 - __clz(rr));
          hi |= top;
          rr ^= top;
        }
        const uint32_t freem = s1 ^ hi;
        const uint32_t fixed = deposit_bits(r, hi);
        uint32_t sub = 0;
        do {
          const uint32_t a1 = fixed | sub;
          if (a1 != s1) {
            u64 x[kWRow], y[kWRow];
            load_row_w(x, cur + row_pos_w(a1) * kWRowStride);
            load_row_w(y, zc + row_pos_w(s1 ^ a1) * kWRowStride);
            conv16(acc, x, y);
          }
          sub = (sub - freem) & freem;
        } while (sub != 0);
      }
      for (int off = G >> 1; off > 0; off >>= 1) {
#pragma unroll
        for (int i = 0; i < kWRow; ++i) {
          const u64 o = __shfl_xor_sync(0xFFFFFFFFu, acc[i], off);
          acc[i] = o < acc[i] ? o : acc[i];
        }
      }
      if (active && r == 0) {
#pragma unroll
        for (int i = 0; i < kWRow; ++i) {
          const uint32_t o = best_word_w((s1 << kWB2) | (uint32_t)i);
          if (acc[i] < bkey[o]) {
            bkey[o] = acc[i];
            bsplit[o] = T;
          }
        }
      }
      __syncthreads();
    }
    if (finisher) {
      const uint32_t nat_s1 = info ? perm.nat(s1f << kWB2) : s1f << kWB2;  // stored order undone (pruned recurrence)
      u64 z[kWRow], c[kWRow];
      load_row_w(z, zc);  // row 0 is at position 0
#pragma unroll
      for (int s2 = 0; s2 < kWRow; ++s2) {
        u64 key = ~0ull;
#pragma unroll
        for (int a2 = 0; a2 < kWRow; ++a2) {
          if ((a2 & s2) == a2 && a2 != s2) {
            const u64 k = c[a2] + z[s2 ^ a2];
            key = k < key ? k : key;
          }
        }
        const uint32_t U = (s1f << kWB2) | (uint32_t)s2;
        u64 bk = bkey[best_word_w(U)];
        uint32_t bt = bsplit[best_word_w(U)];
        if (key < bk) {  // ties keep the smaller Ta, a proper part of T
          bk = key;
          bt = T;
        }
        int64_t f;
        uint32_t A;
        if (kh == 1 && U == 0) {  // S = T, a single request
          f = wv[s2];
          A = 0;
        } else {
          const uint32_t Ua = (uint32_t)(bk & kMask) + (nat_s1 | (info ? perm.nat((uint32_t)s2) : (uint32_t)s2)) - kMask;
          f = (int64_t)(bk >> kWB) - wv[s2];
          A = (Ua << L) | bt;
        }
        c[s2] = (u64)f << kWB;
        bsplit[best_word_w(U)] = A;
      }
      ulonglong2* dst = reinterpret_cast<ulonglong2*>(cur + row_pos_w(s1f) * kWRowStride);
#pragma unroll
      for (int q = 0; q < kWRow / 2; ++q) dst[q] = make_ulonglong2(c[2 * q], c[2 * q + 1]);
    }
    __syncthreads();
  }

  for (int u = threadIdx.x; u < (1 << kWB); u += kWTileThreads) {
    const u64 gp = cur[row_pos_w((uint32_t)u >> kWB2) * kWRowStride + (u & (kWRow - 1))];
    const uint32_t A = bsplit[best_word_w((uint32_t)u)];
    const uint32_t nat = info ? perm.nat((uint32_t)u) : (uint32_t)u;
    if (MPT_BAD(flags, valid_split(T | (nat << L), A))) continue;
    Gp[tbase | (uint32_t)u] = gp;
    Gc[tbase | (uint32_t)u] = gp | (u64)(~nat & kMask);
    split_rot[tbase | (uint32_t)u] = A;
  }
}

}  // namespace

int64_t wide_partial_slots(int m, int b) {
  const int L = m - b;
  unsigned long long most = 0;
  for (int k = 2; k <= L; ++k)
    if (h_binom.v[L][k] > most) most = h_binom.v[L][k];
  return most > 0 ? (int64_t)(2 * most) : 1;
}

namespace {

// More slots of a tile than this are folded by a kernel of their own: one
// block reading the 304 slots of the last tile would take as long as the tile.
constexpr uint32_t kWInlineSlots = 4;

// The tiles of step kh >= 1, with `items` slots each (info: the pruned
// recurrence's lists, or null).
void launch_wide_tiles(const Shape& s, const Workspace& ws, int kh, uint32_t items, const uint32_t* info,
                       cudaStream_t stream, int* launches) {
  const unsigned tiles = (unsigned)h_binom.v[s.L][kh];
  uint32_t stride = items;
  if (kh >= 2 && items > kWInlineSlots) {
    k_fold_slots_w<<<tiles << (kWB - 5), 256, 0, stream>>>(ws.partial, ws.partial_ta, items);
    ++*launches;
    items = 1;
  }
  auto run = [&](auto kernel, const auto* wI) {
    kernel<<<tiles, kWTileThreads, kWTileSmemBytes, stream>>>(s.L, kh, wI, ws.partial, ws.partial_ta, items, stride,
                                                              ws.Gp64, ws.Gc64, ws.split_rot, ws.counters + 1, info,
                                                              s.perm);
    ++*launches;
  };
  if (s.lean)
    run(k_dp_tile_w<int32_t>, ws.fw_rot);
  else
    run(k_dp_tile_w<int64_t>, ws.wI_rot);
}

cudaError_t wide_tile_attributes() {
  cudaError_t e = cudaFuncSetAttribute(k_dp_tile_w<int64_t>, cudaFuncAttributeMaxDynamicSharedMemorySize, kWTileSmemBytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_dp_tile_w<int32_t>, cudaFuncAttributeMaxDynamicSharedMemorySize, kWTileSmemBytes);
  return e;
}

}  // namespace

cudaError_t launch_wide_listed_tiles(const Shape& s, const Workspace& ws, int kh, cudaStream_t stream, int* launches) {
  const cudaError_t e = wide_tile_attributes();
  if (e != cudaSuccess) return e;
  launch_wide_tiles(s, ws, kh, 1u, ws.prune_info, stream, launches);
  return cudaGetLastError();
}

cudaError_t launch_dp_wide(const Shape& s, const Workspace& ws, cudaStream_t stream, int* launches,
                           BlockedTiming* timing, int step_begin, int step_end) {
  cudaError_t e = cudaFuncSetAttribute(k_dp_pairs_w, cudaFuncAttributeMaxDynamicSharedMemorySize, kWSmemBytes);
  if (e != cudaSuccess) return e;
  if ((e = wide_tile_attributes()) != cudaSuccess) return e;
  int sms = 0, dev = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;

  const int b = s.b, L = s.L;
  const unsigned long long slots = (unsigned long long)wide_partial_slots(s.m, b);
  constexpr unsigned long long evals_per_pair = 531441ull;
  if (step_end < 0 || step_end > L + 1) step_end = L + 1;
  for (int kh = step_begin < 0 ? 0 : step_begin; kh < step_end; ++kh) {
    const unsigned long long tiles = h_binom.v[L][kh];
    unsigned long long items = 0;
    if (kh >= 2) {
      const uint32_t P = (1u << (kh - 1)) - 1u;
      uint32_t ppi = P;
      const unsigned long long max_items = slots / tiles > 0 ? slots / tiles : 1;
      choose_items(tiles, P, sms, max_items, &items, &ppi);
      if (timing && timing->pair_ev) cudaEventRecord(timing->pair_ev[2 * timing->pair_launches], stream);
      k_dp_pairs_w<<<(unsigned)(tiles * items), kWThreads, kWSmemBytes, stream>>>(
          ws.Gp64, ws.Gc64, ws.partial, ws.partial_ta, L, kh, P, (uint32_t)items, ppi, ws.counters + 1);
      if (timing && timing->pair_ev) cudaEventRecord(timing->pair_ev[2 * timing->pair_launches + 1], stream);
      if (timing) {
        timing->pair_launches++;
        timing->pair_splits += (double)tiles * (double)P * (double)evals_per_pair;
      }
      ++*launches;
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if (timing && timing->tile_ev) cudaEventRecord(timing->tile_ev[2 * timing->tile_launches], stream);
    if (kh == 0) {
      e = launch_tile0(s, ws, stream);
      ++*launches;
    } else {
      launch_wide_tiles(s, ws, kh, (uint32_t)items, nullptr, stream, launches);
    }
    if (e != cudaSuccess) return e;
    if (timing && timing->tile_ev) cudaEventRecord(timing->tile_ev[2 * timing->tile_launches + 1], stream);
    if (timing) timing->tile_launches++;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace mpt
