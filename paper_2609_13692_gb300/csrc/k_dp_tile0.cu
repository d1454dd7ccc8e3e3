// Tile 0 of the blocked recurrences (k_dp_blocked.cu, k_dp_wide.cu,
// k_dp_pruned.cu): the whole Sec. 3.1 recurrence on the b inner bits, in one
// block, with 32- or 64-bit keys.  w(I) is read, and Gp = F << b,
// Gc = Gp | (~U & (2^b - 1)) and split are written, in the stored order of
// the inner bits; the keys and the recurrence use the natural one.
#include "mpt_internal.cuh"

namespace mpt {
namespace {

// Rows of 32 32-bit or 16 64-bit entries, 16 bytes apart beyond their 128, so
// that consecutive rows start in different bank groups.
template <typename Key>
struct Tile0Cfg {
  static constexpr int kRB = sizeof(Key) == 4 ? 5 : 4;
  static constexpr int kRow = 1 << kRB;
  static constexpr int kStride = kRow + 16 / (int)sizeof(Key);
  static constexpr int kRows = 1 << (12 - kRB);
  static constexpr int kLevelRows = sizeof(Key) == 4 ? 35 : 70;  // C(7, 3), C(8, 4)
  static constexpr int kSmem = (kRows * kStride + kRows * (kRow + 1) + kLevelRows * (kRow + 1)) * (int)sizeof(Key);
};
constexpr int kT0Threads = 384;

__device__ __forceinline__ uint32_t row_pos0(uint32_t r) { return r ^ (((r >> 3) ^ (r >> 6)) & 7u); }

template <typename Key, int kRow>
__device__ __forceinline__ void load_row0(Key (&v)[kRow], const Key* p) {
  const uint4* q = reinterpret_cast<const uint4*>(p);
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const uint4 t = q[c];
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

template <typename Key>
__device__ __forceinline__ Key min0(Key a, Key b) { return b < a ? b : a; }

// One finished entry: gp = F(U) << b, A = split(U).
template <typename Key>
__device__ __forceinline__ void put_tile0(int L, int b, const InnerPerm& perm, uint32_t U, Key gp, uint32_t A,
                                          Key* __restrict__ Gp, Key* __restrict__ Gc,
                                          uint32_t* __restrict__ split_rot, int32_t* __restrict__ flags) {
  const uint32_t idx = perm.stored(U);
  if (MPT_BAD(flags, idx < (1u << b) && valid_split(U << L, A << L))) return;
  Gp[idx] = gp;
  Gc[idx] = gp | (Key)(~U & ((1u << b) - 1u));
  split_rot[idx] = A << L;
}

// b <= 5: one warp, lane = U, level by level in |U|.
template <typename Key, typename Tab>
__global__ void __launch_bounds__(32)
k_dp_tile0_small(int L, int b, InnerPerm perm, const Tab* __restrict__ wIr, Key* __restrict__ Gp,
                 Key* __restrict__ Gc, uint32_t* __restrict__ split_rot, int32_t* __restrict__ flags) {
  __shared__ Key cur[32];
  const uint32_t U = threadIdx.x, mask = (1u << b) - 1u, low = U & (~U + 1u);
  const bool has = U <= mask;
  const Key w = has ? (Key)wIr[U] : (Key)0;
  Key gp = 0;
  uint32_t A = 0;
  for (int p = 0; p <= b; ++p) {
    if (has && __popc(U) == p) {
      if (p == 1) gp = w << b;
      if (p >= 2) {
        Key best = ~(Key)0;
        const uint32_t rest = U ^ low;
        for (uint32_t sub = 0; sub != rest; sub = (sub - rest) & rest) {
          const uint32_t a = low | sub;
          best = min0<Key>(best, cur[a] + cur[U ^ a] + a);  // (value << b) + A
        }
        gp = ((best >> b) - w) << b;
        A = (uint32_t)best & mask;
      }
      cur[U] = gp;
    }
    __syncwarp();
  }
  if (has) put_tile0<Key>(L, b, perm, U, gp, A, Gp, Gc, split_rot, flags);
}

// acc[s2] = min over a2 within s2 holding lowbit(s2) of x[a2] + y[s2 ^ a2], s2 >= 1
template <typename Key, int kRow>
__device__ __forceinline__ void conv_rows_low(Key (&acc)[kRow], const Key (&x)[kRow], const Key (&y)[kRow]) {
#pragma unroll
  for (int a2 = 1; a2 < kRow; ++a2) {
#pragma unroll
    for (int s2 = 1; s2 < kRow; ++s2)
      if ((a2 & s2) == a2 && (a2 & (s2 & -s2)) != 0) acc[s2] = min0<Key>(acc[s2], x[a2] + y[s2 ^ a2]);
  }
}

// b >= 6, row-blocked: U = (s1, s2), rows s1 of kRow entries, level by level
// in |s1|.  A split of U names its part A = (a1, a2) holding lowbit(U):
//   * s2 != 0: a2 holds lowbit(s2), any a1 within s1; a1 not in {0, s1}: rows
//     of earlier levels, a register convolution of two rows (phase A); a1 = 0
//     and a1 = s1: the in-row recurrence, in increasing s2, in registers
//     (phase B, one thread per row);
//   * s2 = 0: a1 holds lowbit(s1), the entry-0 column of the same row pairs.
// cur holds F << b; the key of A | B is cur[A] + cur[B] + A = (value << b) + A.
// One block is all there is to run, so its chains bound it: phase A spreads a
// row's 2^p1 - 2 row pairs over as many lanes as the block has for it (at
// most 2^(p1 - 1) and a warp), and the minima of a row then reduce by
// shuffles.  m = 12, 32-bit keys: 275 us with one subset per lane group and a
// block barrier per size of U (a lane per few submasks, each two dependent
// shared loads), 34 us in this form (64-bit keys: 49 us).
template <typename Key, typename Tab>
__global__ void __launch_bounds__(kT0Threads)
k_dp_tile0(int L, int b, InnerPerm perm, const Tab* __restrict__ wIr, Key* __restrict__ Gp, Key* __restrict__ Gc,
           uint32_t* __restrict__ split_rot, int32_t* __restrict__ flags) {
  using C = Tile0Cfg<Key>;
  constexpr int kRB = C::kRB, kRow = C::kRow;
  constexpr Key kNone = ~(Key)0;
  extern __shared__ __align__(16) unsigned char t0sm[];
  Key* cur = reinterpret_cast<Key*>(t0sm);
  Key* ws = cur + C::kRows * C::kStride;    // w(I), then split
  Key* amin = ws + C::kRows * (kRow + 1);   // phase A minima of a level's rows
  const int t = threadIdx.x, nb = b - kRB;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // k_dp_pruned's first layer gets ready meanwhile
  const uint32_t mask = (1u << b) - 1u;
  for (uint32_t v = t; v <= mask; v += kT0Threads) {
    const uint32_t U = perm.nat(v);
    ws[U + (U >> kRB)] = (Key)wIr[v];
  }
  __syncthreads();
  // level 0: row 0, the recurrence on the lowest inner requests
  if (t == 0) {
    Key c[kRow];
#pragma unroll
    for (int s2 = 0; s2 < kRow; ++s2) {
      Key f = 0;
      uint32_t A = 0;
      if ((s2 & (s2 - 1)) == 0) {
        f = s2 ? ws[s2] : (Key)0;
      } else {
        Key key = kNone;
#pragma unroll
        for (int a2 = 1; a2 < kRow; ++a2)
          if ((a2 & s2) == a2 && (a2 & (s2 & -s2)) != 0 && a2 != s2)
            key = min0<Key>(key, c[a2] + c[s2 ^ a2] + (Key)a2);
        f = (key >> b) - ws[s2];
        A = (uint32_t)key & mask;
      }
      c[s2] = f << b;
      ws[s2] = A;
    }
#pragma unroll
    for (int i = 0; i < kRow; ++i) cur[i] = c[i];  // row 0 is at position 0
  }
  __syncthreads();
  for (int p1 = 1; p1 <= nb; ++p1) {
    const int rows = (int)c_binom.v[nb][p1];
    if (p1 >= 2) {
      int g = p1 - 1 < 5 ? p1 - 1 : 5;  // log2(lanes per row)
      while ((rows << g) > kT0Threads) --g;
      const int G = 1 << g;
      const int ri = t >> g;
      const uint32_t r = (uint32_t)t & (uint32_t)(G - 1);
      Key acc[kRow];
#pragma unroll
      for (int i = 0; i < kRow; ++i) acc[i] = kNone;
      if (ri < rows) {
        const uint32_t s1 = colex_unrank((unsigned long long)ri, p1, nb);
        const uint32_t lowb = s1 & (~s1 + 1u);
        uint32_t hi = 0, rr = s1;
        for (int q = 0; q < g; ++q) {
          const uint32_t top = 1u << (31 - __clz(rr));
          hi |= top;
          rr ^= top;
        }
        const uint32_t freem = s1 ^ hi;
        const uint32_t fixed = deposit_bits(r, hi);
        uint32_t sub = 0;
        do {
          const uint32_t a1 = fixed | sub;
          if (a1 != 0 && a1 != s1) {
            Key x[kRow], y[kRow];
            load_row0<Key, kRow>(x, cur + row_pos0(a1) * C::kStride);
            load_row0<Key, kRow>(y, cur + row_pos0(s1 ^ a1) * C::kStride);
#pragma unroll
            for (int i = 0; i < kRow; ++i) x[i] += (Key)((a1 << kRB) | (uint32_t)i);
            conv_rows_low<Key, kRow>(acc, x, y);
            if (a1 & lowb) acc[0] = min0<Key>(acc[0], x[0] + y[0]);
          }
          sub = (sub - freem) & freem;
        } while (sub != 0);
      }
      for (int off = G >> 1; off > 0; off >>= 1) {
#pragma unroll
        for (int i = 0; i < kRow; ++i) acc[i] = min0<Key>(acc[i], __shfl_xor_sync(0xFFFFFFFFu, acc[i], off));
      }
      if (ri < rows && r == 0) {
#pragma unroll
        for (int i = 0; i < kRow; ++i) amin[ri * (kRow + 1) + i] = acc[i];
      }
      __syncthreads();
    }
    if (t < rows) {
      const uint32_t s1 = colex_unrank((unsigned long long)t, p1, nb), S1 = s1 << kRB;
      Key* own = ws + s1 * (kRow + 1);
      Key z[kRow], c[kRow];
      load_row0<Key, kRow>(z, cur);
#pragma unroll
      for (int s2 = 0; s2 < kRow; ++s2) {
        const Key w = own[s2];
        Key f = w;
        uint32_t A = 0;
        if (!(s2 == 0 && p1 == 1)) {  // else U = (s1, 0) is a single request
          // two independent minima (a1 = 0 and a1 = s1) shorten the chains
          Key k0 = p1 >= 2 ? amin[t * (kRow + 1) + s2] : kNone, k1 = kNone;
#pragma unroll
          for (int a2 = 1; a2 < kRow; ++a2) {
            if ((a2 & s2) == a2 && (a2 & (s2 & -s2)) != 0) {
              k0 = min0<Key>(k0, z[a2] + c[s2 ^ a2] + (Key)a2);
              if (a2 != s2) k1 = min0<Key>(k1, c[a2] + z[s2 ^ a2] + (Key)(S1 | (uint32_t)a2));
            }
          }
          const Key key = min0<Key>(k0, k1);
          f = (key >> b) - w;
          A = (uint32_t)key & mask;
        }
        c[s2] = f << b;
        own[s2] = A;
      }
      Key* dst = cur + row_pos0(s1) * C::kStride;
#pragma unroll
      for (int i = 0; i < kRow; ++i) dst[i] = c[i];
    }
    __syncthreads();
  }
  for (uint32_t U = t; U <= mask; U += kT0Threads)
    put_tile0<Key>(L, b, perm, U, cur[row_pos0(U >> kRB) * C::kStride + (U & (kRow - 1))],
                   (uint32_t)ws[U + (U >> kRB)], Gp, Gc, split_rot, flags);
}

template <typename Key, typename Tab>
cudaError_t tile0(const Shape& s, const Workspace& ws, const Tab* wIr, Key* Gp, Key* Gc, cudaStream_t stream) {
  if (s.b <= 5) {
    k_dp_tile0_small<<<1, 32, 0, stream>>>(s.L, s.b, s.perm, wIr, Gp, Gc, ws.split_rot, ws.counters + 1);
    return cudaGetLastError();
  }
  auto k = k_dp_tile0<Key, Tab>;
  const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, Tile0Cfg<Key>::kSmem);
  if (e != cudaSuccess) return e;
  k<<<1, kT0Threads, Tile0Cfg<Key>::kSmem, stream>>>(s.L, s.b, s.perm, wIr, Gp, Gc, ws.split_rot, ws.counters + 1);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_tile0(const Shape& s, const Workspace& ws, cudaStream_t stream) {
  if (s.wide)
    return s.lean ? tile0(s, ws, ws.fw_rot, ws.Gp64, ws.Gc64, stream) : tile0(s, ws, ws.wI_rot, ws.Gp64, ws.Gc64, stream);
  return s.lean ? tile0(s, ws, ws.fw_rot, ws.Gp, ws.Gc, stream) : tile0(s, ws, ws.wI_rot, ws.Gp, ws.Gc, stream);
}

}  // namespace mpt
