// Natural-order views of the blocked path's tables.
//
// The blocked recurrence (k_dp_blocked.cu) keeps every table in rotated
// order, idx(S) = (T << b) | U with T = S mod 2^L and U = S >> L, so that the
// 2^b subsets of one tile are contiguous.  The natural order S = (U << L) | T
// is the transpose of that 2^L x 2^b matrix; it is produced only when the
// tables themselves are asked for, by a shared-memory tiled transpose (reads
// coalesced along U, writes along T).  The same pass adds back
// the weights that the blocked recurrence leaves out (k_scatter_zeta.cu):
// the private pi_i and the universal u, i.e. sum_{i in S} pi_i + u to F(S)
// for non-empty S, u to every w(I(S)), plus pi_i at S = {i} and sum_i pi_i at
// S = {}, the weight of the union of all requests.
#include "mpt_internal.cuh"

namespace mpt {
namespace {

constexpr int kTileT = 32;  // T values of a block
constexpr int kLanes = 32, kWarpsT = 8;

struct Copy {
  template <typename S>
  __device__ static S apply(S v, int) { return v; }
};
struct GpToF {
  __device__ static uint32_t apply(uint32_t v, int b) { return v >> b; }
};
struct Gp64ToF {
  __device__ static unsigned long long apply(unsigned long long v, int b) { return v >> b; }
};

enum Offset { kNone, kPiOfS, kPiOfSingletons };

// dst[(U << L) | T] = Op(src[(T << b) | U]) + offset(S) for T < 2^L, U < 2^b,
// S = (U << L) | T: offset pi(S) + u for S non-empty (F), or u plus pi_i at
// S = {i} and sum_i pi_i at S = {} (w(I)), or none; priv null means no
// offsets.  info (the pruned recurrence's lists, or null): src is 0, and not
// there to be read, in the tiles T != 0 without a member.
//
// HBM-bound.  A block has 16 loads per thread in flight, after one round of
// loads for what its offsets need; tiles of 32 x 32 with four loads, and the
// offsets summed from global memory, took 1.92 ms for the three tables at
// m = 28 (5.0 TB/s), this form 1.36 ms with w(I) read only where it is not 0.
template <typename Src, typename Dst, typename Op, Offset Off, int kTileU>
__global__ void __launch_bounds__(kLanes * kWarpsT)
k_unrotate(const Src* __restrict__ src, Dst* __restrict__ dst, int L, int b,
           const unsigned long long* __restrict__ priv, int m, InnerPerm perm, const uint32_t* __restrict__ info) {
  __shared__ Dst t[kTileT][kTileU + 1];
  __shared__ long long pi[kUniversalSlot], piT[kTileT], piU[kTileU], pi_all, univ;
  __shared__ uint32_t nat_of[kTileU];  // the stored order of the block's U values undone
  __shared__ uint32_t live;            // the T values whose entries are there to be read
  const size_t nT = (size_t)1 << L, nU = (size_t)1 << b;
  const size_t T0 = (size_t)blockIdx.x * kTileT, U0 = (size_t)blockIdx.y * kTileU;
  const int tx = threadIdx.x, ty = threadIdx.y;
  if (ty == 0) {
    const size_t T = T0 + tx;
    const bool here = T < nT && (!info || T == 0 || info[T] != 0);
    const uint32_t all = __ballot_sync(0xFFFFFFFFu, here);
    if (tx == 0) live = all;
  } else if (ty == 1) {
    if (Off != kNone) pi[tx] = priv && tx < m ? (long long)priv[tx] : 0;
  } else if (ty == 2) {
    if (Off != kNone && tx == 0) univ = priv ? (long long)priv[kUniversalSlot] : 0;
  }
  __syncthreads();
  Src v[kTileT / kWarpsT][kTileU / kLanes];
#pragma unroll
  for (int j = 0; j < kTileT / kWarpsT; ++j) {
    const int row = ty + j * kWarpsT;
    const bool there = (live >> row & 1u) != 0;
#pragma unroll
    for (int q = 0; q < kTileU / kLanes; ++q) {
      const size_t U = U0 + tx + q * kLanes;
      v[j][q] = there && U < nU ? src[((T0 + row) << b) | U] : (Src)0;
    }
  }
  if (ty >= 1 && ty <= kTileU / kLanes) {
    const int u = tx + (ty - 1) * kLanes;
    const uint32_t nat = perm.nat((uint32_t)U0 + u);
    nat_of[u] = nat;
    long long sum = 0;
    if (Off != kNone && U0 + u < nU)
      for (uint32_t r = nat; r; r &= r - 1) sum += pi[L + __ffs(r) - 1];
    piU[u] = sum;
  } else if (Off != kNone && ty == 0) {
    long long sum = 0;
    if (T0 + tx < nT)
      for (uint32_t r = (uint32_t)(T0 + tx); r; r &= r - 1) sum += pi[__ffs(r) - 1];
    piT[tx] = sum;
  } else if (Off != kNone && ty == kWarpsT - 1) {
    long long sum = pi[tx];
    for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, off);
    if (tx == 0) pi_all = sum;
  }
#pragma unroll
  for (int j = 0; j < kTileT / kWarpsT; ++j) {
#pragma unroll
    for (int q = 0; q < kTileU / kLanes; ++q) t[ty + j * kWarpsT][tx + q * kLanes] = (Dst)Op::apply(v[j][q], b);
  }
  __syncthreads();
  const size_t T = T0 + tx;
  if (T >= nT) return;
#pragma unroll 8
  for (int u = ty; u < kTileU; u += kWarpsT) {
    if (U0 + u >= nU) break;
    Dst x = t[tx][u];
    const size_t nat = nat_of[u];
    const uint32_t S = ((uint32_t)nat << L) | (uint32_t)T;
    if (Off == kPiOfS) {
      if (S != 0) x += (Dst)(piT[tx] + piU[u] + univ);
    } else if (Off == kPiOfSingletons) {
      x += (Dst)univ;
      if (S == 0)
        x += (Dst)pi_all;
      else if ((S & (S - 1)) == 0)
        x += (Dst)(T ? piT[tx] : piU[u]);
    }
    dst[(nat << L) | T] = x;
  }
}

template <typename Src, typename Dst, typename Op, Offset Off>
cudaError_t unrotate(const Src* src, Dst* dst, const Shape& s, const unsigned long long* priv, cudaStream_t stream,
                     const uint32_t* info = nullptr) {
  // 128 U values to a block from the first full T tile on; below (m < 17) a
  // launch is a few blocks and bound by one block's chain
  auto run = [&](auto kernel, int tile_u) {
    const dim3 grid((unsigned)((((size_t)1 << s.L) + kTileT - 1) / kTileT),
                    (unsigned)((((size_t)1 << s.b) + tile_u - 1) / tile_u));
    kernel<<<grid, dim3(kLanes, kWarpsT), 0, stream>>>(src, dst, s.L, s.b, priv, s.m, s.perm, info);
  };
  if (s.L < 5)
    run(k_unrotate<Src, Dst, Op, Off, 32>, 32);
  else
    run(k_unrotate<Src, Dst, Op, Off, 128>, 128);
  return cudaGetLastError();
}

}  // namespace

cudaError_t unrotate_tables(const Shape& s, const uint32_t* split_rot, uint32_t* split_nat, const int64_t* wI_rot,
                            int64_t* wI_nat, const uint32_t* Gp, int64_t* F_nat, int32_t* F32_nat,
                            const unsigned long long* priv, cudaStream_t stream, const uint32_t* info) {
  cudaError_t e = cudaSuccess;
  if (split_nat && (e = unrotate<uint32_t, uint32_t, Copy, kNone>(split_rot, split_nat, s, nullptr, stream)) !=
                       cudaSuccess)
    return e;
  if (wI_nat && (e = unrotate<int64_t, int64_t, Copy, kPiOfSingletons>(wI_rot, wI_nat, s, priv, stream, info)) !=
                    cudaSuccess)
    return e;
  if (F_nat && (e = unrotate<uint32_t, int64_t, GpToF, kPiOfS>(Gp, F_nat, s, priv, stream)) != cudaSuccess) return e;
  if (F32_nat && (e = unrotate<uint32_t, int32_t, GpToF, kPiOfS>(Gp, F32_nat, s, priv, stream)) != cudaSuccess)
    return e;
  return cudaSuccess;
}

cudaError_t unrotate_tables_wide(const Shape& s, const uint32_t* split_rot, uint32_t* split_nat,
                                 const int64_t* wI_rot, int64_t* wI_nat, const unsigned long long* Gp64,
                                 int64_t* F_nat, int32_t* F32_nat, const unsigned long long* priv,
                                 cudaStream_t stream, const uint32_t* info) {
  cudaError_t e = cudaSuccess;
  if (split_nat && (e = unrotate<uint32_t, uint32_t, Copy, kNone>(split_rot, split_nat, s, nullptr, stream)) !=
                       cudaSuccess)
    return e;
  if (wI_nat && (e = unrotate<int64_t, int64_t, Copy, kPiOfSingletons>(wI_rot, wI_nat, s, priv, stream, info)) !=
                    cudaSuccess)
    return e;
  if (F_nat && (e = unrotate<unsigned long long, int64_t, Gp64ToF, kPiOfS>(Gp64, F_nat, s, priv, stream)) !=
                   cudaSuccess)
    return e;
  if (F32_nat && (e = unrotate<unsigned long long, int32_t, Gp64ToF, kPiOfS>(Gp64, F32_nat, s, priv, stream)) !=
                     cudaSuccess)
    return e;
  return cudaSuccess;
}

}  // namespace mpt
