// C ABI of the batched small-instance solver (include/mpt.h, mpt_batch_*):
// argument checks, workspace carve-up and one grid per instance size m, the
// grids on side streams forked from the caller's stream.
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <memory>
#include <new>
#include <string>
#include <thread>
#include <vector>

#include "../../include/mpt.h"
#include "mpt_internal.cuh"

namespace mpt {
size_t batch_smem_bytes(int max_m, int occ_cap);
size_t batch_rows_smem_bytes(int m, int occ_cap);
size_t batch_rows_scratch_words(int m);
cudaError_t launch_batch(int count, int m, int occ_cap, const int64_t* weights, const int64_t* inst_req,
                         const int64_t* req_off, const int32_t* chunks, const int64_t* tab_off,
                         const int32_t* inst_list, const uint8_t* flags, int64_t* opt, int64_t* F,
                         uint32_t* split, int32_t* perm, int32_t* dfs, int32_t* status, cudaStream_t stream);
cudaError_t launch_batch_rows(int count, int m, int occ_cap, const int64_t* weights, const int64_t* inst_req,
                              const int64_t* req_off, const int32_t* chunks, const int64_t* tab_off,
                              const int32_t* inst_list, const uint8_t* flags, int64_t* opt, int64_t* F,
                              uint32_t* split, int32_t* perm, int32_t* dfs, int32_t* status, uint32_t* rows_scratch,
                              cudaStream_t stream);
int batch_members_cap(int m, int occ_cap);
cudaError_t launch_batch_members(int count, int m, int occ_cap, const int64_t* weights, const int64_t* inst_req,
                                 const int64_t* req_off, const int32_t* chunks, const int64_t* tab_off,
                                 const int32_t* inst_list, const uint8_t* flags, int64_t* opt, int64_t* F,
                                 uint32_t* split, int32_t* perm, int32_t* dfs, int32_t* status,
                                 uint32_t* rows_scratch, cudaStream_t stream);
}  // namespace mpt

struct mpt_batch {
  int32_t batch = 0;
  int64_t n = 0, requests = 0, occurrences = 0, table_entries = 0;
  int max_m = 0, occ_cap = 1;
  std::vector<int64_t> w, inst_req, req_off, tab_off;
  // chunk ids fit 32 bits (n < 2^31); not initialised, written by mpt_batch_create's threads
  std::unique_ptr<int32_t[]> chunks;
  // instances grouped by size m: inst_list[group_start[m] .. group_start[m+1]),
  // those for the kernel over the members (m >= 14, packed keys, few members)
  // first, up to group_members_end[m], then those for the row-blocked kernel
  // (m >= 6, packed keys), up to group_rows_end[m]; each part with its own
  // occurrence cap
  std::vector<int32_t> inst_list;
  std::vector<int64_t> group_start, group_members_end, group_rows_end;
  std::vector<int> group_occ_cap_members, group_occ_cap_rows, group_occ_cap;
  // per instance: kFlagPacked when the shared weight is below 2^(32 - m)
  // (32-bit keys), kFlagOffsets when sum_i w(R_i) is not (private and
  // universal chunks kept out of the kernels' values, k_batch.cu)
  std::vector<uint8_t> flags;
  // results of the last solve
  bool solved = false;
  std::vector<int64_t> opt;
  std::unique_ptr<int32_t[]> perm;
  std::vector<int32_t> dfs, status;
  const int64_t* d_F = nullptr;
  const uint32_t* d_split = nullptr;
  void* own_ws = nullptr;
  size_t own_bytes = 0;
  // side streams for the per-size launches (created on first use, on the
  // device current then), with the events that fork them from and join them
  // to the caller's stream
  int side_device = -1;
  std::vector<cudaStream_t> side;
  std::vector<cudaEvent_t> join;
  cudaEvent_t fork = nullptr;
};

namespace {

constexpr int kBatchMaxM = 16;  // m = 16: packed keys only (the row-blocked kernel)
constexpr size_t kBatchMaxSmem = 227 * 1024;  // shared memory of one block
constexpr int kBatchSideStreams = 4;

// Destroys the side streams and events on the device they were made on,
// restoring the caller's current device.
void release_side_streams(mpt_batch* b) {
  int cur = -1;
  const bool switch_dev = b->side_device >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != b->side_device &&
                          cudaSetDevice(b->side_device) == cudaSuccess;
  for (cudaStream_t st : b->side) cudaStreamDestroy(st);
  for (cudaEvent_t ev : b->join) cudaEventDestroy(ev);
  if (b->fork) cudaEventDestroy(b->fork);
  if (switch_dev) cudaSetDevice(cur);
  b->side.clear();
  b->join.clear();
  b->fork = nullptr;
  b->side_device = -1;
}

// The side streams of the current device, created on first use; false when
// they cannot be made (the launches then stay on the caller's stream).
bool side_streams(mpt_batch* b) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  if (b->side_device == dev) return true;
  release_side_streams(b);
  if (cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming) != cudaSuccess) {
    b->fork = nullptr;
    return false;
  }
  for (int i = 0; i < kBatchSideStreams; ++i) {
    cudaStream_t st = nullptr;
    cudaEvent_t ev = nullptr;
    if (cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking) != cudaSuccess) break;
    if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) {
      cudaStreamDestroy(st);
      break;
    }
    b->side.push_back(st);
    b->join.push_back(ev);
  }
  if ((int)b->side.size() < kBatchSideStreams) {
    release_side_streams(b);
    cudaGetLastError();
    return false;
  }
  b->side_device = dev;
  return true;
}
constexpr int kBatchMaxOcc = 2048;
constexpr int64_t kBatchSumLimit = (int64_t)1 << 62;

// One instance: its chunk ids (in range, no repeat inside a request), its
// flags, and whether its kernel can hold it.  Distinct chunks are counted in a
// small open-addressing table (at most 2 x 2048 slots, so it stays in the
// first-level cache) whose slots carry the instance's number, so that it is
// never cleared.  Sorting every request and the whole instance instead took
// 43 of the 45 ms of a pass over 20,000 groups of 8-13 requests.
struct ChunkSlot {
  int64_t inst = -1;  // the instance that filled the slot
  int32_t chunk = 0;
  uint16_t mask = 0, count = 0;  // the instance's requests that hold the chunk, and their number
};

// Members of an instance (k_batch.cu: requests that share a chunk which not
// all share), at most, from the sets of requests that share one; 0 where
// k_batch_rows is the faster kernel or the smaller ones have no other.  Pairs
// are counted as they are, larger members once for every set that holds them.
// The line is on the tests of the lists, sum over the members A of
// 2^(m - 1 - lowest(A)), against the 3^m that the row form's splits are half of:
// it lies where the heaviest of some hundred instances, two to an SM, takes what
// the rows take.  m = 14, 300 groups of 8 passages out of 100, 60, 50 and 40 each
// (tests 0.044, 0.07, 0.11 and 0.22 of 3^m): rows 0.24 ms, members 0.18, 0.23, 0.31 and
// 0.37; m = 15 (0.03, 0.06, 0.10, 0.15): 0.54 and 0.28, 0.36, 0.53, 0.90; m = 16 (0.02,
// 0.05, 0.08, 0.12, 0.26, the heaviest of them twice that): 3.8 and 0.42, 0.64, 1.0,
// 1.8, 2.1, where one group of the rows' alone takes 1.7.
constexpr int kMembersFromM = 14;

// A set's larger members by its bytes, so that the loop has no branch on its
// bits: request i of a byte with a_i requests above it in the byte, and c in the
// byte above, is the lowest of 2^(a_i + c) - 1 - (a_i + c) of them, 2^(7 - i) tests
// each in units of the byte.  (0.4 us an instance bit by bit, of 1.9 us that
// mpt_batch_create takes for one of 15 requests of 8 chunks.)
struct ByteSums {
  uint32_t power[256] = {};  // sum of 2^a_i 2^(7 - i)
  uint16_t more[256] = {};   // sum of (1 + a_i) 2^(7 - i)
  uint8_t units[256] = {};   // sum of 2^(7 - i)
  uint8_t bits[256] = {};
};
constexpr ByteSums make_byte_sums() {
  ByteSums t{};
  for (int v = 0; v < 256; ++v)
    for (int i = 7; i >= 0; --i)
      if (v >> i & 1) {
        t.power[v] += (1u << t.bits[v]) << (7 - i);
        t.more[v] = (uint16_t)(t.more[v] + ((1 + t.bits[v]) << (7 - i)));
        t.units[v] = (uint8_t)(t.units[v] + (1 << (7 - i)));
        ++t.bits[v];
      }
  return t;
}

int members_bound(int m, const uint16_t* sets, int n) {
  static constexpr ByteSums kByte = make_byte_sums();
  static constexpr uint64_t kLine[3] = {10, 8, 2};
  uint16_t pairs[16] = {};
  uint16_t seen[32] = {};  // sets, by a hash: one met again is mostly left out
  uint64_t tests = 0, splits = 1, members = 0;
  for (int k = 0; k < n; ++k) {
    const uint32_t N = sets[k], lo = N & 255u, hi = N >> 8;
    for (int l = 0; l < 16; ++l) pairs[l] = (uint16_t)(pairs[l] | ((N & (1u << l)) != 0 ? N : 0u));
    uint16_t& slot = seen[N * 0x9E37u >> 8 & 31u];
    const uint64_t once = slot != N;
    slot = (uint16_t)N;
    const uint64_t c = kByte.bits[hi], size = c + kByte.bits[lo];
    tests += once * (256 * (((uint64_t)kByte.power[lo] << c) - kByte.more[lo] - c * kByte.units[lo]) +
                     kByte.power[hi] - kByte.more[hi]);
    members += once * (((uint64_t)1 << size) - 1 - size - size * (size - 1) / 2);
  }
  for (int l = 0; l < m; ++l) {
    const uint32_t above = (uint32_t)pairs[l] >> l >> 1;
    const uint64_t own = 1 + kByte.bits[above & 255u] + kByte.bits[above >> 8];  // the single request and the pairs
    tests += own << (15 - l);
    members += own;
    splits *= 3;
  }
  return (tests >> (16 - m)) * kLine[m - kMembersFromM] < splits && members < 1 << 30 ? (int)members : 0;
}

mpt_status check_instance(const int64_t* weights, int64_t n_chunks, int64_t b, int64_t r0, int64_t r1,
                          const int64_t* req_offsets, const int64_t* chunk_ids, ChunkSlot* table,
                          int32_t* ids32, uint8_t* flags, int32_t* members) {
  const int m = (int)(r1 - r0);
  const int64_t occ = req_offsets[r1] - req_offsets[r0];
  if (occ > kBatchMaxOcc) return MPT_ERR_TOO_LARGE;
  int lg = 4;
  while (((int64_t)1 << lg) < 2 * occ) ++lg;
  const uint32_t mask = (1u << lg) - 1u;
  uint16_t used[kBatchMaxOcc];
  int distinct = 0;
  for (int64_t r = r0; r < r1; ++r) {
    for (int64_t j = req_offsets[r]; j < req_offsets[r + 1]; ++j) {
      const int64_t x = chunk_ids[j];
      if (x < 0 || x >= n_chunks) return MPT_ERR_INVALID_ARG;
      ids32[j] = (int32_t)x;
      uint32_t h = ((uint32_t)x * 2654435761u) >> (32 - lg);
      while (table[h].inst == b && table[h].chunk != (int32_t)x) h = (h + 1u) & mask;
      ChunkSlot& e = table[h];
      if (e.inst != b) {
        e.inst = b;
        e.chunk = (int32_t)x;
        e.mask = e.count = 0;
        used[distinct++] = (uint16_t)h;
      } else if (e.mask >> (r - r0) & 1u) {
        return MPT_ERR_INVALID_ARG;  // twice in one request
      }
      e.mask = (uint16_t)(e.mask | 1u << (r - r0));
      ++e.count;
    }
  }
  // sum_i w(R_i) (below 2^62) and the shared weight W (below 2^31): the
  // request weight less the chunks that one or all m >= 2 requests hold,
  // which the kernels keep out of their 32-bit values (k_batch.cu)
  int64_t sum = 0, shared = 0;
  uint16_t sets[kBatchMaxOcc / 2];
  int n_sets = 0;
  for (int k = 0; k < distinct; ++k) {
    const ChunkSlot& e = table[used[k]];
    const int64_t cnt = e.count, wx = weights[e.chunk];
    if (wx > (kBatchSumLimit - 1 - sum) / cnt) return MPT_ERR_OVERFLOW;
    sum += cnt * wx;
    if (cnt >= 2 && cnt < m) {
      shared += cnt * wx;
      if (shared >= ((int64_t)1 << 31)) return MPT_ERR_OVERFLOW;
      if (m >= kMembersFromM) sets[n_sets++] = e.mask;  // two occurrences or more each
    }
  }
  *flags = (uint8_t)((shared < ((int64_t)1 << (32 - m)) ? mpt::kFlagPacked : 0) |
                     (sum >= ((int64_t)1 << (32 - m)) ? mpt::kFlagOffsets : 0));
  // the instance's kernel must hold its shared-memory arrays: the
  // per-subset kernel keeps the 2^m tables there (m = 15: room for 1024
  // occurrences; m = 16 does not fit, so 16 requests need packed keys),
  // the row-blocked kernel its rows up to m = 15
  int cap = 1;
  while (cap < occ) cap <<= 1;
  const bool rows = m >= 6 && (*flags & mpt::kFlagPacked);
  if ((rows ? mpt::batch_rows_smem_bytes(m, cap) : mpt::batch_smem_bytes(m, cap)) > kBatchMaxSmem)
    return MPT_ERR_TOO_LARGE;
  *members = 0;
  if (rows && m >= kMembersFromM) *members = members_bound(m, sets, n_sets);
  return MPT_OK;
}

// Every instance, and its chunk ids as 32-bit numbers; *bad: the status of
// the first one that fails.  Ranges of instances run on up to eight threads (one per 2^15
// occurrences); a thread that cannot be started has its range done here.
void check_instances(const int64_t* weights, int64_t n_chunks, int32_t batch, const int64_t* inst_requests,
                     const int64_t* req_offsets, const int64_t* chunk_ids, int32_t* ids32, uint8_t* flags,
                     int32_t* members, mpt_status* bad) {
  const int64_t occ = req_offsets[inst_requests[batch]];
  const int64_t cores = occ >> 15 ? std::max<int64_t>(1, (int64_t)std::thread::hardware_concurrency()) : 1;
  const int64_t ranges = std::min<int64_t>({8, cores, 1 + (occ >> 15), batch});
  int64_t most = 8, slots = 16;  // of the largest instance
  for (int32_t b = 0; b < batch; ++b)
    most = std::max<int64_t>(most, req_offsets[inst_requests[b + 1]] - req_offsets[inst_requests[b]]);
  while (slots < 2 * std::min<int64_t>(most, kBatchMaxOcc)) slots <<= 1;
  struct Range {
    std::vector<ChunkSlot> table;
    mpt_status status = MPT_OK;
  };
  std::vector<Range> out((size_t)ranges);
  for (Range& r : out) r.table.resize((size_t)slots);  // here, so that a thread has nothing that throws
  auto work = [&](int64_t k) {
    Range& r = out[(size_t)k];
    const int32_t end = (int32_t)(batch * (k + 1) / ranges);
    for (int32_t b = (int32_t)(batch * k / ranges); b < end && r.status == MPT_OK; ++b) {
      r.status = check_instance(weights, n_chunks, b, inst_requests[b], inst_requests[b + 1], req_offsets, chunk_ids,
                                r.table.data(), ids32, flags + b, members + b);
    }
  };
  std::vector<std::thread> threads;
  threads.reserve((size_t)ranges);
  for (int64_t k = 1; k < ranges; ++k) {
    try {
      threads.emplace_back(work, k);
    } catch (...) {
      work(k);
    }
  }
  work(0);
  for (std::thread& t : threads) t.join();
  for (const Range& r : out)
    if (r.status != MPT_OK) {
      *bad = r.status;
      return;
    }
}

struct BatchCarve {
  int64_t *weights, *inst_req, *req_off, *tab_off, *opt, *F;
  int32_t *chunks, *perm;
  uint32_t *split, *rows_scratch;
  int32_t *dfs, *status, *inst_list;
  uint8_t* flags;
};

size_t carve(const mpt_batch* b, char* base, BatchCarve* c) {
  size_t off = 0;
  auto take = [&](size_t bytes) -> char* {
    const size_t o = off;
    off += (bytes + 255) & ~(size_t)255;
    return base ? base + o : nullptr;
  };
  c->weights = reinterpret_cast<int64_t*>(take((size_t)b->n * 8));
  c->inst_req = reinterpret_cast<int64_t*>(take(((size_t)b->batch + 1) * 8));
  c->req_off = reinterpret_cast<int64_t*>(take(((size_t)b->requests + 1) * 8));
  c->chunks = reinterpret_cast<int32_t*>(take((size_t)std::max<int64_t>(b->occurrences, 1) * 4));
  c->tab_off = reinterpret_cast<int64_t*>(take(((size_t)b->batch + 1) * 8));
  c->opt = reinterpret_cast<int64_t*>(take((size_t)b->batch * 8));
  c->F = reinterpret_cast<int64_t*>(take((size_t)b->table_entries * 8));
  c->split = reinterpret_cast<uint32_t*>(take((size_t)b->table_entries * 4));
  c->perm = reinterpret_cast<int32_t*>(take((size_t)std::max<int64_t>(b->occurrences, 1) * 4));
  c->dfs = reinterpret_cast<int32_t*>(take((size_t)b->requests * 4));
  c->status = reinterpret_cast<int32_t*>(take((size_t)b->batch * 4));
  c->inst_list = reinterpret_cast<int32_t*>(take((size_t)b->batch * 4));
  c->flags = reinterpret_cast<uint8_t*>(take((size_t)b->batch));
  // rows of the row-blocked instances too large for shared memory, one slot
  // per block of their size's launch
  size_t scratch_words = 0;
  if (!b->group_rows_end.empty())
    for (int m = 1; m <= kBatchMaxM; ++m)
      scratch_words = std::max(scratch_words, (size_t)(b->group_rows_end[(size_t)m] - b->group_start[(size_t)m]) *
                                                  mpt::batch_rows_scratch_words(m));
  c->rows_scratch = scratch_words ? reinterpret_cast<uint32_t*>(take(scratch_words * 4)) : nullptr;
  return off;
}

}  // namespace

extern "C" {

mpt_status mpt_batch_create(const int64_t* weights, int64_t n_chunks, int32_t batch, const int64_t* inst_requests,
                            const int64_t* req_offsets, const int64_t* chunk_ids, mpt_batch** out) {
  if (!weights || !inst_requests || !req_offsets || !out || n_chunks < 1 || n_chunks > INT32_MAX || batch < 1)
    return MPT_ERR_INVALID_ARG;
  if (inst_requests[0] != 0) return MPT_ERR_INVALID_ARG;
  for (int32_t b = 0; b < batch; ++b) {
    const int64_t m = inst_requests[b + 1] - inst_requests[b];
    if (m < 1) return MPT_ERR_INVALID_ARG;
    if (m > kBatchMaxM) return MPT_ERR_TOO_LARGE;
  }
  const int64_t R = inst_requests[batch];
  if (req_offsets[0] != 0) return MPT_ERR_INVALID_ARG;
  for (int64_t r = 0; r < R; ++r)
    if (req_offsets[r + 1] < req_offsets[r]) return MPT_ERR_INVALID_ARG;
  const int64_t occ_total = req_offsets[R];
  if (occ_total > 0 && !chunk_ids) return MPT_ERR_INVALID_ARG;
  for (int64_t x = 0; x < n_chunks; ++x)
    if (weights[x] <= 0) return MPT_ERR_INVALID_ARG;
  mpt_batch* c = new (std::nothrow) mpt_batch();
  if (!c) return MPT_ERR_OUT_OF_MEMORY;
  try {
    c->tab_off.resize((size_t)batch + 1);
    c->flags.assign((size_t)batch, 0);
    std::vector<int> inst_occ((size_t)batch);
    std::vector<int32_t> members((size_t)batch);
    // the instances' own checks and weights, on several threads when there
    // are many occurrences; the first failing instance decides the status
    mpt_status bad = MPT_OK;
    c->chunks.reset(new int32_t[(size_t)std::max<int64_t>(occ_total, 1)]);
    check_instances(weights, n_chunks, batch, inst_requests, req_offsets, chunk_ids, c->chunks.get(),
                    c->flags.data(), members.data(), &bad);
    if (bad != MPT_OK) {
      delete c;
      return bad;
    }
    int64_t tab = 0;
    for (int32_t b = 0; b < batch; ++b) {
      const int64_t r0 = inst_requests[b], r1 = inst_requests[b + 1];
      const int m = (int)(r1 - r0);
      const int64_t occ = req_offsets[r1] - req_offsets[r0];
      c->tab_off[(size_t)b] = tab;
      tab += (int64_t)1 << m;
      c->max_m = std::max(c->max_m, m);
      while (c->occ_cap < occ) c->occ_cap <<= 1;
      inst_occ[(size_t)b] = (int)occ;
    }
    c->tab_off[(size_t)batch] = tab;
    // group the instances by m (stable), each group with its own occurrence cap
    c->group_start.assign(kBatchMaxM + 2, 0);
    for (int32_t b = 0; b < batch; ++b) ++c->group_start[(size_t)(inst_requests[b + 1] - inst_requests[b]) + 1];
    for (int m = 1; m <= kBatchMaxM + 1; ++m) c->group_start[(size_t)m] += c->group_start[(size_t)m - 1];
    c->inst_list.resize((size_t)batch);
    c->group_occ_cap_members.assign(kBatchMaxM + 1, 1);
    c->group_occ_cap_rows.assign(kBatchMaxM + 1, 1);
    c->group_occ_cap.assign(kBatchMaxM + 1, 1);
    // the members have to fit beside the most occurrences of their part
    int room[kBatchMaxM + 1] = {};
    for (int32_t b = 0; b < batch; ++b) {
      if (members[(size_t)b] == 0) continue;
      const int m = (int)(inst_requests[b + 1] - inst_requests[b]);
      int& most = c->group_occ_cap_members[(size_t)m];
      int cap = most;
      while (cap < inst_occ[(size_t)b]) cap <<= 1;
      if (cap != most || room[m] == 0) {
        const int fits = mpt::batch_members_cap(m, cap);
        if (fits == 0) {
          members[(size_t)b] = 0;
          continue;
        }
        most = cap;
        room[m] = fits;
      }
    }
    // where each part of a size starts, then its instances in order
    std::vector<uint8_t> part((size_t)batch);
    int64_t count[kBatchMaxM + 1][3] = {};
    for (int32_t b = 0; b < batch; ++b) {
      const int m = (int)(inst_requests[b + 1] - inst_requests[b]), k = members[(size_t)b];
      const int p = k > 0 && k <= room[m] ? 0 : m >= 6 && (c->flags[(size_t)b] & mpt::kFlagPacked) ? 1 : 2;
      part[(size_t)b] = (uint8_t)p;
      ++count[m][p];
      if (p == 0) continue;
      int& cap = p == 1 ? c->group_occ_cap_rows[(size_t)m] : c->group_occ_cap[(size_t)m];
      while (cap < inst_occ[(size_t)b]) cap <<= 1;
    }
    c->group_members_end = c->group_rows_end = c->group_start;
    int64_t fill[kBatchMaxM + 1][3];
    for (int m = 0; m <= kBatchMaxM; ++m) {
      fill[m][0] = c->group_start[(size_t)m];
      fill[m][1] = c->group_members_end[(size_t)m] = fill[m][0] + count[m][0];
      fill[m][2] = c->group_rows_end[(size_t)m] = fill[m][1] + count[m][1];
    }
    for (int32_t b = 0; b < batch; ++b)
      c->inst_list[(size_t)fill[inst_requests[b + 1] - inst_requests[b]][part[(size_t)b]]++] = b;
    c->table_entries = tab;
    c->w.assign(weights, weights + n_chunks);
    c->inst_req.assign(inst_requests, inst_requests + batch + 1);
    c->req_off.assign(req_offsets, req_offsets + R + 1);
  } catch (...) {
    delete c;
    return MPT_ERR_OUT_OF_MEMORY;
  }
  c->batch = batch;
  c->n = n_chunks;
  c->requests = R;
  c->occurrences = occ_total;
  *out = c;
  return MPT_OK;
}

mpt_status mpt_batch_workspace_bytes(const mpt_batch* b, size_t* bytes) {
  if (!b || !bytes) return MPT_ERR_INVALID_ARG;
  BatchCarve c{};
  *bytes = carve(b, nullptr, &c);
  return MPT_OK;
}

mpt_status mpt_batch_solve(mpt_batch* b, void* d_workspace, size_t workspace_bytes, void* stream_ptr) {
  if (!b) return MPT_ERR_INVALID_ARG;
  cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_ptr);
  b->solved = false;
  BatchCarve c{};
  const size_t need = carve(b, nullptr, &c);
  char* base = nullptr;
  if (d_workspace) {
    if (workspace_bytes < need) return MPT_ERR_WORKSPACE_TOO_SMALL;
    if (reinterpret_cast<uintptr_t>(d_workspace) & 255) return MPT_ERR_INVALID_ARG;
    base = static_cast<char*>(d_workspace);
  } else {
    if (b->own_bytes < need) {
      if (b->own_ws) cudaFree(b->own_ws);
      b->own_ws = nullptr;
      b->own_bytes = 0;
      if (mpt::device_alloc(&b->own_ws, need) != cudaSuccess) return MPT_ERR_OUT_OF_MEMORY;
      b->own_bytes = need;
    }
    base = static_cast<char*>(b->own_ws);
  }
  carve(b, base, &c);
  const size_t B = (size_t)b->batch;
  try {
    b->opt.resize(B);
    b->status.resize(B);
    if (!b->perm) b->perm.reset(new int32_t[(size_t)std::max<int64_t>(b->occurrences, 1)]);
    b->dfs.resize((size_t)b->requests);
  } catch (...) {
    return MPT_ERR_OUT_OF_MEMORY;
  }
  cudaError_t e = cudaSuccess;
  auto h2d = [&](void* d, const void* h, size_t bytes) {
    if (e == cudaSuccess && bytes) e = cudaMemcpyAsync(d, h, bytes, cudaMemcpyHostToDevice, stream);
  };
  auto d2h = [&](void* h, const void* d, size_t bytes) {
    if (e == cudaSuccess && bytes) e = cudaMemcpyAsync(h, d, bytes, cudaMemcpyDeviceToHost, stream);
  };
  h2d(c.weights, b->w.data(), (size_t)b->n * 8);
  h2d(c.inst_req, b->inst_req.data(), (B + 1) * 8);
  h2d(c.req_off, b->req_off.data(), ((size_t)b->requests + 1) * 8);
  h2d(c.chunks, b->chunks.get(), (size_t)b->occurrences * 4);
  h2d(c.tab_off, b->tab_off.data(), (B + 1) * 8);
  h2d(c.inst_list, b->inst_list.data(), B * 4);
  h2d(c.flags, b->flags.data(), B);
  // One grid per instance size, largest first.  The grids write disjoint
  // instances, so they run on side streams forked from the caller's stream
  // after the uploads and joined back before the downloads: the short grids
  // of small sizes then fill the SMs that the long ones leave idle.
  const bool forked = e == cudaSuccess && side_streams(b);
  if (forked) {
    e = cudaEventRecord(b->fork, stream);
    for (int i = 0; i < kBatchSideStreams && e == cudaSuccess; ++i) e = cudaStreamWaitEvent(b->side[(size_t)i], b->fork, 0);
  }
  int next_side = 0;
  for (int m = kBatchMaxM; m >= 1 && e == cudaSuccess; --m) {
    const int64_t g0 = b->group_start[(size_t)m], gm = b->group_members_end[(size_t)m],
                  gr = b->group_rows_end[(size_t)m], g1 = b->group_start[(size_t)m + 1];
    if (g1 == g0) continue;
    auto side = [&]() { return forked ? b->side[(size_t)(next_side++ % kBatchSideStreams)] : stream; };
    // the parts of a size run at the same time: each block has its own slot of the scratch rows
    uint32_t* after = c.rows_scratch ? c.rows_scratch + (size_t)(gm - g0) * mpt::batch_rows_scratch_words(m) : nullptr;
    cudaStream_t st = side();
    if (gr > gm)
      e = mpt::launch_batch_rows((int)(gr - gm), m, b->group_occ_cap_rows[(size_t)m], c.weights, c.inst_req, c.req_off,
                                 c.chunks, c.tab_off, c.inst_list + gm, c.flags, c.opt, c.F, c.split, c.perm, c.dfs,
                                 c.status, after, st);
    if (e == cudaSuccess && gm > g0)
      e = mpt::launch_batch_members((int)(gm - g0), m, b->group_occ_cap_members[(size_t)m], c.weights, c.inst_req,
                                    c.req_off, c.chunks, c.tab_off, c.inst_list + g0, c.flags, c.opt, c.F, c.split,
                                    c.perm, c.dfs, c.status, c.rows_scratch, gr > gm ? side() : st);
    if (e == cudaSuccess && g1 > gr)
      e = mpt::launch_batch((int)(g1 - gr), m, b->group_occ_cap[(size_t)m], c.weights, c.inst_req, c.req_off,
                            c.chunks, c.tab_off, c.inst_list + gr, c.flags, c.opt, c.F, c.split, c.perm, c.dfs,
                            c.status, st);
  }
  if (forked) {
    // join every side stream, also after a failed launch, so that no work
    // of this call runs on after it returns
    for (int i = 0; i < kBatchSideStreams; ++i) {
      cudaError_t ej = cudaEventRecord(b->join[(size_t)i], b->side[(size_t)i]);
      if (ej == cudaSuccess) ej = cudaStreamWaitEvent(stream, b->join[(size_t)i], 0);
      if (ej != cudaSuccess) {
        cudaStreamSynchronize(b->side[(size_t)i]);
        if (e == cudaSuccess) e = ej;
      }
    }
  }
  d2h(b->opt.data(), c.opt, B * 8);
  d2h(b->status.data(), c.status, B * 4);
  d2h(b->perm.get(), c.perm, (size_t)b->occurrences * 4);
  d2h(b->dfs.data(), c.dfs, (size_t)b->requests * 4);
  if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? MPT_ERR_OUT_OF_MEMORY : MPT_ERR_CUDA;
  for (size_t i = 0; i < B; ++i)
    if (b->status[i] != 0) return MPT_ERR_INTERNAL;
  b->d_F = c.F;
  b->d_split = c.split;
  b->solved = true;
  return MPT_OK;
}

mpt_status mpt_batch_results(const mpt_batch* b, int64_t* opt, int64_t* perm_chunks, int32_t* dfs_order) {
  if (!b) return MPT_ERR_INVALID_ARG;
  if (!b->solved) return MPT_ERR_NOT_SOLVED;
  if (opt) std::memcpy(opt, b->opt.data(), b->opt.size() * 8);
  if (perm_chunks) std::copy(b->perm.get(), b->perm.get() + b->occurrences, perm_chunks);
  if (dfs_order && !b->dfs.empty()) std::memcpy(dfs_order, b->dfs.data(), b->dfs.size() * 4);
  return MPT_OK;
}

mpt_status mpt_batch_tables(const mpt_batch* b, const int64_t** d_F, const uint32_t** d_split,
                            int64_t* table_offsets) {
  if (!b) return MPT_ERR_INVALID_ARG;
  if (!b->solved) return MPT_ERR_NOT_SOLVED;
  if (d_F) *d_F = b->d_F;
  if (d_split) *d_split = b->d_split;
  if (table_offsets) std::memcpy(table_offsets, b->tab_off.data(), b->tab_off.size() * 8);
  return MPT_OK;
}

void mpt_batch_destroy(mpt_batch* b) {
  if (!b) return;
  if (b->own_ws) cudaFree(b->own_ws);
  release_side_streams(b);
  delete b;
}

}  // extern "C"
