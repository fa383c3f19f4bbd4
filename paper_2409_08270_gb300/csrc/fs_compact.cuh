// Decoupled look-back over block counts (Merrill and Garland 2016), and the
// ordered compaction built on it.
#pragma once

#include "fs_common.cuh"
#include "fs_internal.h"

namespace fs {

constexpr unsigned long long kLbCount = 1ull << 32;   // word holds the block's own count
constexpr unsigned long long kLbPrefix = 2ull << 32;  // word holds the inclusive prefix

// Decoupled look-back by one warp: the sum of the counts of blocks 0 .. vb - 1,
// 32 predecessors at a time (lane l reads block vb - 1 - l).  Sums stop at
// 2^32 - 1, so a list that is too long is seen as such.
__device__ __forceinline__ uint32_t look_back(const unsigned long long* status, uint32_t vb,
                                              unsigned long long* counters, int spin_limit,
                                              int lane) {
  const volatile unsigned long long* vs = status;
  uint32_t excl = 0;
  for (int64_t base = static_cast<int64_t>(vb) - 1; base >= 0; base -= 32) {
    const int64_t q = base - lane;
    unsigned long long word = kLbPrefix;  // before block 0: an empty prefix
    if (q >= 0) {
      word = vs[q];
      int spins = 0;
      while ((word >> 32) == 0ull && spins < spin_limit) {
        __nanosleep(32);
        word = vs[q];
        ++spins;
      }
      if ((word >> 32) == 0ull) {  // gave up: report, count it as an empty prefix
        atomicAdd(&counters[kLookbackTimeout], 1ull);
        word = kLbPrefix;
      }
    }
    const uint32_t pre = __ballot_sync(0xffffffffu, (word & ~0xFFFFFFFFull) == kLbPrefix);
    const int first = pre ? __ffs(pre) - 1 : 31;  // nearest predecessor holding a prefix
    const uint32_t v = lane <= first ? static_cast<uint32_t>(word & 0xFFFFFFFFull) : 0u;
    const uint64_t sum =
        excl + __reduce_add_sync(0xffffffffu, v & 0xFFFFu) +
        (static_cast<uint64_t>(__reduce_add_sync(0xffffffffu, v >> 16)) << 16);
    excl = static_cast<uint32_t>(min(sum, static_cast<uint64_t>(0xFFFFFFFFu)));
    if (pre) break;
  }
  return excl;
}

__device__ __forceinline__ uint32_t add_sat(uint32_t a, uint32_t b) {
  return a + b < a ? 0xFFFFFFFFu : a + b;
}

// The values of positions [p0, p0 + n_pos) (or range_in[0 .. 1), at most n_pos
// of them) that `sel` keeps, in order, to out, and {0, their number} to
// range_out: one launch, where flags, a scan and a scatter took five.  A warp
// takes 512 consecutive positions, 32 per load, all loads in flight; the block's
// place comes from the look-back, blocks taking tickets in launch order.
// sel.value(position) is loaded ahead of sel.keep(value); a value of
// 0xFFFFFFFF is never kept.
constexpr int kCompactItems = 16, kCompactWarps = 8;
constexpr int kCompactTile = 32 * kCompactItems * kCompactWarps;
template <typename Select>
__global__ void __launch_bounds__(32 * kCompactWarps) compact_kernel(
    Select sel, int64_t p0, int64_t n_pos, uint32_t* __restrict__ out,
    unsigned long long* __restrict__ status, uint32_t* __restrict__ ticket,
    int64_t* __restrict__ range_out, unsigned long long* __restrict__ counters, int spin_limit,
    const int64_t* __restrict__ range_in) {
  __shared__ uint32_t s_vb, s_boff, s_cnt[kCompactWarps];
  if (range_in) {
    p0 = range_in[0];
    n_pos = min(n_pos, range_in[1] - range_in[0]);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    const uint32_t t = atomicAdd(ticket, 1u);
    s_vb = gave_up(counters) ? kGaveUpTotal : t;  // the values may be incomplete
  }
  __syncthreads();
  const uint32_t vb = s_vb;
  if (vb == kGaveUpTotal) return;
  const int64_t j0 = static_cast<int64_t>(vb) * kCompactTile + warp * 32 * kCompactItems + lane;
  uint32_t g[kCompactItems], bal[kCompactItems], cnt = 0;
#pragma unroll
  for (int i = 0; i < kCompactItems; ++i)
    g[i] = j0 + 32 * i < n_pos ? sel.value(p0 + j0 + 32 * i) : 0xFFFFFFFFu;
#pragma unroll
  for (int i = 0; i < kCompactItems; ++i) {
    bal[i] = __ballot_sync(0xffffffffu, g[i] != 0xFFFFFFFFu && sel.keep(g[i]));
    cnt += __popc(bal[i]);
  }
  if (lane == 0) s_cnt[warp] = cnt;
  __syncthreads();
  if (warp == 0) {
    uint32_t btot = 0;
    for (int w = 0; w < kCompactWarps; ++w) btot += s_cnt[w];
    if (lane == 0) atomicExch(&status[vb], (vb == 0 ? kLbPrefix : kLbCount) | btot);
    const uint32_t excl = look_back(status, vb, counters, spin_limit, lane);
    if (lane == 0) {
      if (vb > 0) atomicExch(&status[vb], kLbPrefix | (excl + btot));
      s_boff = excl;
      if (vb == gridDim.x - 1) {
        range_out[0] = 0;
        range_out[1] = excl + btot;
      }
    }
  }
  __syncthreads();
  uint32_t o = s_boff;
  for (int w = 0; w < warp; ++w) o += s_cnt[w];
#pragma unroll
  for (int i = 0; i < kCompactItems; ++i) {
    if ((bal[i] >> lane) & 1u) out[o + __popc(bal[i] & ((1u << lane) - 1u))] = g[i];
    o += __popc(bal[i]);
  }
}

// lookback: bin_fused_temp_bytes(n_pos) of scratch.
template <typename Select>
cudaError_t launch_compact(const Select& sel, int64_t p0, int64_t n_pos, uint32_t* out,
                           int64_t* range_out, void* lookback, unsigned long long* counters,
                           cudaStream_t stream, const int64_t* range_in) {
  if (n_pos <= 0) return cudaMemsetAsync(range_out, 0, 2 * sizeof(int64_t), stream);
  const int64_t blocks = (n_pos + kCompactTile - 1) / kCompactTile;
  uint32_t* ticket = static_cast<uint32_t*>(lookback);
  unsigned long long* status = reinterpret_cast<unsigned long long*>(
      static_cast<char*>(lookback) + 256);
  cudaError_t e = cudaMemsetAsync(lookback, 0, 256 + static_cast<size_t>(blocks) * 8, stream);
  if (e != cudaSuccess) return e;
  compact_kernel<<<static_cast<unsigned>(blocks), 32 * kCompactWarps, 0, stream>>>(
      sel, p0, n_pos, out, status, ticket, range_out, counters, kLookbackSpinLimit, range_in);
  return cudaGetLastError();
}

}  // namespace fs
