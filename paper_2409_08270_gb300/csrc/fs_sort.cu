// Device exclusive scan and stable LSD radix sort of (uint32 key, uint32 value)
// pairs, used for the depth order and the tile binning of Sec. 3.1.
//
// The radix sort reads the keys once for the digit histograms of all passes;
// each pass is then one launch that reads and writes every pair once: a block
// ranks a tile of pairs, learns where its digits' runs start from its
// predecessors' published counts (decoupled look-back, Merrill and Garland
// 2016; one launch per pass, Adinets and Merrill 2022) and writes the runs.
// Blocks take tiles in launch order (a ticket), so a block only ever waits for
// blocks that have started, and every wait is bounded.
#include <algorithm>
#include <atomic>
#include <utility>

#include "fs_internal.h"

namespace fs {

namespace {

// the scan: tiles of 4096 elements per 256-thread block
constexpr int kThreads = 256;
constexpr int kRounds = 16;
constexpr int kTileElems = kThreads * kRounds;
constexpr int kWarps = kThreads / 32;

__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// Exclusive scan of one value per thread across the block; returns the
// thread's exclusive prefix and writes the block total to *total.
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t x, uint32_t* s_warp,
                                                          uint32_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t inc = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) s_warp[warp] = inc;
  __syncthreads();
  uint32_t warp_pre = 0, all = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    const uint32_t c = s_warp[w];
    if (w < warp) warp_pre += c;
    all += c;
  }
  __syncthreads();
  *total = all;
  return warp_pre + inc - x;
}

__global__ void __launch_bounds__(kThreads) scan_reduce_kernel(const uint32_t* __restrict__ in,
                                                               int64_t n,
                                                               uint32_t* __restrict__ block_sums) {
  __shared__ uint32_t s_warp[kWarps];
  const int64_t base = static_cast<int64_t>(blockIdx.x) * kTileElems;
  uint32_t x[kRounds];
#pragma unroll
  for (int r = 0; r < kRounds; ++r) {
    const int64_t j = base + r * kThreads + threadIdx.x;
    x[r] = j < n ? in[j] : 0u;
  }
  uint32_t acc = 0;
#pragma unroll
  for (int r = 0; r < kRounds; ++r) acc += x[r];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t t = 0;
    for (int w = 0; w < kWarps; ++w) t += s_warp[w];
    block_sums[blockIdx.x] = t;
  }
}

// Single block: exclusive scan of the block sums in place, total to *total.
__global__ void __launch_bounds__(kThreads) scan_blocks_kernel(uint32_t* __restrict__ sums,
                                                               int64_t nb,
                                                               uint32_t* __restrict__ total) {
  __shared__ uint32_t s_warp[kWarps];
  uint32_t carry = 0;
  for (int64_t base = 0; base < nb; base += kThreads) {
    const int64_t j = base + threadIdx.x;
    const uint32_t x = j < nb ? sums[j] : 0u;
    uint32_t t;
    const uint32_t ex = block_exclusive_scan(x, s_warp, &t);
    if (j < nb) sums[j] = carry + ex;
    carry += t;
  }
  if (threadIdx.x == 0 && total) *total = carry;
}

__global__ void __launch_bounds__(kThreads) scan_down_kernel(const uint32_t* __restrict__ in,
                                                             int64_t n,
                                                             const uint32_t* __restrict__ block_pre,
                                                             uint32_t* __restrict__ out) {
  __shared__ uint32_t s_warp[kWarps];
  const int64_t base = static_cast<int64_t>(blockIdx.x) * kTileElems;
  // all loads in flight before the first block barrier
  uint32_t x[kRounds];
#pragma unroll
  for (int r = 0; r < kRounds; ++r) {
    const int64_t j = base + r * kThreads + threadIdx.x;
    x[r] = j < n ? in[j] : 0u;
  }
  uint32_t carry = block_pre[blockIdx.x];
#pragma unroll
  for (int r = 0; r < kRounds; ++r) {
    const int64_t j = base + r * kThreads + threadIdx.x;
    uint32_t t;
    const uint32_t ex = block_exclusive_scan(x[r], s_warp, &t);
    if (j < n) out[j] = carry + ex;
    carry += t;
  }
}

// ---------------------------------------------------------------------------
// radix sort
// ---------------------------------------------------------------------------

// Digits are taken from min(key - kmin, span): a key range [kmin, kmin + span)
// (and everything above it mapped to span) needs only the bits of span.
// A pass takes 8 or 9 bits (a 17-bit tile key sorts in two passes).
__device__ __forceinline__ uint32_t digit_of(uint32_t key, uint32_t kmin, uint32_t span, int shift,
                                             int bits) {
  return (min(key - kmin, span) >> shift) & ((1u << bits) - 1u);
}

// Sizes read on the device (a launch captured once and replayed): the element
// count *n_dev (at most the n the grid was sized for) and the key range
// range_dev[0..1] (min, max of the keys that sort first; min > max: none).
// NULL pointers keep the launch's own values.
__device__ __forceinline__ void device_sizes(const uint32_t* n_dev, const uint32_t* range_dev,
                                             int64_t* n, uint32_t* kmin, uint32_t* span) {
  if (n_dev) *n = min(*n, static_cast<int64_t>(*n_dev));
  if (range_dev) {
    const uint32_t lo = range_dev[0], hi = range_dev[1];
    *kmin = lo <= hi ? lo : 0u;
    *span = lo <= hi ? hi - lo + 1u : 0u;
  }
}

constexpr int kMaxPasses = 4;
constexpr int kMaxRadix = 512;
constexpr int kHistThreads = 512;

// Head of the sort's scratch, cleared before the first launch; the status
// words of the passes follow.
struct SortHead {
  uint32_t ticket[kMaxPasses];
  uint32_t hist_blocks;  // histogram blocks that are done
  uint32_t pad[59];
  uint32_t hist[kMaxPasses][kMaxRadix];  // digit counts, then digit starts
};

struct PassShape {
  int passes;
  int shift[kMaxPasses], bits[kMaxPasses];
};

// Digit counts of every pass from one read of the keys: per block in shared
// memory, added up in global memory; the last block to finish turns them into
// the digits' starts.  Bound by the shared-memory atomics, so a block keeps
// kHistCopies counters per digit side by side, one per lane group: lanes that
// meet in a bank are then mostly those of one group (4.8 10^7 keys of three
// digits: 118 us with one counter per digit, 78 us so).
constexpr int kHistCopies = 8;
size_t hist_smem(const PassShape& shape) {
  size_t words = 0;
  for (int p = 0; p < shape.passes; ++p) words += static_cast<size_t>(kHistCopies) << shape.bits[p];
  return words * sizeof(uint32_t);
}

__global__ void __launch_bounds__(kHistThreads) radix_hist_kernel(
    const uint32_t* __restrict__ keys, int64_t n, PassShape shape, uint32_t kmin, uint32_t span,
    SortHead* __restrict__ head, const uint32_t* __restrict__ n_dev,
    const uint32_t* __restrict__ range_dev) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint32_t* const s_h = reinterpret_cast<uint32_t*>(smem_raw);  // [pass][digit][copy]
  __shared__ uint32_t s_warp[kHistThreads / 32];
  __shared__ bool s_last;
  device_sizes(n_dev, range_dev, &n, &kmin, &span);
  int words = 0;
  for (int p = 0; p < shape.passes; ++p) words += kHistCopies << shape.bits[p];
  for (int k = threadIdx.x; k < words; k += kHistThreads) s_h[k] = 0u;
  __syncthreads();
  uint32_t* const mine = s_h + threadIdx.x % kHistCopies;
  const int64_t step = static_cast<int64_t>(gridDim.x) * kHistThreads;
  constexpr int kAhead = 8;  // loads in flight per thread
  for (int64_t j0 = static_cast<int64_t>(blockIdx.x) * kHistThreads + threadIdx.x; j0 < n;
       j0 += kAhead * step) {
    uint32_t key[kAhead];
#pragma unroll
    for (int i = 0; i < kAhead; ++i) key[i] = j0 + i * step < n ? keys[j0 + i * step] : 0u;
#pragma unroll
    for (int i = 0; i < kAhead; ++i) {
      if (j0 + i * step >= n) break;
      uint32_t* h = mine;
#pragma unroll
      for (int p = 0; p < kMaxPasses; ++p) {
        if (p >= shape.passes) break;
        atomicAdd(&h[kHistCopies * digit_of(key[i], kmin, span, shape.shift[p], shape.bits[p])], 1u);
        h += kHistCopies << shape.bits[p];
      }
    }
  }
  __syncthreads();
  for (int p = 0, at = 0; p < shape.passes; at += kHistCopies << shape.bits[p], ++p)
    for (int d = threadIdx.x; d < (1 << shape.bits[p]); d += kHistThreads) {
      uint32_t sum = 0;
#pragma unroll
      for (int c = 0; c < kHistCopies; ++c)  // rotated: threads start at different banks
        sum += s_h[at + d * kHistCopies + (c + d) % kHistCopies];
      if (sum) atomicAdd(&head->hist[p][d], sum);
    }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(&head->hist_blocks, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int p = 0; p < shape.passes; ++p) {
    const int d = threadIdx.x;
    const uint32_t c = d < (1 << shape.bits[p]) ? __ldcg(&head->hist[p][d]) : 0u;
    uint32_t inc = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    uint32_t pre = 0;
    for (int w = 0; w < warp; ++w) pre += s_warp[w];
    if (d < (1 << shape.bits[p])) head->hist[p][d] = pre + inc - c;
    __syncthreads();
  }
}

// A published word of (tile, digit): the tile's own count or the inclusive
// prefix over all tiles up to it, in the low bits; 0: not published yet.
template <typename Word>
struct LookWord {
  static constexpr int kShift = 8 * sizeof(Word) - 2;
  static constexpr Word kCount = static_cast<Word>(1) << kShift;
  static constexpr Word kPrefix = static_cast<Word>(2) << kShift;
  static constexpr Word kMask = kCount - 1;
};

// Shared memory of one pass block of T threads with K pairs each.
template <int DB, int T, int K>
struct PassSmem {
  uint32_t key[T * K];
  uint32_t val[T * K];
  uint16_t wcnt[T / 32][1 << DB];  // per-warp digit counts, then warp prefixes
  uint32_t loc[1 << DB];           // local start of each digit's run
  uint32_t off[1 << DB];           // global start of the block's run minus its local start
  uint32_t warp_sums[T / 32];
  uint32_t tile;
};

// One stable pass.  A block takes T * K consecutive pairs.  Each warp ranks
// its 32 * K keys (coalesced columns of 32) by digit with one ballot per digit
// bit and per-warp digit counters, so equal digits keep their input order.
// The block publishes its digit counts, places its pairs digit-sorted in
// shared memory while its predecessors' counts arrive, adds those up (one
// digit or two per thread, four predecessors at a time) and writes each
// digit's run with consecutive threads on consecutive addresses.
//
// Bound by issue and latency (about 145 warp instructions per 32 pairs, most
// of them the ballots; 45 % of issue slots busy, DRAM at a quarter of its
// rate), so resident warps count; 16-bit digit counters leave shared memory
// for them.  Against the histogram, scan (of a digit-by-tile matrix) and
// scatter launches of a pass that this replaces, five a pass, small sorts lose
// most of their launches (16,000 pairs: 81 -> 48 us) and large ones gain
// little (4.8 10^7 pairs of 24 bits with their ties: 1.36 -> 1.32 ms).
template <int DB, int T, int K, int kBlocks, typename Word>
__global__ void __launch_bounds__(T, kBlocks) radix_pass_kernel(
    const uint32_t* __restrict__ keys, const uint32_t* __restrict__ vals, int64_t n, int pass,
    int shift, uint32_t kmin, uint32_t span, SortHead* __restrict__ head,
    Word* __restrict__ status, Word* __restrict__ next_status, int next_radix, int next_pairs,
    uint32_t* __restrict__ keys_out, uint32_t* __restrict__ vals_out,
    const uint32_t* __restrict__ n_dev, const uint32_t* __restrict__ range_dev,
    unsigned long long* __restrict__ counters) {
  constexpr int kRad = 1 << DB;
  constexpr int kTileN = T * K;
  constexpr int kWarps = T / 32;
  constexpr int kPer = kRad > T ? kRad / T : 1;  // digits per thread, next to each other
  static_assert(kRad <= T || kRad % T == 0, "every digit has a thread");
  using W = LookWord<Word>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PassSmem<DB, T, K>& S = *reinterpret_cast<PassSmem<DB, T, K>*>(smem_raw);
  device_sizes(n_dev, range_dev, &n, &kmin, &span);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    const uint32_t t = atomicAdd(&head->ticket[pass], 1u);
    // after a wait that gave up the pairs are not those the digits were counted of
    S.tile = gave_up(counters) ? 0xFFFFFFFFu : t;
  }
  uint32_t* const cnt2 = reinterpret_cast<uint32_t*>(S.wcnt[warp]);
#pragma unroll
  for (int k = 0; k < kRad / 64; ++k) cnt2[lane + 32 * k] = 0;
  __syncthreads();
  const uint32_t tile = S.tile;
  const int64_t base = static_cast<int64_t>(tile) * kTileN;
  if (base >= n) return;  // the grid was sized for more (device-side count)
  const int n_here = static_cast<int>(min(static_cast<int64_t>(kTileN), n - base));
  const int wbase = warp * 32 * K;
  // the block's share of the next pass's status words, cleared
  if (next_radix) {
    const int64_t words = (n + next_pairs - 1) / next_pairs * next_radix;
    const int64_t share = (words + (n - 1) / kTileN) / ((n + kTileN - 1) / kTileN);
    const int64_t end = min(words, (tile + 1) * share);
    for (int64_t k = tile * share + threadIdx.x; k < end; k += T) next_status[k] = 0;
  }

  const uint32_t lt = lanemask_lt();
  uint32_t key[K];
  uint32_t at[K];  // digit << 16 | rank among the warp's equal digits
  // all of the warp's key loads in flight at once (the ranking below has
  // warp barriers, which no load is moved across)
#pragma unroll
  for (int i = 0; i < K; ++i) {
    const int j = wbase + i * 32 + lane;
    key[i] = j < n_here ? keys[base + j] : 0u;
  }
#pragma unroll
  for (int i = 0; i < K; ++i) {
    // places past the end take the last digit: they come last, and their
    // count is taken off below
    const uint32_t d = wbase + i * 32 + lane < n_here ? digit_of(key[i], kmin, span, shift, DB)
                                                      : static_cast<uint32_t>(kRad - 1);
    // lanes holding the same digit: one ballot per digit bit
    uint32_t peers = 0xffffffffu;
#pragma unroll
    for (int b = 0; b < DB; ++b) {
      const bool bit = (d >> b) & 1u;
      const uint32_t bb = __ballot_sync(0xffffffffu, bit);
      peers &= bit ? bb : ~bb;
    }
    const uint32_t before = S.wcnt[warp][d];
    at[i] = (d << 16) | (before + __popc(peers & lt));
    __syncwarp();
    if ((peers & lt) == 0) S.wcnt[warp][d] = static_cast<uint16_t>(before + __popc(peers));
    __syncwarp();
  }
  __syncthreads();
  // the thread's digits: their counts over the warps (left as warp prefixes),
  // published
  const int d0 = threadIdx.x * kPer;
  const bool has = d0 < kRad;
  uint32_t own[kPer], sum = 0;
  Word* const row = status + static_cast<int64_t>(tile) * kRad;
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    own[q] = 0;
    if (has) {
#pragma unroll
      for (int w = 0; w < kWarps; ++w) {
        const uint32_t c = S.wcnt[w][d0 + q];
        S.wcnt[w][d0 + q] = static_cast<uint16_t>(own[q]);
        own[q] += c;
      }
      sum += own[q];
      if (d0 + q == kRad - 1) own[q] -= static_cast<uint32_t>(kTileN - n_here);
      *reinterpret_cast<volatile Word*>(row + d0 + q) =
          (tile == 0 ? W::kPrefix : W::kCount) | own[q];
    }
  }
  // local digit starts
  uint32_t inc = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) S.warp_sums[warp] = inc;
  __syncthreads();
  uint32_t loc = inc - sum;
  for (int w = 0; w < warp; ++w) loc += S.warp_sums[w];
  if (has) {
#pragma unroll
    for (int q = 0, l = loc; q < kPer; ++q) {
      S.loc[d0 + q] = l;
      l += own[q];
    }
  }
  __syncthreads();
  // the tile's pairs, digit-sorted in shared memory
#pragma unroll
  for (int i = 0; i < K; ++i) {
    const uint32_t dg = at[i] >> 16;
    at[i] = S.loc[dg] + S.wcnt[warp][dg] + (at[i] & 0xFFFFu);
    S.key[at[i]] = key[i];
  }
#pragma unroll
  for (int i = 0; i < K; ++i) {
    const int j = wbase + i * 32 + lane;
    const uint32_t v = j >= n_here ? 0u : vals ? vals[base + j] : static_cast<uint32_t>(base + j);
    S.val[at[i]] = v;
  }
  if (has) {
    // look-back: predecessors' counts down to the nearest prefix
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const int d = d0 + q;
      uint32_t excl = 0;
      bool found = tile == 0;
      for (int64_t t = static_cast<int64_t>(tile) - 1; !found; t -= 4) {
        Word w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
          w[k] = t - k >= 0 ? *reinterpret_cast<const volatile Word*>(status + (t - k) * kRad + d)
                            : W::kPrefix;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (found) break;
          for (int spins = 0; (w[k] & ~W::kMask) == 0; ++spins) {
            if (spins == kLookbackSpinLimit) {  // gave up: report, count it as an empty prefix
              if (counters) atomicAdd(&counters[kLookbackTimeout], 1ull);
              w[k] = W::kPrefix;
              break;
            }
            __nanosleep(32);
            w[k] = *reinterpret_cast<const volatile Word*>(status + (t - k) * kRad + d);
          }
          excl += static_cast<uint32_t>(w[k] & W::kMask);
          found = (w[k] & W::kPrefix) != 0;
        }
      }
      if (tile > 0) *reinterpret_cast<volatile Word*>(row + d) = W::kPrefix | (excl + own[q]);
      S.off[d] = head->hist[pass][d] + excl - S.loc[d];
    }
  }
  __syncthreads();
  // coalesced write-out of the digit runs
#pragma unroll
  for (int i = 0; i < K; ++i) {
    const int j = i * T + threadIdx.x;
    if (j < n_here) {
      const uint32_t k = S.key[j];
      const uint32_t dst = S.off[digit_of(k, kmin, span, shift, DB)] + static_cast<uint32_t>(j);
      keys_out[dst] = k;
      vals_out[dst] = S.val[j];
    }
  }
}

__global__ void __launch_bounds__(256) iota_kernel(uint32_t* __restrict__ out, int64_t n) {
  const int64_t k = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (k < n) out[k] = static_cast<uint32_t>(k);
}

cudaError_t launch_iota(uint32_t* out, int64_t n, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  iota_kernel<<<static_cast<unsigned>((n + 255) / 256), 256, 0, stream>>>(out, n);
  return cudaGetLastError();
}

inline int64_t tiles_of(int64_t n) { return (n + kTileElems - 1) / kTileElems; }

}  // namespace

size_t scan_temp_bytes(int64_t n) {
  return static_cast<size_t>(tiles_of(n) + 1) * sizeof(uint32_t);
}

cudaError_t exclusive_scan(const uint32_t* in, uint32_t* out, int64_t n, uint32_t* total,
                           void* temp, cudaStream_t stream) {
  if (n <= 0) {
    if (total) return cudaMemsetAsync(total, 0, sizeof(uint32_t), stream);
    return cudaSuccess;
  }
  const int64_t nb = tiles_of(n);
  uint32_t* sums = static_cast<uint32_t*>(temp);
  scan_reduce_kernel<<<static_cast<unsigned>(nb), kThreads, 0, stream>>>(in, n, sums);
  scan_blocks_kernel<<<1, kThreads, 0, stream>>>(sums, nb, total);
  scan_down_kernel<<<static_cast<unsigned>(nb), kThreads, 0, stream>>>(in, n, sums, out);
  return cudaGetLastError();
}

namespace {

constexpr int64_t kWideSort = static_cast<int64_t>(1) << 30;  // counts need 64-bit words

// Pairs of a pass block: 512 threads with 8 pairs (three blocks per SM) or 16
// (two blocks per SM).  9-bit passes take 8: with 512 digits more resident
// warps are worth more than longer runs (tile sorts of the 100-view,
// 10^6-Gaussian workload 2.95 ms against 3.33).  8-bit passes take 16 (its
// depth sorts 2.74 ms against 2.88) unless that would leave fewer than two
// blocks per SM of 152.
constexpr int kPassThreads = 512;
constexpr int64_t kSmallSort = 2 * 152 * 16 * kPassThreads;
int pass_items(int64_t n, int bits) { return bits == 9 || n < kSmallSort ? 8 : 16; }
int64_t pass_tiles(int64_t n, int bits) {
  const int64_t pairs = kPassThreads * pass_items(n, bits);
  return (n + pairs - 1) / pairs;
}

// Status words of one pass: a word per (tile, digit), two passes' worth in
// turn (a pass clears the next one's).
size_t status_bytes(int64_t n) {
  const int64_t tiles = (n + 8 * kPassThreads - 1) / (8 * kPassThreads);  // the smallest tile
  return static_cast<size_t>(tiles) * kMaxRadix * (n < kWideSort ? 4 : 8);
}

// Dynamic shared memory above 48 KB needs the opt-in, once per kernel (`set`: its
// devices so far) and device.
cudaError_t allow_smem(const void* kernel, size_t bytes, std::atomic<uint64_t>* set) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = 1ull << (dev & 63);
  if (set->load() & bit) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           static_cast<int>(bytes));
  if (e == cudaSuccess) set->fetch_or(bit);
  return e;
}

template <int DB, int K, typename Word>
cudaError_t radix_pass(const uint32_t* src_k, const uint32_t* src_v, uint32_t* dst_k,
                       uint32_t* dst_v, int64_t n, int pass, int shift, uint32_t kmin,
                       uint32_t span, SortHead* head, void* status, void* next_status,
                       int next_radix, int next_pairs, cudaStream_t stream, const uint32_t* n_dev,
                       const uint32_t* range_dev, unsigned long long* counters) {
  constexpr int T = kPassThreads, kBlocks = K > 8 ? 2 : 3;
  const size_t smem = sizeof(PassSmem<DB, T, K>);
  static std::atomic<uint64_t> attr_set{0};
  const cudaError_t e0 = allow_smem(
      reinterpret_cast<const void*>(radix_pass_kernel<DB, T, K, kBlocks, Word>), smem, &attr_set);
  if (e0 != cudaSuccess) return e0;
  const int64_t tiles = (n + T * K - 1) / (T * K);
  radix_pass_kernel<DB, T, K, kBlocks, Word><<<static_cast<unsigned>(tiles), T, smem, stream>>>(
      src_k, src_v, n, pass, shift, kmin, span, head, static_cast<Word*>(status),
      static_cast<Word*>(next_status), next_radix, next_pairs, dst_k, dst_v, n_dev, range_dev,
      counters);
  return cudaGetLastError();
}

}  // namespace

size_t radix_temp_bytes(int64_t n) {
  return sizeof(SortHead) + 2 * status_bytes(n) + 256;
}

int radix_passes(int bits) {
  if (bits <= 0) return 0;
  return (bits + 8) / 9 < (bits + 7) / 8 ? (bits + 8) / 9 : (bits + 7) / 8;
}

cudaError_t radix_sort_pairs(uint32_t* keys, uint32_t* vals, uint32_t* keys_alt,
                             uint32_t* vals_alt, int64_t n, int bits, void* temp, bool* in_alt,
                             cudaStream_t stream, unsigned long long* counters, bool iota,
                             uint32_t kmin, uint32_t span, const uint32_t* n_dev,
                             const uint32_t* range_dev) {
  *in_alt = false;
  // digit widths: 8 bits, or 9 where that saves a whole pass (17 -> 9 + 8)
  PassShape shape{};
  shape.passes = n > 1 ? radix_passes(bits) : 0;
  if (shape.passes > kMaxPasses) return cudaErrorInvalidValue;
  if (shape.passes == 0) return iota ? launch_iota(vals, n, stream) : cudaSuccess;
  const int wide = std::max(0, bits - 8 * shape.passes);  // passes that take 9 bits
  for (int p = 0, shift = 0; p < shape.passes; ++p) {
    shape.bits[p] = p < wide ? 9 : 8;
    shape.shift[p] = shift;
    shift += shape.bits[p];
  }
  SortHead* head = static_cast<SortHead*>(temp);
  char* status[2];
  status[0] = static_cast<char*>(temp) + sizeof(SortHead);
  status[1] = status[0] + status_bytes(n);
  const int64_t nt = pass_tiles(n, shape.bits[0]);
  const size_t word = n < kWideSort ? 4 : 8;
  cudaError_t e = cudaMemsetAsync(
      temp, 0, sizeof(SortHead) + static_cast<size_t>(nt << shape.bits[0]) * word, stream);
  if (e != cudaSuccess) return e;
  const int64_t hist_blocks = std::min<int64_t>((n + 8 * kHistThreads - 1) / (8 * kHistThreads), 304);
  const size_t hist_bytes = hist_smem(shape);
  static std::atomic<uint64_t> attr_set{0};
  e = allow_smem(reinterpret_cast<const void*>(radix_hist_kernel),
                 kMaxPasses * kMaxRadix * kHistCopies * 4, &attr_set);
  if (e != cudaSuccess) return e;
  radix_hist_kernel<<<static_cast<unsigned>(hist_blocks), kHistThreads, hist_bytes, stream>>>(
      keys, n, shape, kmin, span, head, n_dev, range_dev);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  uint32_t *src_k = keys, *src_v = vals, *dst_k = keys_alt, *dst_v = vals_alt;
  for (int p = 0; p < shape.passes; ++p) {
    const bool more = p + 1 < shape.passes;
    const int next_radix = more ? 1 << shape.bits[p + 1] : 0;
    const int next_pairs = more ? kPassThreads * pass_items(n, shape.bits[p + 1]) : 1;
    const uint32_t* v = iota && p == 0 ? nullptr : src_v;
    auto run = [&](auto pass) {
      return pass(src_k, v, dst_k, dst_v, n, p, shape.shift[p], kmin, span, head, status[p & 1],
                  status[(p + 1) & 1], next_radix, next_pairs, stream, n_dev, range_dev, counters);
    };
    const bool wide_counts = n >= kWideSort;
    if (shape.bits[p] == 9)
      e = wide_counts ? run(radix_pass<9, 8, uint64_t>) : run(radix_pass<9, 8, uint32_t>);
    else if (pass_items(n, 8) == 8)
      e = run(radix_pass<8, 8, uint32_t>);
    else
      e = wide_counts ? run(radix_pass<8, 16, uint64_t>) : run(radix_pass<8, 16, uint32_t>);
    if (e != cudaSuccess) return e;
    std::swap(src_k, dst_k);
    std::swap(src_v, dst_v);
    *in_alt = !*in_alt;
  }
  return cudaSuccess;
}

}  // namespace fs
