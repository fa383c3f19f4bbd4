// Closed-form optimal assignment (Sec. 3.2 "Regularized ILP for Noise
// Reduction", Sec. 3.3 Eq. 7, Supp. Sec. 6 Listing 1).
//
// Per Gaussian i with row A[i, :] and S = sum_e A[i, e] (taken once), for each
// label e: others = S - A_e; both are L1-normalised by
// n = max(|others| + |A_e|, 1e-12); the Gaussian belongs to e iff
// A_e/n > others/n + gamma (a tie is not a membership), evaluated as
// A_e - others > gamma n.  One thread per Gaussian; the decision is made in
// the table's precision.
#include <math.h>

#include "fs_compact.cuh"
#include "fs_internal.h"

namespace fs {

namespace {

struct Decision {
  uint64_t bits;
  int32_t label;
  float margin;
};

// The comparison a/n > others/n + gamma is taken as a - others > gamma n
// (n > 0: the same decision, without a division per label: FP64 divisions
// are costly on this part), and the margins share one reciprocal of S.
template <typename T>
__device__ __forceinline__ Decision decide(const T* row, int E, T gamma) {
  T S = 0;
  for (int e = 0; e < E; ++e) S += row[e];
  uint64_t b = 0;
  int members = 0, lab = -1;
  float mmin = INFINITY;
  const T one = 1;
  const T inv_s = S > 0 ? one / S : T(0);
  for (int e = 0; e < E; ++e) {
    const T a = row[e];
    const T others = S - a;
    T nrm = fabs(others) + fabs(a);
    if (nrm < T(1e-12)) nrm = T(1e-12);
    if (a - others > gamma * nrm) {
      if (e < 64) b |= (1ull << e);
      ++members;
      lab = e;
    }
    if (S > 0) {
      const T mg = fabs((one - gamma) * a - (one + gamma) * others) * inv_s;
      mmin = fminf(mmin, static_cast<float>(mg));
    }
  }
  return {b, members == 1 ? lab : -1, mmin};
}

// The same decision for an FP64 row of contributions (every entry +0 or
// above), at two FP64 operations per label instead of eleven: |others| + |a| is
// S then, so a - others > gamma n and the margin's term are the sign and the
// size of t = 2 a - (1 + gamma) S.  Signs and sizes of doubles compare as
// integers.  Unseen rows (S = 0) take the same path, the others -- a negative
// or non-finite entry, a sum at the clamp of n or near overflow -- the general
// form.  Bound by the FP64 pipe: 3M rows of 33 labels, with the rounding of
// the table, took 2.43 ms in the general form, 0.95 ms in this one.
__device__ __forceinline__ Decision decide_row(const double* row, int E, double gamma) {
  double S = 0.0;
  int signs = 0;  // sign bits of the entries
  for (int e = 0; e < E; ++e) {
    const double a = row[e];
    S += a;
    signs |= __double2hiint(a);
  }
  // S <= 1e300 also leaves out NaN and infinities
  if (signs < 0 || !(S <= 1e300) || (S > 0.0 && S < 1e-12)) return decide<double>(row, E, gamma);
  // an unseen row is a member of everything for gamma < 0 and of nothing else
  const double cS = S > 0.0 ? (1.0 + gamma) * S : gamma < 0.0 ? -1e-300 : 0.0;
  uint64_t b = 0;
  int members = 0, lab = -1;
  unsigned long long least = ~0ull;  // smallest |t|, as bits
  for (int e = 0; e < E; ++e) {
    const long long t = __double_as_longlong(fma(2.0, row[e], -cS));
    const unsigned long long size = static_cast<unsigned long long>(t) & 0x7FFFFFFFFFFFFFFFull;
    if (t > 0) {  // above +0: a tie (+-0) is no membership
      if (e < 64) b |= (1ull << e);
      ++members;
      lab = e;
    }
    least = min(least, size);
  }
  const float m =
      S > 0.0 ? static_cast<float>(__longlong_as_double(static_cast<long long>(least)) * (1.0 / S))
              : INFINITY;
  return {b, members == 1 ? lab : -1, m};
}
__device__ __forceinline__ Decision decide_row(const float* row, int E, float gamma) {
  return decide<float>(row, E, gamma);
}

template <typename T>
__global__ void __launch_bounds__(256) assign_kernel(const T* __restrict__ table, int64_t n, int E,
                                                     T gamma, uint64_t* __restrict__ bits,
                                                     int32_t* __restrict__ label,
                                                     float* __restrict__ margin) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const Decision d = decide_row(table + i * E, E, gamma);
  if (bits) bits[i] = d.bits;
  if (label) label[i] = d.label;
  if (margin) margin[i] = d.margin;
}

// The same with the block's rows staged through shared memory: rows of E
// values at a stride of E are read by consecutive threads at consecutive
// addresses (the direct form above reads one row per thread, E * 8 bytes
// apart).  128 rows per block.  Bound by HBM for FP32 tables, so the rows go
// straight to shared memory in 16-byte asynchronous copies, all of a block's
// in flight at once (3M rows of 33 labels: 92 us with loads and stores, 75 us
// so, 87 % of the measured copy rate).
constexpr int kAssignRows = 128;

// bytes (any number) from src to shared memory at dst, by the whole block.
__device__ __forceinline__ void stage_rows(void* dst, const void* src, int bytes) {
  const bool aligned = (reinterpret_cast<uintptr_t>(src) & 15u) == 0;
  const int whole = aligned ? bytes / 16 : 0;
  const uint32_t to = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  for (int k = threadIdx.x; k < whole; k += kAssignRows)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + 16 * k),
                 "l"(static_cast<const char*>(src) + 16 * k));
  for (int k = 4 * whole + threadIdx.x; k < bytes / 4; k += kAssignRows)
    static_cast<uint32_t*>(dst)[k] = static_cast<const uint32_t*>(src)[k];
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
}
template <typename T>
__global__ void __launch_bounds__(kAssignRows) assign_staged_kernel(
    const T* __restrict__ table, int64_t n, int E, T gamma, uint64_t* __restrict__ bits,
    int32_t* __restrict__ label, float* __restrict__ margin) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* rows = reinterpret_cast<T*>(smem_raw);
  const int64_t i0 = static_cast<int64_t>(blockIdx.x) * kAssignRows;
  const int n_rows = static_cast<int>(min(static_cast<int64_t>(kAssignRows), n - i0));
  stage_rows(rows, table + i0 * E, n_rows * E * static_cast<int>(sizeof(T)));
  if (static_cast<int>(threadIdx.x) >= n_rows) return;
  const int64_t i = i0 + threadIdx.x;
  const Decision d = decide_row(rows + threadIdx.x * E, E, gamma);
  if (bits) bits[i] = d.bits;
  if (label) label[i] = d.label;
  if (margin) margin[i] = d.margin;
}

__global__ void __launch_bounds__(256) round_table_kernel(int64_t count,
                                                          const double* __restrict__ src,
                                                          float* __restrict__ dst) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i < count) dst[i] = static_cast<float>(src[i]);
}

// Rows re-evaluated in FP64: row j of R belongs to Gaussian F[j].  The row
// replaces the table's (rounded to its type) and the decision is taken again
// in FP64.
template <typename TableT>
__global__ void __launch_bounds__(256) assign_rows_kernel(
    const double* __restrict__ R, const uint32_t* __restrict__ F, int64_t n_rows, int E,
    double gamma, TableT* __restrict__ table, uint64_t* __restrict__ bits,
    int32_t* __restrict__ label, float* __restrict__ margin) {
  const int64_t j = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (j >= n_rows) return;
  const double* row = R + j * E;
  const int64_t i = F[j];
  for (int e = 0; e < E; ++e) table[i * E + e] = static_cast<TableT>(row[e]);
  const Decision d = decide_row(row, E, gamma);
  if (bits) bits[i] = d.bits;
  if (label) label[i] = d.label;
  if (margin) margin[i] = d.margin;
}

// The Gaussians in none of the objects of `remove`.
struct KeptGaussians {
  const uint64_t* bits;
  uint64_t remove;
  __device__ __forceinline__ uint32_t value(int64_t p) const { return static_cast<uint32_t>(p); }
  __device__ __forceinline__ bool keep(uint32_t i) const { return (bits[i] & remove) == 0ull; }
};

}  // namespace

cudaError_t launch_keep(int64_t n, const uint64_t* member_bits, uint64_t remove, int32_t* keep,
                        int64_t* range_out, void* lookback, unsigned long long* counters,
                        cudaStream_t stream) {
  return launch_compact(KeptGaussians{member_bits, remove}, 0, n,
                        reinterpret_cast<uint32_t*>(keep), range_out, lookback, counters, stream,
                        nullptr);
}

cudaError_t launch_assign(const void* table, int table_dtype, int64_t n, int E, float gamma,
                          uint64_t* member_bits, int32_t* label, float* margin,
                          cudaStream_t stream) {
  if (n == 0) return cudaSuccess;
  const size_t elem = table_dtype == 0 ? 4 : 8;
  const size_t smem = static_cast<size_t>(kAssignRows) * E * elem;
  if (E > 4 && smem <= 48 * 1024) {
    const unsigned blocks = static_cast<unsigned>((n + kAssignRows - 1) / kAssignRows);
    if (table_dtype == 0)
      assign_staged_kernel<float><<<blocks, kAssignRows, smem, stream>>>(
          static_cast<const float*>(table), n, E, gamma, member_bits, label, margin);
    else
      assign_staged_kernel<double><<<blocks, kAssignRows, smem, stream>>>(
          static_cast<const double*>(table), n, E, static_cast<double>(gamma), member_bits,
          label, margin);
    return cudaGetLastError();
  }
  const int threads = 256;
  const unsigned blocks = static_cast<unsigned>((n + threads - 1) / threads);
  if (table_dtype == 0)
    assign_kernel<float><<<blocks, threads, 0, stream>>>(static_cast<const float*>(table), n, E,
                                                         gamma, member_bits, label, margin);
  else
    assign_kernel<double><<<blocks, threads, 0, stream>>>(static_cast<const double*>(table), n, E,
                                                          static_cast<double>(gamma), member_bits,
                                                          label, margin);
  return cudaGetLastError();
}

cudaError_t launch_round_table(int64_t count, const double* src, float* dst,
                               cudaStream_t stream) {
  if (count == 0) return cudaSuccess;
  const int threads = 256;
  round_table_kernel<<<static_cast<unsigned>((count + threads - 1) / threads), threads, 0,
                       stream>>>(count, src, dst);
  return cudaGetLastError();
}

cudaError_t launch_assign_rows(const double* R, const uint32_t* F, int64_t n_rows, int E,
                               float gamma, void* table, int table_dtype, uint64_t* member_bits,
                               int32_t* label, float* margin, cudaStream_t stream) {
  if (n_rows == 0) return cudaSuccess;
  const int threads = 256;
  const unsigned blocks = static_cast<unsigned>((n_rows + threads - 1) / threads);
  if (table_dtype == 0)
    assign_rows_kernel<float><<<blocks, threads, 0, stream>>>(
        R, F, n_rows, E, static_cast<double>(gamma), static_cast<float*>(table), member_bits,
        label, margin);
  else
    assign_rows_kernel<double><<<blocks, threads, 0, stream>>>(
        R, F, n_rows, E, static_cast<double>(gamma), static_cast<double*>(table), member_bits,
        label, margin);
  return cudaGetLastError();
}

}  // namespace fs
