// Novel-view mask rendering (Sec. 3.4; Supp. Sec. 8.2): the segmentation's
// objects are rendered one at a time into views that may have no mask.
//
// A view batch is projected and depth-sorted once.  For object e the sorted
// slots are compacted to the visible members of {G_i}_e (order kept), binned
// into tiles in one list, and composited per pixel (Eq. 1 over the subset):
// rho^e = sum alpha T and the alpha-weighted depth sum.  The same pass folds
// the object into the mask: where rho^e > tau and its depth D^e = sum alpha T
// z / rho^e is below the best depth so far, the pixel takes label e.  Objects
// run in increasing e, so equal depths keep the smaller e.
#include <cuda_fp16.h>

#include "fs_common.cuh"
#include "fs_compact.cuh"
#include "fs_internal.h"

namespace fs {

namespace {

// Sorted slots whose Gaussian has bit `bit`.
struct MemberSlots {
  SlotView sv;
  const uint32_t* sorted_val;
  const uint64_t* member;
  uint64_t bit;
  __device__ __forceinline__ uint32_t value(int64_t p) const { return sorted_val[p]; }
  __device__ __forceinline__ bool keep(uint32_t g) const {
    return (member[g - sv(g) * sv.n] & bit) != 0ull;
  }
};

constexpr int kRenderThreads = 128;  // four warps: the 8x8 sub-tiles of a 16x16 tile
constexpr int kRenderBatch = kRenderThreads;  // records staged at a time, one per thread
// Records a warp takes between looks at its pixels' stops (1, 2, 4 at ten blocks
// per SM: 4.18, 4.10, 4.05 ms a call; eight blocks, whose 64 registers hold the
// loads of a step: 4.02).
constexpr int kRenderStep = 4;

// One block per (tile, view), one warp per 8x8 sub-tile, two pixels per lane
// (rows y and y + 4) in packed FP32; the tile's list is walked in depth order
// in batches of records staged in shared memory.  Plain FP32 compositing with
// the solve's rules: alpha = min(0.99, o 2^-|W (p - m)|^2), skipped below
// 1/255, and the pixel stops before a Gaussian that takes T below 1e-4.
// best[] holds, per pixel of the batch, the smallest depth of a passing object
// so far (written on the first object).
//
// Bound by issue.  Where a record is staged, it is tested against the four
// sub-tiles (over which w = W (p - m) stays in a box around its centre's); a
// warp then evaluates only the records that can reach it, and the others are
// below 1/255 at all of its pixels anyway.  A record's loads, its list entry
// and the loop are paid once for two pixels, and the pixel step is free of
// branches: with one pixel per lane, 8x4 pixels per warp and divergent skips
// and stops, 384 us for the first of 8 objects, 284 us so (500k
// Gaussians, 8 views 1008x756; the whole call 4.43 -> 4.02 ms).
template <typename OutT>
__global__ void __launch_bounds__(kRenderThreads, 8) render_kernel(
    const ViewParams* __restrict__ views, const RenderOut* __restrict__ outs,
    const uint2* __restrict__ ranges, const uint32_t* __restrict__ list_val,
    const ProjRecord* __restrict__ rec, const CompactRecord* __restrict__ rec16, int e,
    int first, float tau, float* __restrict__ best) {
  // one record more than the batch: o = 0, which no pixel takes
  __shared__ float4 s_w[kRenderBatch + 1];  // W (row-major 2x2)
  __shared__ float4 s_m[kRenderBatch + 1];  // mean as float pairs (mx, my, mx_lo, my_lo)
  __shared__ float4 s_o[kRenderBatch + 1];  // (-log2 o, clamp, depth, -)
  __shared__ uint8_t s_keep[kRenderBatch];                             // bit w: reaches warp w
  __shared__ uint8_t s_list[kRenderThreads / 32][kRenderBatch + kRenderStep];  // per warp: its records
  const int v = blockIdx.y;
  const ViewParams& vp = views[v];
  const int tiles_x = vp.tiles_x;
  const int tile = blockIdx.x;
  if (tile >= tiles_x * vp.tiles_y) return;  // whole block
  const int tx = tile % tiles_x, ty = tile / tiles_x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int px = tx * kTile + 8 * (warp & 1) + (lane & 7);
  const int py = ty * kTile + 8 * (warp >> 1) + (lane >> 3);
  const uint2 rg = ranges[vp.tile_base + tile];
  const float pxc = static_cast<float>(px) + 0.5f;
  const float2 pyc = make_float2(static_cast<float>(py) + 0.5f, static_cast<float>(py + 4) + 0.5f);
  const float tcx = static_cast<float>(tx * kTile), tcy = static_cast<float>(ty * kTile);
  const float2 one = make_float2(1.f, 1.f);
  float2 T = one, rho = make_float2(0.f, 0.f), zsum = make_float2(0.f, 0.f);
  bool done0 = px >= vp.width || py >= vp.height;
  bool done1 = px >= vp.width || py + 4 >= vp.height;
  if (threadIdx.x == 0) {
    s_w[kRenderBatch] = s_m[kRenderBatch] = make_float4(0.f, 0.f, 0.f, 0.f);
    s_o[kRenderBatch] = make_float4(__int_as_float(0x7f800000), 0.f, 0.f, 0.f);
  }
  for (uint32_t base = rg.x; base < rg.y; base += kRenderBatch) {
    if (__syncthreads_and(done0 && done1 ? 1 : 0)) break;  // every pixel of the tile stopped
    const uint32_t k = base + threadIdx.x;
    uint32_t keep = 0u;
    if (k < rg.y) {
      const uint32_t g = list_val[k];
      float4 w, m;
      float qc;
      if (rec16) {
        const CompactRecord r = rec16[g];
        const float2 wa = __half22float2(*reinterpret_cast<const __half2*>(&r.w01));
        const float2 wb = __half22float2(*reinterpret_cast<const __half2*>(&r.w23));
        w = make_float4(wa.x, wa.y, wb.x, wb.y);
        m = make_float4(r.mx, r.my, 0.f, 0.f);
        s_o[threadIdx.x] = make_float4(r.nlo, r.o > kAlphaMax ? 1.f : 0.f, r.depth, 0.f);
        qc = r.q_cut;
      } else {
        const ProjRecord r = rec[g];
        w = r.w_hi;
        m = r.m;
        s_o[threadIdx.x] = make_float4(r.misc.z, r.misc.x > kAlphaMax ? 1.f : 0.f, r.misc.w, 0.f);
        qc = r.misc.y;
      }
      s_w[threadIdx.x] = w;
      s_m[threadIdx.x] = m;
      // sub-tile q: pixel centres within 3.5 of its own centre.  This test's rows
      // and a pixel's are each off by less than 2^-21 of their terms' sizes
      // (|p - m| <= the tile centre's + 8), taken off here: means any distance
      // away lose no pixel that its own evaluation would take
      const float ex = fmaf(0x1p-20f, fabsf((tcx + 8.f) - m.x) + 8.f, 3.5f);
      const float ey = fmaf(0x1p-20f, fabsf((tcy + 8.f) - m.y) + 8.f, 3.5f);
      const float h0 = fmaf(fabsf(w.x), ex, fabsf(w.y) * ey);
      const float h1 = fmaf(fabsf(w.z), ex, fabsf(w.w) * ey);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float dx = ((tcx + 8.f * (q & 1) + 4.f) - m.x) - m.z;
        const float dy = ((tcy + 8.f * (q >> 1) + 4.f) - m.y) - m.w;
        const float d0 = fmaxf(0.f, fabsf(fmaf(w.x, dx, w.y * dy)) - h0);
        const float d1 = fmaxf(0.f, fabsf(fmaf(w.z, dx, w.w * dy)) - h1);
        if (fmaf(d0, d0, d1 * d1) <= qc) keep |= 1u << q;
      }
    }
    s_keep[threadIdx.x] = static_cast<uint8_t>(keep);
    __syncthreads();
    // the warp's records, in list order, filled up to whole steps
    int count = 0;
#pragma unroll
    for (int q = 0; q < kRenderBatch; q += 32) {
      const bool on = (s_keep[q + lane] >> warp) & 1u;
      const uint32_t bal = __ballot_sync(0xffffffffu, on);
      if (on)
        s_list[warp][count + __popc(bal & ((1u << lane) - 1u))] = static_cast<uint8_t>(q + lane);
      count += __popc(bal);
    }
    if (lane < kRenderStep) s_list[warp][count + lane] = static_cast<uint8_t>(kRenderBatch);
    __syncwarp();
    for (int c = 0; c < count; c += kRenderStep) {
      if (__all_sync(0xffffffffu, done0 && done1)) break;
#pragma unroll
      for (int u = 0; u < kRenderStep; ++u) {
        const int j = s_list[warp][c + u];
        const float4 w = s_w[j], m = s_m[j], o = s_o[j];
        const float dx = (pxc - m.x) - m.z;
        const float2 dX = make_float2(dx, dx);
        const float2 dY = add2(add2(pyc, make_float2(-m.y, -m.y)), make_float2(-m.w, -m.w));
        const float2 w0 = __ffma2_rn(make_float2(w.x, w.x), dX,
                                     __fmul2_rn(make_float2(w.y, w.y), dY));
        const float2 w1 = __ffma2_rn(make_float2(w.z, w.z), dX,
                                     __fmul2_rn(make_float2(w.w, w.w), dY));
        const float2 q = __ffma2_rn(w0, w0, __ffma2_rn(w1, w1, make_float2(o.x, o.x)));
        float a0 = ex2_approx(-q.x), a1 = ex2_approx(-q.y);
        if (o.y != 0.f) {
          a0 = fminf(a0, kAlphaMax);
          a1 = fminf(a1, kAlphaMax);
        }
        // a pixel that skips takes alpha = 0, which leaves T as it is
        if (done0 || a0 < kAlphaMin) a0 = 0.f;
        if (done1 || a1 < kAlphaMin) a1 = 0.f;
        const float2 tn = __fmul2_rn(T, __ffma2_rn(make_float2(a0, a1), make_float2(-1.f, -1.f), one));
        const bool stop0 = tn.x < kTMin, stop1 = tn.y < kTMin;
        done0 = done0 || stop0;
        done1 = done1 || stop1;
        if (stop0) a0 = 0.f;
        if (stop1) a1 = 0.f;
        const float2 al = make_float2(a0, a1);
        const float2 cT = __fmul2_rn(al, T);
        rho = add2(rho, cT);
        if (a0 != 0.f) zsum.x = fmaf(cT.x, o.z, zsum.x);  // no 0 times an overflown depth
        if (a1 != 0.f) zsum.y = fmaf(cT.y, o.z, zsum.y);
        if (!stop0) T.x = tn.x;
        if (!stop1) T.y = tn.y;
      }
    }
    __syncthreads();  // the batch is read by every thread before the next one lands
  }
  const int64_t npix = static_cast<int64_t>(vp.width) * vp.height;
  const RenderOut ro = outs[v];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int y = py + 4 * i;
    if (px >= vp.width || y >= vp.height) continue;
    const int64_t p = static_cast<int64_t>(y) * vp.width + px;
    const float r = i ? rho.y : rho.x, zs = i ? zsum.y : zsum.x;
    const float depth = r > 0.f ? zs / r : 0.f;
    if (ro.rho) ro.rho[static_cast<int64_t>(e - 1) * npix + p] = r;
    if (ro.depth) ro.depth[static_cast<int64_t>(e - 1) * npix + p] = depth;
    float* const bp = best + vp.state_off + p;
    OutT* const mp = static_cast<OutT*>(ro.mask) + p;
    float b = first ? __int_as_float(0x7f800000) : *bp;
    OutT lab = first ? static_cast<OutT>(0) : *mp;
    if (r > tau && depth < b) {
      b = depth;
      lab = static_cast<OutT>(e);
    }
    *bp = b;
    *mp = lab;
  }
}

}  // namespace

cudaError_t launch_member_slots(int64_t n_pos, int64_t n, const uint32_t* sorted_val,
                                const uint64_t* member, uint64_t bit, uint32_t* out,
                                int64_t* range_out, void* lookback, unsigned long long* counters,
                                cudaStream_t stream) {
  return launch_compact(MemberSlots{SlotView(n > 0 ? n : 1), sorted_val, member, bit}, 0, n_pos,
                        out, range_out, lookback, counters, stream, nullptr);
}

cudaError_t launch_render(const ViewParams* views, const RenderOut* outs, int n_views,
                          int max_tiles_per_view, const uint2* ranges, const uint32_t* list_val,
                          const ProjRecord* rec, const CompactRecord* rec16, int e, bool first,
                          float tau, float* best, int out_dtype, cudaStream_t stream) {
  if (n_views == 0 || max_tiles_per_view == 0) return cudaSuccess;
  dim3 grid(static_cast<unsigned>(max_tiles_per_view), static_cast<unsigned>(n_views));
  if (out_dtype == 4)
    render_kernel<uint8_t><<<grid, kRenderThreads, 0, stream>>>(
        views, outs, ranges, list_val, rec, rec16, e, first ? 1 : 0, tau, best);
  else
    render_kernel<int32_t><<<grid, kRenderThreads, 0, stream>>>(
        views, outs, ranges, list_val, rec, rec16, e, first ? 1 : 0, tau, best);
  return cudaGetLastError();
}

}  // namespace fs
