// Re-check of near-tie decisions at float-pair ("double-float") precision.
//
// The blend composites in FP32, so every table entry carries a relative error
// of about 1e-5 and the biased argmax (Sec. 3.2, Supp. Sec. 6 Listing 1) can
// come out differently from an exact evaluation for a Gaussian whose decision
// margin is that close to zero.  Such Gaussians (margin below a threshold)
// are re-evaluated here: every pixel of every view that one of them can reach
// is composited again front to back (Eq. 1: alpha, T, the 1/255 and 1e-4
// decisions) in float-pair arithmetic, about 1e-11 relative, up to its last
// re-checked Gaussian; their contributions alpha_i T_i go into an FP64 table
// of their own (Eq. 6/7) which then replaces their rows.  Float pairs keep
// the work on the FP32 pipe (GB300's FP64 rate is a small fraction of it).
//
// The per-tile depth-ordered lists come either from the main pass (its depth
// chunks, kept in memory) or from a dedicated binning of just the tiles the
// re-checked Gaussians reach.  A tile that saturated in the main pass has no
// list entries in later chunks; when a re-checked Gaussian sits in such a
// chunk ("deep" tile), a pixel it reaches is walked to its stop, and a pixel
// still compositing at the end of the kept lists (the FP32 and the exact stop
// decisions differ there) is reported so the caller redoes the batch with the
// dedicated binning.
//
// alpha = o 2^-|W (p - m)|^2 from the float-pair whitening record of the
// projection; 2^-q follows Tang's table-driven method (ACM TOMS 15(2), 1989):
// a 64-entry table of 2^(-j/64) (computed in FP64) times a degree-4 Taylor
// polynomial of e^-x on the remaining [0, ln2/64).
#include <cuda_fp16.h>
#include <math.h>

#include <algorithm>

#include "fs_binning.cuh"
#include "fs_common.cuh"
#include "fs_internal.h"

namespace fs {

namespace {

__global__ void flag_margin_kernel(int64_t n, const float* __restrict__ margin, float tau,
                                   uint32_t* __restrict__ flag) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float m = margin[i];
  flag[i] = (m < tau) ? 1u : 0u;  // +inf (unseen) and NaN are never flagged
}

__global__ void scatter_flagged_kernel(int64_t n, const uint32_t* __restrict__ flag,
                                       const uint32_t* __restrict__ offs,
                                       uint32_t* __restrict__ F, int32_t* __restrict__ map) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  if (flag[i]) {
    F[offs[i]] = static_cast<uint32_t>(i);
    map[i] = static_cast<int32_t>(offs[i]);
  } else {
    map[i] = -1;
  }
}

// The slot's depth key: its record holds the FP32 depth.
__device__ __forceinline__ uint32_t slot_key(const ProjRecord* __restrict__ rec,
                                             const CompactRecord* __restrict__ rec16,
                                             uint32_t slot) {
  return depth_key(rec16 ? rec16[slot].depth : rec[slot].misc.w);
}

// Position of slot a before-or-equal slot b in the batch's depth order:
// (depth key, view, low word of the depth, slot).
__device__ __forceinline__ bool order_le(uint32_t a, uint32_t b, int64_t n,
                                         const ProjRecord* __restrict__ rec,
                                         const CompactRecord* __restrict__ rec16,
                                         const uint32_t* __restrict__ dlo) {
  const uint32_t ka = slot_key(rec, rec16, a), kb = slot_key(rec, rec16, b);
  if (ka != kb) return ka < kb;
  const uint32_t va = a / static_cast<uint32_t>(n), vb = b / static_cast<uint32_t>(n);
  if (va != vb) return va < vb;
  if (dlo[a] != dlo[b]) return dlo[a] < dlo[b];
  return a <= b;
}

// Clears, in the skip bit array, every tile that a re-checked Gaussian's
// footprint reaches in a view of the batch (the array starts all ones), and
// counts the visible (view, re-checked Gaussian) pairs in *visible.  With
// kept chunk lists (bound != NULL), a tile that saturated in an earlier chunk
// than the re-checked Gaussian's own gets its `deep` bit set.
__global__ void mark_tiles_kernel(int64_t n_flagged, int v_begin, int n_views, int64_t n,
                                  const uint32_t* __restrict__ F,
                                  const ViewParams* __restrict__ views,
                                  const TileBox* __restrict__ box,
                                  const Footprint* __restrict__ foot,
                                  unsigned long long* __restrict__ skip,
                                  uint32_t* __restrict__ visible,
                                  const uint32_t* __restrict__ bound, int chunks,
                                  const ProjRecord* __restrict__ rec,
                                  const CompactRecord* __restrict__ rec16,
                                  const uint32_t* __restrict__ dlo,
                                  const uint8_t* __restrict__ sat_chunk,
                                  unsigned long long* __restrict__ deep) {
  const int64_t idx = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx >= n_flagged * n_views) return;
  const int v = v_begin + static_cast<int>(idx / n_flagged);
  const int64_t slot = static_cast<int64_t>(v) * n + F[idx % n_flagged];
  if (!box_visible(box[slot])) return;
  atomicAdd(visible, 1u);
  int my_chunk = 0;
  if (bound) {
    my_chunk = chunks - 1;
    for (int ci = 0; ci < chunks - 1; ++ci)
      if (bound[ci] != 0xFFFFFFFFu &&  // an empty chunk holds nothing
          order_le(static_cast<uint32_t>(slot), bound[ci], n, rec, rec16, dlo)) {
        my_chunk = ci;
        break;
      }
  }
  const Footprint f = foot[slot];
  const ViewParams& vp = views[v];
  int ty0, ty1;
  footprint_rows(f, &ty0, &ty1);
  for (int ty = ty0; ty <= ty1; ++ty) {
    int tx0, tx1;
    if (!row_span(f, ty, vp.width, &tx0, &tx1) || !clip_cols(vp.cols, slot, &tx0, &tx1)) continue;
    const int a = vp.tile_base + ty * vp.tiles_x + tx0;
    const int b = vp.tile_base + ty * vp.tiles_x + tx1;
    for (int w = a >> 6; w <= (b >> 6); ++w) {
      unsigned long long m = ~0ull;
      if (w == (a >> 6)) m &= ~0ull << (a & 63);
      if (w == (b >> 6)) m &= ~0ull >> (63 - (b & 63));
      atomicAnd(&skip[w], ~m);
    }
    if (bound) {
      for (int t = a; t <= b; ++t)
        if (sat_chunk[t] < my_chunk) atomicOr(&deep[t >> 6], 1ull << (t & 63));
    }
  }
}

// flag[slot] = 1 iff the slot's footprint reaches a tile left unskipped.
__global__ void candidates_kernel(int64_t k_total, int64_t n, const ViewParams* __restrict__ views,
                                  const TileBox* __restrict__ box,
                                  const Footprint* __restrict__ foot,
                                  const uint64_t* __restrict__ skip, uint32_t* __restrict__ flag) {
  const int64_t slot = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (slot >= k_total) return;
  uint32_t hit = 0;
  if (box_visible(box[slot])) {
    const int v = static_cast<int>(slot / n);
    const ViewParams& vp = views[v];
    const Footprint f = foot[slot];
    int ty0, ty1;
    footprint_rows(f, &ty0, &ty1);
    for (int ty = ty0; ty <= ty1 && !hit; ++ty) {
      int tx0, tx1;
      if (!row_span(f, ty, vp.width, &tx0, &tx1) || !clip_cols(vp.cols, slot, &tx0, &tx1)) continue;
      const int base = vp.tile_base + ty * vp.tiles_x;
      if (count_free(skip, base + tx0, base + tx1)) hit = 1;
    }
  }
  flag[slot] = hit;
}

__global__ void compact_kernel(int64_t k_total, const uint32_t* __restrict__ flag,
                               const uint32_t* __restrict__ offs,
                               const ProjRecord* __restrict__ rec,
                               const CompactRecord* __restrict__ rec16,
                               uint32_t* __restrict__ out_key, uint32_t* __restrict__ out_val) {
  const int64_t slot = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (slot >= k_total || !flag[slot]) return;
  const uint32_t o = offs[slot];
  out_key[o] = slot_key(rec, rec16, static_cast<uint32_t>(slot));
  out_val[o] = static_cast<uint32_t>(slot);
}

constexpr int kRound = 32;       // list entries a warp stages and composites at once
constexpr int kRing = 64;        // a warp's ring of kept entries: a partial round and a step
constexpr int kFlagTest = 256;   // re-checked Gaussians tested per piece at most (see below)
constexpr int kCountShare = 128;  // above: one in this many Gaussians counted from the lists at most
constexpr int kRWarps = 4;       // warps of a block
constexpr int kSubs = 8;         // 8x4-pixel pieces of a tile, one warp's work each

// Float-pair constants of the compositing rule (Sec. 3.1 Eq. 1 conventions).
constexpr double kAlphaMinD = 1.0 / 255.0, kAlphaMaxD = 0.99, kTMinD = 1e-4;
constexpr double kLn2D = 0.69314718055994530942;
#define FS_F2C(d) f2{static_cast<float>(d), static_cast<float>((d) - static_cast<double>(static_cast<float>(d)))}

// w = W l + b at the pixel offset (lx, ly) (exact small half-integers), both rows
// side by side in packed FP32, as float pairs: the products' and sums' rounding
// errors are gathered in one float per row and put back once (a compensated dot
// product, Ogita, Rump and Oishi 2005), about 25 operations a row where a chain
// of float-pair products and sums takes 34.  wx, wy: columns of W.
__device__ __forceinline__ f2x2 f2x2_rows(float2 wxh, float2 wxl, float2 wyh, float2 wyl,
                                          float2 bh, float2 bl, float lx, float ly) {
  const float2 X = make_float2(lx, lx), Y = make_float2(ly, ly);
  const float2 p0 = __fmul2_rn(wxh, X), p1 = __fmul2_rn(wyh, Y);
  float2 err = add2(__ffma2_rn(wxh, X, neg2(p0)), __ffma2_rn(wyh, Y, neg2(p1)));
  err = __ffma2_rn(wxl, X, err);
  err = __ffma2_rn(wyl, Y, err);
  const float2 s = add2(p0, p1);  // two_sum(p0, p1), then two_sum(s, b)
  float2 bb = sub2(s, p0);
  err = add2(err, add2(sub2(p0, sub2(s, bb)), sub2(p1, bb)));
  const float2 u = add2(s, bh);
  bb = sub2(u, s);
  err = add2(err, add2(sub2(s, sub2(u, bb)), sub2(bh, bb)));
  err = add2(err, bl);
  const float2 r = add2(u, err);
  return {r, sub2(err, sub2(r, u))};
}

// |w|^2 of a pair of float pairs, likewise with one gathered error.
__device__ __forceinline__ f2 f2_norm2(const f2x2& w) {
  const float2 p = __fmul2_rn(w.hi, w.hi);
  const float2 e = __ffma2_rn(w.hi, w.hi, neg2(p));
  const float2 t = __ffma2_rn(add2(w.hi, w.hi), w.lo, e);
  const f2 s = two_sum(p.x, p.y);
  return fast_two_sum(s.hi, __fadd_rn(__fadd_rn(t.x, t.y), s.lo));
}

// o 2^-q for q >= 0 as a float pair (about 1e-11 relative): q = k + j/64 + s,
// 2^-q = 2^-k * 2^(-j/64) * e^(-s ln 2) with a degree-4 Taylor polynomial of
// e^-x for x = s ln 2 in [0, ln2/64) (truncation below 1.3e-12).  x and the
// product with the table stay unnormalised (hi, lo) pairs; the polynomial
// takes x's low part to first order.
__device__ __forceinline__ f2 f2_exp2_neg(f2 q, float o, const float2* __restrict__ tab) {
  const float k = floorf(q.hi);
  const float r = q.hi - k;                        // exact
  const float jf = floorf(r * 64.f);
  const float s = r - jf * (1.f / 64.f);           // exact (Sterbenz)
  const f2 t = fast_two_sum(s, q.lo);              // s is 0 or a multiple of ulp(q.hi)
  const f2 ln2 = FS_F2C(kLn2D);
  const float xh = __fmul_rn(t.hi, ln2.hi);
  float xl = __fmaf_rn(t.hi, ln2.hi, -xh);
  xl = __fmaf_rn(t.hi, ln2.lo, xl);
  xl = __fmaf_rn(t.lo, ln2.hi, xl);
  float p = xh * xh * fmaf(xh, fmaf(xh, 1.f / 24.f, -1.f / 6.f), 0.5f);
  p = __fmaf_rn(xh, xl, p);
  const f2 e0 = fast_two_sum(1.f, -xh);
  const f2 e1 = fast_two_sum(e0.hi, p);
  const float el = __fadd_rn(e1.lo, __fsub_rn(e0.lo, xl));
  const float2 tj = tab[static_cast<int>(jf)];
  const float mh = __fmul_rn(e1.hi, tj.x);
  float ml = __fmaf_rn(e1.hi, tj.x, -mh);
  ml = __fmaf_rn(e1.hi, tj.y, ml);
  ml = __fmaf_rn(el, tj.x, ml);
  const float os = o * __int_as_float((127 - static_cast<int>(k)) << 23);  // o 2^-k, k <= 126
  f2 a = two_prod(mh, os);
  a.lo = __fmaf_rn(ml, os, a.lo);
  return fast_two_sum(a.hi, a.lo);
}

// Staged list entries of one warp, one array per 16-byte part so that lanes that
// read different entries spread over the banks: W by columns (hi and lo parts),
// b = W (ctr - m) relative to the tile centre, the cut with slack, the opacity and the
// re-check row (-1: none).
struct Stage {
  float4 w_hi[kRound];
  float4 w_lo[kRound];
  float4 bq[kRound];  // (b0 hi, b1 hi, q_cut + slack, opacity)
  float2 b_lo[kRound];
  int j[kRound];
};

__device__ __forceinline__ void stage_entry(Stage& S, int e, const ProjRecord& r, float cx,
                                            float cy, int j) {
  const f2 w0 = {r.w_hi.x, r.w_lo.x}, w1 = {r.w_hi.y, r.w_lo.y};
  const f2 w2 = {r.w_hi.z, r.w_lo.z}, w3 = {r.w_hi.w, r.w_lo.w};
  // b = W (ctr - m) with the difference of the centre and the float-pair mean
  const f2 dx = f2_sub(f2_from(cx), f2{r.m.x, r.m.z});
  const f2 dy = f2_sub(f2_from(cy), f2{r.m.y, r.m.w});
  const f2 b0 = f2_add(f2_mul(w0, dx), f2_mul(w1, dy));
  const f2 b1 = f2_add(f2_mul(w2, dx), f2_mul(w3, dy));
  S.w_hi[e] = make_float4(r.w_hi.x, r.w_hi.z, r.w_hi.y, r.w_hi.w);
  S.w_lo[e] = make_float4(r.w_lo.x, r.w_lo.z, r.w_lo.y, r.w_lo.w);
  // near the cut the FP32 screen |W_hi l + b_hi|^2 is off by far less than 0.05
  S.bq[e] = make_float4(b0.hi, b1.hi, r.misc.y + 0.05f, r.misc.x);
  S.b_lo[e] = make_float2(b0.lo, b1.lo);
  S.j[e] = j;
}

// Reduced-precision record: W16 and the FP32 mean are exact float values, so
// b = W (ctr - m) is formed from the exact difference in float pairs.
__device__ __forceinline__ void stage_compact(Stage& S, int e, const CompactRecord& r, float o,
                                              float cx, float cy, int j) {
  const float2 wa = __half22float2(*reinterpret_cast<const __half2*>(&r.w01));
  const float2 wb = __half22float2(*reinterpret_cast<const __half2*>(&r.w23));
  const f2 dx = two_sum(cx, -r.mx), dy = two_sum(cy, -r.my);
  const f2 b0 = f2_add(f2_mul_f(dx, wa.x), f2_mul_f(dy, wa.y));
  const f2 b1 = f2_add(f2_mul_f(dx, wb.x), f2_mul_f(dy, wb.y));
  S.w_hi[e] = make_float4(wa.x, wb.x, wa.y, wb.y);
  S.w_lo[e] = make_float4(0.f, 0.f, 0.f, 0.f);
  S.bq[e] = make_float4(b0.hi, b1.hi, fmaxf(log2f(255.f * o), 0.f) * 1.001f + 1e-3f + 0.05f, o);
  S.b_lo[e] = make_float2(b0.lo, b1.lo);
  S.j[e] = j;
}

// FP32 screen: can the entry's alpha >= 1/255 region reach this pixel?
__device__ __forceinline__ bool reaches(const Stage& S, int e, float lx, float ly) {
  const float4 w = S.w_hi[e], b = S.bq[e];
  const float2 q = __ffma2_rn(make_float2(w.x, w.y), make_float2(lx, lx),
                              __ffma2_rn(make_float2(w.z, w.w), make_float2(ly, ly),
                                         make_float2(b.x, b.y)));
  return fmaf(q.x, q.x, q.y * q.y) <= b.z;
}

// alpha of one (pixel, staged entry) pair, clamped: a float pair.
__device__ __forceinline__ f2 pair_alpha(const Stage& S, int e, float lx, float ly,
                                         const float2* __restrict__ tab) {
  const float4 wh = S.w_hi[e], wl = S.w_lo[e], bq = S.bq[e];
  const float2 bl = S.b_lo[e];
  const f2x2 w = f2x2_rows(make_float2(wh.x, wh.y), make_float2(wl.x, wl.y),
                           make_float2(wh.z, wh.w), make_float2(wl.z, wl.w),
                           make_float2(bq.x, bq.y), bl, lx, ly);
  const f2 a_max = FS_F2C(kAlphaMaxD);
  const f2 a = f2_exp2_neg(f2_norm2(w), bq.w, tab);
  return f2_lt(a_max, a) ? a_max : a;
}

// list[1 + k] (k < list[0]): view << 24 | tile of every tile whose skip bit
// is clear, in no particular order.
__global__ void __launch_bounds__(256) collect_tiles_kernel(const ViewParams* __restrict__ views,
                                                            const uint64_t* __restrict__ skip,
                                                            uint32_t* __restrict__ count,
                                                            uint32_t* __restrict__ list) {
  const ViewParams& vp = views[blockIdx.y];
  const int tile = static_cast<int>(blockIdx.x * blockDim.x + threadIdx.x);
  if (tile >= vp.tiles_x * vp.tiles_y) return;
  const int g = vp.tile_base + tile;
  if ((skip[g >> 6] >> (g & 63)) & 1ull) return;
  list[atomicAdd(count, 1u)] = (blockIdx.y << 24) | static_cast<uint32_t>(tile);
}

// Composites again the pixels that a re-checked Gaussian contributes to, in
// float pairs, front to back, until the last one's contribution or the stop.
// A work item is an 8x4-pixel piece of a listed tile; every warp of the grid
// takes items from a counter until none is left, and no warp waits for
// another.
//
// Bound by the ~130 FP32 operations of a (pixel, entry) pair and by the
// latency of the list and record gathers ahead of them.  An entry covers only
// some of a warp's pixels, and few pieces of a tile hold a pixel to re-check,
// so
//  * a piece first counts, per pixel, the re-checked Gaussians that
//    contribute (the exact alpha test); without one it is done;
//  * the tile's list is read 32 entries at a time, one per lane, and the
//    slots that can reach the piece's rectangle go to the warp's ring (a
//    plain FP32 test); 32 of them at a time are staged as float pairs, so that
//    every lane has one to stage;
//  * a pixel then screens the 32 into a bit mask and walks its own bits: lanes
//    work on different entries at the same time, and a round takes as many
//    steps as its busiest pixel has entries, not as many as its pixels have
//    between them.
// With more than kFlagTest re-checked Gaussians the count walks the tile's
// lists for them.  With more than one in kCountShare, whose last one lies near
// a pixel's stop anyway, and in deep tiles, every labelled pixel is walked to
// its stop instead.  (10^6 Gaussians in 24 views 1008x756, re-check stage in ms
// counted | walked: 300 re-checked 5.4 | 5.7, 3,000 7.1 | 7.6, 20,000 10.6 |
// 10.1; faint ones, which stop no pixel: 300 27.0 | 40.9, 2,000 41.7 | 46.3.)
template <typename LabelT>
__global__ void __launch_bounds__(32 * kRWarps, 8) recheck_blend_kernel(
    const ViewParams* __restrict__ views, RecheckLists L, const uint32_t* __restrict__ n_tiles,
    const uint32_t* __restrict__ tiles, uint32_t* __restrict__ ticket,
    const ProjRecord* __restrict__ rec, const CompactRecord* __restrict__ rec16,
    const float4* __restrict__ pos_op, int64_t n, int E, const int32_t* __restrict__ map,
    double* __restrict__ R, unsigned long long* __restrict__ counters) {
  __shared__ Stage s_stage[kRWarps];
  __shared__ uint32_t s_ring[kRWarps][kRing];
  __shared__ float2 s_tab[64];
  const int lane = threadIdx.x & 31;
  Stage& S = s_stage[threadIdx.x >> 5];
  uint32_t* const ring = s_ring[threadIdx.x >> 5];
  if (threadIdx.x < 64) {
    const double d = exp2(-static_cast<double>(threadIdx.x) / 64.0);
    const float hi = static_cast<float>(d);
    s_tab[threadIdx.x] = make_float2(hi, static_cast<float>(d - static_cast<double>(hi)));
  }
  __syncthreads();
  const uint32_t n_items = kSubs * *n_tiles;
  const uint32_t lt = (1u << lane) - 1u;
  const f2 a_min = FS_F2C(kAlphaMinD), t_min = FS_F2C(kTMinD);
  unsigned long long evals = 0;
  for (;;) {
    uint32_t item = 0u;
    if (lane == 0) item = atomicAdd(ticket, 1u);
    item = __shfl_sync(0xffffffffu, item, 0);
    if (item >= n_items) break;
    const uint32_t vt = tiles[item / kSubs];
    const int view = static_cast<int>(vt >> 24), tile = static_cast<int>(vt & 0xFFFFFFu);
    const int sub = static_cast<int>(item % kSubs);
    const ViewParams& vp = views[view];
    const int gtile = vp.tile_base + tile;
    const int tx = tile % vp.tiles_x, ty = tile / vp.tiles_x;
    const int x = tx * kTile + 8 * (sub & 1) + (lane & 7);
    const int y = ty * kTile + 4 * (sub >> 1) + (lane >> 3);
    int label = -1;
    if (x < vp.width && y < vp.height) {
      const int l = static_cast<int>(
          static_cast<const LabelT*>(vp.mask)[static_cast<int64_t>(y) * vp.width + x]);
      if (l >= 0 && l < E) label = l;
    }
    if (!__any_sync(0xffffffffu, label >= 0)) continue;
    const float cx = static_cast<float>(tx * kTile) + 0.5f * kTile;
    const float cy = static_cast<float>(ty * kTile) + 0.5f * kTile;
    // pixel centre (x + 0.5, y + 0.5) and the piece's centre relative to the
    // tile centre: exact
    const float lx = static_cast<float>(x) + 0.5f - cx, ly = static_cast<float>(y) + 0.5f - cy;
    const float rx = 8.f * static_cast<float>(sub & 1) - 4.f;
    const float ry = 4.f * static_cast<float>(sub >> 1) - 6.f;
    const uint32_t slot0 = static_cast<uint32_t>(static_cast<int64_t>(view) * n);

    // can the slot reach one of the piece's pixel centres?  (FP32: the rows'
    // products are off by less than 2^-21 of their terms' sizes, which is taken
    // off them, so that means any distance away lose no pixel; the rest is
    // within the slack of the per-pixel screen)
    auto meets = [&](uint32_t slot) -> bool {
      float4 w;
      float bx, by, qc;
      if (rec16) {
        const CompactRecord r = rec16[slot];
        const float2 wa = __half22float2(*reinterpret_cast<const __half2*>(&r.w01));
        const float2 wb = __half22float2(*reinterpret_cast<const __half2*>(&r.w23));
        w = make_float4(wa.x, wa.y, wb.x, wb.y);
        bx = (cx + rx) - r.mx;
        by = (cy + ry) - r.my;
        qc = r.q_cut;
      } else {
        const ProjRecord& r = rec[slot];
        const float4 m = r.m;
        w = r.w_hi;
        bx = ((cx + rx) - m.x) - m.z;
        by = ((cy + ry) - m.y) - m.w;
        qc = r.misc.y;
      }
      const float rel = 0x1p-21f;
      const float sx = fmaf(rel, fabsf(bx), 3.5f), sy = fmaf(rel, fabsf(by), 1.5f);
      const float d0 = fmaxf(0.f, fabsf(fmaf(w.x, bx, w.y * by)) -
                                      fmaf(fabsf(w.x), sx, fabsf(w.y) * sy));
      const float d1 = fmaxf(0.f, fabsf(fmaf(w.z, bx, w.w * by)) -
                                      fmaf(fabsf(w.z), sx, fabsf(w.w) * sy));
      return fmaf(d0, d0, d1 * d1) <= qc + 0.05f;
    };
    // ring entries first .. first + count - 1 into the stage, one per lane
    auto stage = [&](int first, int count) {
      if (lane < count) {
        const uint32_t slot = ring[(first + lane) & (kRing - 1)];
        const int j = map[slot - slot0];
        if (rec16)
          stage_compact(S, lane, rec16[slot], pos_op[slot - slot0].w, cx, cy, j);
        else
          stage_entry(S, lane, rec[slot], cx, cy, j);
      }
      __syncwarp();
    };
    // appends the lanes' slots that are kept at ring position `at`
    auto append = [&](bool keep, uint32_t slot, int at) -> int {
      const uint32_t bal = __ballot_sync(0xffffffffu, keep);
      if (keep) ring[(at + __popc(bal & lt)) & (kRing - 1)] = slot;
      __syncwarp();
      return __popc(bal);
    };

    const int n_chunks =
        L.sat_chunk ? min(L.chunks, static_cast<int>(L.sat_chunk[gtile]) + 1) : L.chunks;
    const bool deep = L.deep && ((L.deep[gtile >> 6] >> (gtile & 63)) & 1ull);
    // the re-checked Gaussians that contribute at each pixel: of those whose
    // footprint lists this tile, the ones with alpha >= 1/255.  Where they are
    // many they are found in the tile's lists, which hold them all unless the
    // tile is deep.
    int left = 0;
    if (L.n_flagged <= kFlagTest) {
      for (int k0 = 0; k0 < L.n_flagged; k0 += 32) {
        bool on = k0 + lane < L.n_flagged;
        const uint32_t slot = slot0 + (on ? L.flagged[k0 + lane] : 0u);
        on = on && box_visible(L.box[slot]);
        if (on) {
          const Footprint f = L.foot[slot];
          int r0, r1, c0, c1;
          footprint_rows(f, &r0, &r1);
          on = ty >= r0 && ty <= r1 && row_span(f, ty, vp.width, &c0, &c1) &&
               clip_cols(vp.cols, slot, &c0, &c1) && tx >= c0 && tx <= c1;
        }
        const int m = append(on && meets(slot), slot, 0);
        stage(0, m);
        if (label >= 0)
          for (int e = 0; e < m; ++e)
            if (reaches(S, e, lx, ly) && !f2_lt(pair_alpha(S, e, lx, ly, s_tab), a_min)) ++left;
        __syncwarp();
      }
    } else if (deep || static_cast<int64_t>(L.n_flagged) * kCountShare > n) {
      if (label >= 0) left = 0x7FFFFFFF;
    } else {
      int head = 0, queued = 0;
      auto count = [&](int first, int m) {
        stage(first, m);
        if (label >= 0)
          for (int e = 0; e < m; ++e)
            if (reaches(S, e, lx, ly) && !f2_lt(pair_alpha(S, e, lx, ly, s_tab), a_min)) ++left;
        __syncwarp();
      };
      for (int c = 0; c < n_chunks; ++c) {
        const uint2 rg = L.ranges[c][gtile];
        const uint32_t* __restrict__ val = L.val[c];
        for (uint32_t b0 = rg.x; b0 < rg.y; b0 += 32) {
          const uint32_t slot = b0 + lane < rg.y ? val[b0 + lane] : slot0;
          const bool on = b0 + lane < rg.y && map[slot - slot0] >= 0;
          queued += append(on && meets(slot), slot, head + queued);
          if (queued >= kRound) {
            count(head, kRound);
            head += kRound;
            queued -= kRound;
          }
        }
      }
      if (queued > 0) count(head, queued);
    }

    f2 T = f2_from(1.f);
    // one round: `count` kept entries from ring position `first` on
    auto composite = [&](int first, int count) {
      stage(first, count);
      uint32_t m = 0u;
      if (left > 0) {
#pragma unroll 8
        for (int k = 0; k < kRound; ++k) m |= reaches(S, k, lx, ly) ? 1u << k : 0u;
        if (count < kRound) m &= (1u << count) - 1u;
      }
      evals += __popc(m);
      while (m) {
        const int e = __ffs(m) - 1;
        m &= m - 1u;
        const f2 a = pair_alpha(S, e, lx, ly, s_tab);
        if (f2_lt(a, a_min)) continue;
        // T (1 - a): 1 - a needs no normalisation for the product
        const f2 om = fast_two_sum(1.f, -a.hi);
        f2 t = two_prod(T.hi, om.hi);
        t.lo = __fmaf_rn(T.hi, __fsub_rn(om.lo, a.lo), __fmaf_rn(T.lo, om.hi, t.lo));
        t = fast_two_sum(t.hi, t.lo);
        if (f2_lt(t, t_min)) {
          left = 0;  // the pixel's stop
        } else {
          const int j = S.j[e];
          if (j >= 0) {
            const f2 ct = f2_mul(a, T);
            atomicAdd(&R[static_cast<int64_t>(j) * E + label],
                      static_cast<double>(ct.hi) + static_cast<double>(ct.lo));
            --left;
          }
          T = t;
        }
        if (left == 0) {
          evals -= __popc(m);  // not evaluated
          break;
        }
      }
      __syncwarp();
    };
    if (!__any_sync(0xffffffffu, left > 0)) continue;
    int head = 0, queued = 0;
    bool some = true;
    for (int c = 0; c < n_chunks && some; ++c) {
      const uint2 rg = L.ranges[c][gtile];
      const uint32_t* __restrict__ val = L.val[c];
      uint32_t next = rg.x + lane < rg.y ? val[rg.x + lane] : 0u;
      for (uint32_t b0 = rg.x; b0 < rg.y && some; b0 += 32) {
        const uint32_t slot = next;
        if (b0 + 32 + lane < rg.y) next = val[b0 + 32 + lane];
        queued += append(b0 + lane < rg.y && meets(slot), slot, head + queued);
        if (queued >= kRound) {
          composite(head, kRound);
          head += kRound;
          queued -= kRound;
          some = __any_sync(0xffffffffu, left > 0);
        }
      }
    }
    if (some && queued > 0) composite(head, queued);
    // still compositing where a deep tile's kept lists end: the exact walk
    // needs entries the main pass never listed
    if (n_chunks < L.chunks && deep && __any_sync(0xffffffffu, left > 0) && lane == 0)
      atomicAdd(&counters[kRecheckIncomplete], 1ull);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) evals += __shfl_xor_sync(0xffffffffu, evals, o);
  if (lane == 0 && evals) atomicAdd(&counters[kRecheckPairs], evals);
}

__global__ void add_rows_kernel(int64_t count, const double* __restrict__ src,
                                double* __restrict__ dst) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i < count) dst[i] += src[i];
}

inline unsigned blocks_for(int64_t n, int threads) {
  return static_cast<unsigned>((n + threads - 1) / threads);
}

}  // namespace

cudaError_t launch_flag_margin(int64_t n, const float* margin, float tau, uint32_t* flag,
                               cudaStream_t stream) {
  if (n == 0) return cudaSuccess;
  flag_margin_kernel<<<blocks_for(n, 256), 256, 0, stream>>>(n, margin, tau, flag);
  return cudaGetLastError();
}

cudaError_t launch_scatter_flagged(int64_t n, const uint32_t* flag, const uint32_t* offs,
                                   uint32_t* F, int32_t* map, cudaStream_t stream) {
  if (n == 0) return cudaSuccess;
  scatter_flagged_kernel<<<blocks_for(n, 256), 256, 0, stream>>>(n, flag, offs, F, map);
  return cudaGetLastError();
}

cudaError_t launch_mark_tiles(int64_t n_flagged, int v_begin, int n_views, int64_t n,
                              const uint32_t* F, const ViewParams* views, const TileBox* box,
                              const Footprint* foot, uint64_t* skip, uint32_t* visible,
                              const uint32_t* bound, int chunks, const ProjRecord* rec,
                              const CompactRecord* rec16, const uint32_t* dlo,
                              const uint8_t* sat_chunk, uint64_t* deep, cudaStream_t stream) {
  const int64_t total = n_flagged * n_views;
  if (total == 0) return cudaSuccess;
  mark_tiles_kernel<<<blocks_for(total, 256), 256, 0, stream>>>(
      n_flagged, v_begin, n_views, n, F, views, box, foot,
      reinterpret_cast<unsigned long long*>(skip),
      visible, bound, chunks, rec, rec16, dlo, sat_chunk,
      reinterpret_cast<unsigned long long*>(deep));
  return cudaGetLastError();
}

cudaError_t launch_add_rows(int64_t count, const double* src, double* dst, cudaStream_t stream) {
  if (count == 0) return cudaSuccess;
  add_rows_kernel<<<blocks_for(count, 256), 256, 0, stream>>>(count, src, dst);
  return cudaGetLastError();
}

cudaError_t launch_candidates(int64_t k_total, int64_t n, const ViewParams* views,
                              const TileBox* box, const Footprint* foot, const uint64_t* skip,
                              uint32_t* flag, cudaStream_t stream) {
  if (k_total == 0) return cudaSuccess;
  candidates_kernel<<<blocks_for(k_total, 256), 256, 0, stream>>>(k_total, n, views, box, foot,
                                                                  skip, flag);
  return cudaGetLastError();
}

cudaError_t launch_compact(int64_t k_total, const uint32_t* flag, const uint32_t* offs,
                           const ProjRecord* rec, const CompactRecord* rec16, uint32_t* out_key,
                           uint32_t* out_val, cudaStream_t stream) {
  if (k_total == 0) return cudaSuccess;
  compact_kernel<<<blocks_for(k_total, 256), 256, 0, stream>>>(k_total, flag, offs, rec, rec16,
                                                               out_key, out_val);
  return cudaGetLastError();
}

size_t recheck_tiles_bytes(int64_t total_tiles) {
  return 256 + static_cast<size_t>(total_tiles) * sizeof(uint32_t);
}

cudaError_t launch_recheck_blend(const ViewParams* views, int n_views, int max_tiles_per_view,
                                 const RecheckLists& lists, const uint64_t* skip, void* tiles_tmp,
                                 int n_sm, const ProjRecord* rec, const CompactRecord* rec16,
                                 const float4* pos_op, int64_t n, int E, int mask_dtype,
                                 const int32_t* map, double* R, unsigned long long* counters,
                                 cudaStream_t stream) {
  if (n_views == 0 || max_tiles_per_view == 0) return cudaSuccess;
  if (lists.chunks < 1 || lists.chunks > kMaxChunks) return cudaErrorInvalidValue;
  uint32_t* words = static_cast<uint32_t*>(tiles_tmp);  // [0] tiles listed, [1] items taken
  uint32_t* tiles = words + 64;
  cudaError_t e = cudaMemsetAsync(words, 0, 2 * sizeof(uint32_t), stream);
  if (e != cudaSuccess) return e;
  const dim3 grid(blocks_for(max_tiles_per_view, 256), static_cast<unsigned>(n_views));
  collect_tiles_kernel<<<grid, 256, 0, stream>>>(views, skip, words, tiles);
  // one full set of resident blocks, fewer when the batch has fewer pieces
  const int64_t items = static_cast<int64_t>(n_views) * max_tiles_per_view * kSubs;
  const unsigned blocks = static_cast<unsigned>(
      std::min<int64_t>(8 * static_cast<int64_t>(n_sm), (items + kRWarps - 1) / kRWarps));
  if (mask_dtype == 4)
    recheck_blend_kernel<uint8_t><<<blocks, 32 * kRWarps, 0, stream>>>(
        views, lists, words, tiles, words + 1, rec, rec16, pos_op, n, E, map, R, counters);
  else
    recheck_blend_kernel<int32_t><<<blocks, 32 * kRWarps, 0, stream>>>(
        views, lists, words, tiles, words + 1, rec, rec16, pos_op, n, E, map, R, counters);
  return cudaGetLastError();
}

}  // namespace fs
