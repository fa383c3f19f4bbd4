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
// chunk ("deep" tile), every pixel of the tile is walked to its stop, and a
// pixel still compositing at the end of the kept lists (the FP32 and the
// exact stop decisions differ there) is reported so the caller redoes the
// batch with the dedicated binning.
//
// alpha = o 2^-|W (p - m)|^2 from the float-pair whitening record of the
// projection; 2^-q follows Tang's table-driven method (ACM TOMS 15(2), 1989):
// a 64-entry table of 2^(-j/64) (computed in FP64) times a degree-4 Taylor
// polynomial of e^-x on the remaining [0, ln2/64).
#include <cuda_fp16.h>
#include <math.h>

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

// Position of slot a before-or-equal slot b in the batch's depth order:
// (depth key, view, low word of the depth, slot).
__device__ __forceinline__ bool order_le(uint32_t a, uint32_t b, int64_t n,
                                         const uint32_t* __restrict__ dkey,
                                         const uint32_t* __restrict__ dlo) {
  if (dkey[a] != dkey[b]) return dkey[a] < dkey[b];
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
__global__ void mark_tiles_kernel(int64_t n_flagged, int n_views, int64_t n,
                                  const uint32_t* __restrict__ F,
                                  const ViewParams* __restrict__ views,
                                  const uint32_t* __restrict__ cnt,
                                  const Footprint* __restrict__ foot,
                                  unsigned long long* __restrict__ skip,
                                  uint32_t* __restrict__ visible,
                                  const uint32_t* __restrict__ bound, int chunks,
                                  const uint32_t* __restrict__ dkey,
                                  const uint32_t* __restrict__ dlo,
                                  const uint8_t* __restrict__ sat_chunk,
                                  unsigned long long* __restrict__ deep) {
  const int64_t idx = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx >= n_flagged * n_views) return;
  const int v = static_cast<int>(idx / n_flagged);
  const int64_t slot = static_cast<int64_t>(v) * n + F[idx % n_flagged];
  if (!cnt[slot]) return;
  atomicAdd(visible, 1u);
  int my_chunk = 0;
  if (bound) {
    my_chunk = chunks - 1;
    for (int ci = 0; ci < chunks - 1; ++ci)
      if (bound[ci] != 0xFFFFFFFFu &&  // an empty chunk holds nothing
          order_le(static_cast<uint32_t>(slot), bound[ci], n, dkey, dlo)) {
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
    if (!row_span(f, ty, vp.width, &tx0, &tx1) || !clip_cols(vp, slot, &tx0, &tx1)) continue;
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
                                  const uint32_t* __restrict__ cnt,
                                  const Footprint* __restrict__ foot,
                                  const uint64_t* __restrict__ skip, uint32_t* __restrict__ flag) {
  const int64_t slot = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (slot >= k_total) return;
  uint32_t hit = 0;
  if (cnt[slot]) {
    const int v = static_cast<int>(slot / n);
    const ViewParams& vp = views[v];
    const Footprint f = foot[slot];
    int ty0, ty1;
    footprint_rows(f, &ty0, &ty1);
    for (int ty = ty0; ty <= ty1 && !hit; ++ty) {
      int tx0, tx1;
      if (!row_span(f, ty, vp.width, &tx0, &tx1) || !clip_cols(vp, slot, &tx0, &tx1)) continue;
      const int base = vp.tile_base + ty * vp.tiles_x;
      if (count_free(skip, base + tx0, base + tx1)) hit = 1;
    }
  }
  flag[slot] = hit;
}

__global__ void compact_kernel(int64_t k_total, const uint32_t* __restrict__ flag,
                               const uint32_t* __restrict__ offs,
                               const uint32_t* __restrict__ key_src,
                               uint32_t* __restrict__ out_key, uint32_t* __restrict__ out_val) {
  const int64_t slot = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (slot >= k_total || !flag[slot]) return;
  const uint32_t o = offs[slot];
  out_key[o] = key_src[slot];
  out_val[o] = static_cast<uint32_t>(slot);
}

constexpr int kRB = kTilePixels;  // list entries staged per step: one per thread
constexpr int kGroup = 64;        // staged entries screened at once per pixel (two mask words)
constexpr int kDeepTest = 256;  // re-checked Gaussians a deep tile tests per pixel at most

// Float-pair constants of the compositing rule (Sec. 3.1 Eq. 1 conventions).
constexpr double kAlphaMinD = 1.0 / 255.0, kAlphaMaxD = 0.99, kTMinD = 1e-4;
constexpr double kLn2D = 0.69314718055994530942;
#define FS_F2C(d) f2{static_cast<float>(d), static_cast<float>((d) - static_cast<double>(static_cast<float>(d)))}

// One row of w = W l + b at the pixel offset l (exact small half-integers) as
// a float pair: the products' and sums' rounding errors are gathered in one
// float and put back once (a compensated dot product, Ogita, Rump and Oishi
// 2005), about 25 operations where a chain of float-pair products and sums
// takes 34.
__device__ __forceinline__ f2 f2_row(float wh0, float wl0, float wh1, float wl1, float bh,
                                     float bl, float lx, float ly) {
  const f2 p0 = two_prod(wh0, lx), p1 = two_prod(wh1, ly);
  const f2 s = two_sum(p0.hi, p1.hi);
  const f2 u = two_sum(s.hi, bh);
  float err = __fadd_rn(p0.lo, p1.lo);
  err = __fmaf_rn(wl0, lx, err);
  err = __fmaf_rn(wl1, ly, err);
  err = __fadd_rn(err, s.lo);
  err = __fadd_rn(err, u.lo);
  err = __fadd_rn(err, bl);
  return fast_two_sum(u.hi, err);
}

// a^2 + b^2 of float pairs, likewise with one gathered error.
__device__ __forceinline__ f2 f2_norm2(f2 a, f2 b) {
  const f2 p0 = two_prod(a.hi, a.hi), p1 = two_prod(b.hi, b.hi);
  const f2 s = two_sum(p0.hi, p1.hi);
  float err = __fadd_rn(p0.lo, p1.lo);
  err = __fmaf_rn(a.hi + a.hi, a.lo, err);
  err = __fmaf_rn(b.hi + b.hi, b.lo, err);
  err = __fadd_rn(err, s.lo);
  return fast_two_sum(s.hi, err);
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

// Staged list entries, one array per 16-byte part so that lanes that read
// different entries spread over the banks: W (hi and lo parts), b = W (ctr - m)
// relative to the tile centre, the cut with slack, the opacity and the
// re-check row (-1: none).
struct Stage {
  float4 w_hi[kRB];
  float4 w_lo[kRB];
  float4 bq[kRB];  // (b0 hi, b1 hi, q_cut + slack, opacity)
  float2 b_lo[kRB];
  int j[kRB];
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
  S.w_hi[e] = r.w_hi;
  S.w_lo[e] = r.w_lo;
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
  S.w_hi[e] = make_float4(wa.x, wa.y, wb.x, wb.y);
  S.w_lo[e] = make_float4(0.f, 0.f, 0.f, 0.f);
  S.bq[e] = make_float4(b0.hi, b1.hi, fmaxf(log2f(255.f * o), 0.f) * 1.001f + 1e-3f + 0.05f, o);
  S.b_lo[e] = make_float2(b0.lo, b1.lo);
  S.j[e] = j;
}

// FP32 screen: can the entry's alpha >= 1/255 region reach this pixel?
__device__ __forceinline__ bool reaches(const Stage& S, int e, float lx, float ly) {
  const float4 w = S.w_hi[e], b = S.bq[e];
  const float q0 = fmaf(w.x, lx, fmaf(w.y, ly, b.x));
  const float q1 = fmaf(w.z, lx, fmaf(w.w, ly, b.y));
  return fmaf(q0, q0, q1 * q1) <= b.z;
}

// Bit k: staged entry e0 + k (k < 32, e0 + k < count) reaches the pixel.  The
// staging array is read past `count` (its old entries, masked off here).
__device__ __forceinline__ uint32_t reach_mask(const Stage& S, int e0, int count, float lx,
                                               float ly) {
  if (e0 >= count) return 0u;
  uint32_t m = 0u;
#pragma unroll 8
  for (int k = 0; k < 32; ++k) m |= reaches(S, e0 + k, lx, ly) ? 1u << k : 0u;
  return count - e0 >= 32 ? m : m & ((1u << (count - e0)) - 1u);
}

// One CTA per 16x16 tile of a view, one thread per pixel (warps of 8x4
// pixels).  Pass 1 finds, per pixel, the last list position holding a
// re-checked Gaussian that can reach the pixel; pass 2 composites the pixel
// in float pairs up to that position (deep tiles: up to its stop).
//
// The work is the ~130 FP32 operations of a (pixel, entry) pair, and an entry
// covers only some of a warp's pixels.  So a pixel first collects the staged
// entries that reach it, 64 at a time, in a bit mask (about ten operations an
// entry), and then walks its own bits: lanes work on different entries at the
// same time and a warp takes as many steps as its busiest pixel has entries,
// not as many as its pixels have between them.
template <typename LabelT>
__global__ void __launch_bounds__(kTilePixels, 4) recheck_blend_kernel(
    const ViewParams* __restrict__ views, RecheckLists L, const uint64_t* __restrict__ skip,
    const ProjRecord* __restrict__ rec, const CompactRecord* __restrict__ rec16,
    const float4* __restrict__ pos_op, int64_t n, int E, const int32_t* __restrict__ map,
    double* __restrict__ R, unsigned long long* __restrict__ counters) {
  __shared__ Stage S;
  __shared__ float2 s_tab[64];
  const ViewParams& vp = views[blockIdx.y];
  const int tile = blockIdx.x;
  if (tile >= vp.tiles_x * vp.tiles_y) return;
  const int gtile = vp.tile_base + tile;
  if ((skip[gtile >> 6] >> (gtile & 63)) & 1ull) return;
  const int n_chunks = L.sat_chunk ? min(L.chunks, static_cast<int>(L.sat_chunk[gtile]) + 1)
                                   : L.chunks;
  const bool truncated = n_chunks < L.chunks;
  const bool deep = L.deep && ((L.deep[gtile >> 6] >> (gtile & 63)) & 1ull);
  if (threadIdx.x < 64) {
    const double d = exp2(-static_cast<double>(threadIdx.x) / 64.0);
    const float hi = static_cast<float>(d);
    s_tab[threadIdx.x] = make_float2(hi, static_cast<float>(d - static_cast<double>(hi)));
  }
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int x0 = (tile % vp.tiles_x) * kTile, y0 = (tile / vp.tiles_x) * kTile;
  const int x = x0 + 8 * (warp & 1) + (lane & 7);
  const int y = y0 + 4 * (warp >> 1) + (lane >> 3);
  int label = -1;
  if (x < vp.width && y < vp.height) {
    const int l = static_cast<int>(
        static_cast<const LabelT*>(vp.mask)[static_cast<int64_t>(y) * vp.width + x]);
    if (l >= 0 && l < E) label = l;
  }
  const float cx = static_cast<float>(x0) + 0.5f * kTile;
  const float cy = static_cast<float>(y0) + 0.5f * kTile;
  // pixel centre (x + 0.5, y + 0.5) relative to the tile centre: exact
  const float lx = static_cast<float>(x - x0) + 0.5f - 0.5f * kTile;
  const float ly = static_cast<float>(y - y0) + 0.5f - 0.5f * kTile;
  // the slots of a view are view * n + index
  const uint32_t slot0 = static_cast<uint32_t>(static_cast<int64_t>(blockIdx.y) * n);
  auto stage = [&](uint32_t slot, int j) {
    if (rec16)
      stage_compact(S, tid, rec16[slot], pos_op[slot - slot0].w, cx, cy, j);
    else
      stage_entry(S, tid, rec[slot], cx, cy, j);
  };

  // pass 1: last re-checked entry (chunk << 32 | index) that may reach the
  // pixel.  Re-checked entries are rare: a step without one costs its loads
  // and one barrier.
  int64_t last = -1;
  for (int c = 0; c < n_chunks; ++c) {
    const uint2 rg = L.ranges[c][gtile];
    for (uint32_t b0 = rg.x; b0 < rg.y; b0 += kRB) {
      const uint32_t at = b0 + tid;
      const uint32_t slot = at < rg.y ? L.val[c][at] : slot0;
      const int j = at < rg.y ? map[slot - slot0] : -1;
      if (__syncthreads_or(j >= 0) == 0) continue;
      S.j[tid] = j;
      if (j >= 0) stage(slot, j);
      __syncthreads();
      if (label >= 0) {
        const int cnt = static_cast<int>(min(static_cast<uint32_t>(kRB), rg.y - b0));
        for (int e = 0; e < cnt; ++e)
          if (S.j[e] >= 0 && reaches(S, e, lx, ly)) last = (static_cast<int64_t>(c) << 32) | (b0 + e);
      }
      __syncthreads();
    }
  }

  // deep tiles: a pixel is walked to its stop only where a re-checked
  // Gaussian visible in this view can reach it (the others hold nothing to
  // re-check); with many re-checked Gaussians every labelled pixel is
  bool deep_px = deep;
  if (deep && L.flagged && L.n_flagged <= kDeepTest) {
    bool reached = false;
    for (int k0 = 0; k0 < L.n_flagged; k0 += kRB) {
      const int cnt = min(kRB, L.n_flagged - k0);
      __syncthreads();
      if (tid < cnt) {
        const uint32_t slot = slot0 + L.flagged[k0 + tid];
        S.j[tid] = -1;
        if (L.cnt[slot]) stage(slot, 0);
      }
      __syncthreads();
      for (int e = 0; e < cnt; ++e)
        if (S.j[e] >= 0 && reaches(S, e, lx, ly)) reached = true;
    }
    deep_px = reached;
  }

  // pass 2: float-pair compositing
  const f2 a_min = FS_F2C(kAlphaMinD), a_max = FS_F2C(kAlphaMaxD), t_min = FS_F2C(kTMinD);
  f2 T = f2_from(1.f);
  bool live = label >= 0 && (deep_px || last >= 0);
  const bool to_stop = deep_px;
  unsigned long long evals = 0;
  bool done_all = false;
  for (int c = 0; c < n_chunks && !done_all; ++c) {
    const uint2 rg = L.ranges[c][gtile];
    for (uint32_t b0 = rg.x; b0 < rg.y; b0 += kRB) {
      if (__syncthreads_or(live) == 0) {
        done_all = true;
        break;
      }
      const int cnt = static_cast<int>(min(static_cast<uint32_t>(kRB), rg.y - b0));
      if (tid < cnt) {
        const uint32_t slot = L.val[c][b0 + tid];
        stage(slot, map[slot - slot0]);
      }
      __syncthreads();
      // the pixel's entries of this step: all of them, or up to its last one
      const int64_t pos0 = (static_cast<int64_t>(c) << 32) | b0;
      const int e_end =
          to_stop ? cnt : static_cast<int>(min(static_cast<int64_t>(cnt), last - pos0 + 1));
      for (int g0 = 0; g0 < cnt; g0 += kGroup) {
        if (!__any_sync(0xffffffffu, live && g0 < e_end)) break;
        uint32_t m0 = 0u, m1 = 0u;
        if (live) {
          m0 = reach_mask(S, g0, e_end, lx, ly);
          m1 = reach_mask(S, g0 + 32, e_end, lx, ly);
        }
        evals += __popc(m0) + __popc(m1);
        while (m0 | m1) {
          int e = g0;
          if (m0) {
            e += __ffs(m0) - 1;
            m0 &= m0 - 1u;
          } else {
            e += 31 + __ffs(m1);
            m1 &= m1 - 1u;
          }
          const float4 wh = S.w_hi[e], wl = S.w_lo[e], bq = S.bq[e];
          const float2 bl = S.b_lo[e];
          const f2 w0 = f2_row(wh.x, wl.x, wh.y, wl.y, bq.x, bl.x, lx, ly);
          const f2 w1 = f2_row(wh.z, wl.z, wh.w, wl.w, bq.y, bl.y, lx, ly);
          f2 a = f2_exp2_neg(f2_norm2(w0, w1), bq.w, s_tab);
          if (f2_lt(a_max, a)) a = a_max;
          if (f2_lt(a, a_min)) continue;
          // T (1 - a): 1 - a needs no normalisation for the product
          const f2 om = fast_two_sum(1.f, -a.hi);
          f2 t = two_prod(T.hi, om.hi);
          t.lo = __fmaf_rn(T.hi, __fsub_rn(om.lo, a.lo), __fmaf_rn(T.lo, om.hi, t.lo));
          t = fast_two_sum(t.hi, t.lo);
          if (f2_lt(t, t_min)) {
            live = false;
            evals -= __popc(m0) + __popc(m1);  // not reached
            break;
          }
          const int j = S.j[e];
          if (j >= 0) {
            const f2 ct = f2_mul(a, T);
            atomicAdd(&R[static_cast<int64_t>(j) * E + label],
                      static_cast<double>(ct.hi) + static_cast<double>(ct.lo));
          }
          T = t;
        }
      }
      if (live && !to_stop && pos0 + cnt > last) live = false;
    }
  }
  // still compositing where a saturated tile's kept lists end: the exact
  // walk needs entries the main pass never listed
  const bool incomplete = live && truncated && to_stop;
  const int n_inc = __syncthreads_count(incomplete);
  if (threadIdx.x == 0 && n_inc) atomicAdd(&counters[kRecheckIncomplete], 1ull);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) evals += __shfl_xor_sync(0xffffffffu, evals, o);
  if ((threadIdx.x & 31) == 0 && evals) atomicAdd(&counters[kRecheckPairs], evals);
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

cudaError_t launch_mark_tiles(int64_t n_flagged, int n_views, int64_t n, const uint32_t* F,
                              const ViewParams* views, const uint32_t* cnt, const Footprint* foot,
                              uint64_t* skip, uint32_t* visible, const uint32_t* bound,
                              int chunks, const uint32_t* dkey, const uint32_t* dlo,
                              const uint8_t* sat_chunk, uint64_t* deep, cudaStream_t stream) {
  const int64_t total = n_flagged * n_views;
  if (total == 0) return cudaSuccess;
  mark_tiles_kernel<<<blocks_for(total, 256), 256, 0, stream>>>(
      n_flagged, n_views, n, F, views, cnt, foot, reinterpret_cast<unsigned long long*>(skip),
      visible, bound, chunks, dkey, dlo, sat_chunk, reinterpret_cast<unsigned long long*>(deep));
  return cudaGetLastError();
}

cudaError_t launch_add_rows(int64_t count, const double* src, double* dst, cudaStream_t stream) {
  if (count == 0) return cudaSuccess;
  add_rows_kernel<<<blocks_for(count, 256), 256, 0, stream>>>(count, src, dst);
  return cudaGetLastError();
}

cudaError_t launch_candidates(int64_t k_total, int64_t n, const ViewParams* views,
                              const uint32_t* cnt, const Footprint* foot, const uint64_t* skip,
                              uint32_t* flag, cudaStream_t stream) {
  if (k_total == 0) return cudaSuccess;
  candidates_kernel<<<blocks_for(k_total, 256), 256, 0, stream>>>(k_total, n, views, cnt, foot,
                                                                  skip, flag);
  return cudaGetLastError();
}

cudaError_t launch_compact(int64_t k_total, const uint32_t* flag, const uint32_t* offs,
                           const uint32_t* key_src, uint32_t* out_key, uint32_t* out_val,
                           cudaStream_t stream) {
  if (k_total == 0) return cudaSuccess;
  compact_kernel<<<blocks_for(k_total, 256), 256, 0, stream>>>(k_total, flag, offs, key_src,
                                                               out_key, out_val);
  return cudaGetLastError();
}

cudaError_t launch_recheck_blend(const ViewParams* views, int n_views, int max_tiles_per_view,
                                 const RecheckLists& lists, const uint64_t* skip,
                                 const ProjRecord* rec, const CompactRecord* rec16,
                                 const float4* pos_op, int64_t n, int E, int mask_dtype,
                                 const int32_t* map, double* R, unsigned long long* counters,
                                 cudaStream_t stream) {
  if (n_views == 0 || max_tiles_per_view == 0) return cudaSuccess;
  if (lists.chunks < 1 || lists.chunks > kMaxChunks) return cudaErrorInvalidValue;
  const dim3 grid(static_cast<unsigned>(max_tiles_per_view), static_cast<unsigned>(n_views));
  if (mask_dtype == 4)
    recheck_blend_kernel<uint8_t><<<grid, kTilePixels, 0, stream>>>(
        views, lists, skip, rec, rec16, pos_op, n, E, map, R, counters);
  else
    recheck_blend_kernel<int32_t><<<grid, kTilePixels, 0, stream>>>(
        views, lists, skip, rec, rec16, pos_op, n, E, map, R, counters);
  return cudaGetLastError();
}

}  // namespace fs
