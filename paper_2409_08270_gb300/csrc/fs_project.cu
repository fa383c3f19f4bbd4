// Scene preparation, EWA projection and tile binning (Sec. 3.1).
//
// Projection of Gaussian i into view v, in float-pair arithmetic (about 48
// significant bits, no FP64 pipe):
//   t = R m + t_c                              (compensated dot product)
//   m2D = (fx tx/tz + cx, fy ty/tz + cy)
//   J = perspective Jacobian at t, tx/tz and ty/tz clamped to 1.3 tan(fov/2)
//   Sigma2D = (J W) Sigma3D (J W)^T + 0.3 I,   W = camera rotation
//   Sigma2D = lambda1 e e^T + lambda2 e' e'^T  (lambda2 = det / lambda1)
// The record stores the whitening matrix W_ws = sqrt(0.5 log2 e)
// diag(lambda1, lambda2)^-1/2 [e e']^T and the mean m2D as float pairs (hi,
// lo), so alpha = o 2^-|W_ws (p - m2D)|^2.  Carrying the eigenvectors
// to ~1e-14 keeps thin ("needle") Gaussians correctly oriented: an FP32
// orientation error of 1e-7 rad moves alpha at the tip of a 4500:1 Gaussian
// by ~1e-4.  Sigma3D = R(q) diag(s^2) R(q)^T is formed once per scene in FP64
// and kept as float pairs.
//
// Binning: a tile is listed for a Gaussian when its pixel centres, widened
// by one pixel, can meet the alpha >= 1/255 ellipse {d^T Sigma2D^-1 d <= r2},
// r2 = 2 ln(255 o) (slightly inflated).  For every tile row the x-extent of
// the ellipse over that row's band is exact (the boundary's extreme points),
// so far fewer tiles are listed than with the bounding box.
#include <cuda_fp16.h>

#include <algorithm>

#include "fs_binning.cuh"
#include "fs_common.cuh"
#include "fs_compact.cuh"
#include "fs_internal.h"

namespace fs {

// ---------------------------------------------------------------------------
// scene preparation: covariance in FP64 (once), packed attributes, validation
// ---------------------------------------------------------------------------

__device__ __forceinline__ float load_attr(const void* p, int64_t idx, int dtype) {
  if (dtype == 0) return static_cast<const float*>(p)[idx];
  const uint16_t bits = static_cast<const uint16_t*>(p)[idx];
  if (dtype == 2) return __uint_as_float(static_cast<uint32_t>(bits) << 16);  // bf16
  return __half2float(__ushort_as_half(bits));                                 // fp16
}

__device__ __forceinline__ void split_d(double x, float* hi, float* lo) {
  const float h = static_cast<float>(x);
  *hi = h;
  *lo = static_cast<float>(x - static_cast<double>(h));
}

__global__ void scene_prep_kernel(int64_t n, const float* __restrict__ mean, const void* quat,
                                  int quat_dtype, const void* scale, int scale_dtype,
                                  const void* opacity, int opacity_dtype, float4* __restrict__ pos_op,
                                  float4* __restrict__ cov, unsigned int* __restrict__ err) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float mx = mean[3 * i], my = mean[3 * i + 1], mz = mean[3 * i + 2];
  const float o = load_attr(opacity, i, opacity_dtype);
  const float q0 = load_attr(quat, 4 * i, quat_dtype), q1 = load_attr(quat, 4 * i + 1, quat_dtype);
  const float q2 = load_attr(quat, 4 * i + 2, quat_dtype), q3 = load_attr(quat, 4 * i + 3, quat_dtype);
  const float s0 = load_attr(scale, 3 * i, scale_dtype), s1 = load_attr(scale, 3 * i + 1, scale_dtype);
  const float s2 = load_attr(scale, 3 * i + 2, scale_dtype);
  bool bad = !(isfinite(mx) && isfinite(my) && isfinite(mz) && isfinite(o) && isfinite(q0) &&
               isfinite(q1) && isfinite(q2) && isfinite(q3) && isfinite(s0) && isfinite(s1) &&
               isfinite(s2));
  const double nn = (double)q0 * q0 + (double)q1 * q1 + (double)q2 * q2 + (double)q3 * q3;
  if (!(nn > 0.0)) bad = true;
  if (bad) {
    atomicOr(err, 1u);
    pos_op[i] = make_float4(0.f, 0.f, -1e30f, 0.f);
    cov[3 * i] = cov[3 * i + 1] = cov[3 * i + 2] = make_float4(0.f, 0.f, 0.f, 0.f);
    return;
  }
  // Sigma3D = Rq diag(s^2) Rq^T in FP64 (once per scene)
  const double inv = 1.0 / sqrt(nn);
  const double w = q0 * inv, x = q1 * inv, y = q2 * inv, z = q3 * inv;
  double Rq[3][3];
  Rq[0][0] = 1.0 - 2.0 * (y * y + z * z);
  Rq[0][1] = 2.0 * (x * y - w * z);
  Rq[0][2] = 2.0 * (x * z + w * y);
  Rq[1][0] = 2.0 * (x * y + w * z);
  Rq[1][1] = 1.0 - 2.0 * (x * x + z * z);
  Rq[1][2] = 2.0 * (y * z - w * x);
  Rq[2][0] = 2.0 * (x * z - w * y);
  Rq[2][1] = 2.0 * (y * z + w * x);
  Rq[2][2] = 1.0 - 2.0 * (x * x + y * y);
  const double sq[3] = {(double)s0 * s0, (double)s1 * s1, (double)s2 * s2};
  const int ia[6] = {0, 0, 0, 1, 1, 2}, ib[6] = {0, 1, 2, 1, 2, 2};
  float h[6], lo[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    double acc = 0.0;
    for (int l = 0; l < 3; ++l) acc += Rq[ia[k]][l] * sq[l] * Rq[ib[k]][l];
    split_d(acc, &h[k], &lo[k]);
  }
  pos_op[i] = make_float4(mx, my, mz, o);
  // (s00, s01, s02, s11, s12, s22) as (hi, lo) pairs
  cov[3 * i] = make_float4(h[0], lo[0], h[1], lo[1]);
  cov[3 * i + 1] = make_float4(h[2], lo[2], h[3], lo[3]);
  cov[3 * i + 2] = make_float4(h[4], lo[4], h[5], lo[5]);
}

// ---------------------------------------------------------------------------
// projection
// ---------------------------------------------------------------------------

__device__ __forceinline__ bool f2_greater(f2 a, float b_hi, float b_lo) {
  return a.hi > b_hi || (a.hi == b_hi && a.lo > b_lo);
}

__device__ __forceinline__ f2 f2_clamp(f2 x, float lim_hi, float lim_lo) {
  const f2 lim = {lim_hi, lim_lo}, nlim = {-lim_hi, -lim_lo};
  if (f2_lt(x, nlim)) return nlim;
  if (f2_lt(lim, x)) return lim;
  return x;
}

// One thread per Gaussian; it projects the Gaussian into the views of its
// block's share (all of them for large scenes, so the scene is read once per
// batch; small scenes spread the views over the grid's second dimension).
// rec16 != NULL: the record is written in the reduced-precision form instead
// (rec is not written).  The paired float-pair quantities (the two rows of the
// Jacobian-rotation product, the two rows of T Sigma3D, the x and y halves of
// the pinhole map, the rows of W) run in packed FP32 (f2x2), bit-identical to
// the scalar form.  Three blocks per SM (80 registers) spill less than four.
// Bound by issue (about 1,100 instructions a slot): one reciprocal and four
// roots, seeded by the hardware's, where six correctly rounded float-pair
// divisions and four roots stood, take 10^6 Gaussians in 100 views from 4.44 to
// 3.74 ms.
template <bool kFast>
__global__ void __launch_bounds__(256, kFast ? 4 : 3) project_kernel(
    int64_t n, int n_views, const ViewParams* __restrict__ views_g,
    const float4* __restrict__ pos_op, const float4* __restrict__ cov3,
    ProjRecord* __restrict__ rec, CompactRecord* __restrict__ rec16, Footprint* __restrict__ foot,
    TileBox* __restrict__ box, uint32_t* __restrict__ key, uint32_t* __restrict__ depth_lo,
    uint32_t* __restrict__ key_range) {
  __shared__ ViewParams views[kMaxViewsPerBatch];
  for (int k = threadIdx.x; k < n_views * (int)(sizeof(ViewParams) / 4); k += blockDim.x)
    reinterpret_cast<uint32_t*>(views)[k] = reinterpret_cast<const uint32_t*>(views_g)[k];
  __syncthreads();
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  uint32_t kmin = 0xFFFFFFFFu, kmax = 0u;  // visible depth keys of this thread
  uint32_t n_vis = 0;                       // and their number
  if (i < n) {
  const float4 po = pos_op[i];
  const float4 ca = cov3[3 * i], cb = cov3[3 * i + 1], cc = cov3[3 * i + 2];
  const f2 S00 = {ca.x, ca.y}, S01 = {ca.z, ca.w}, S02 = {cb.x, cb.y};
  const f2 S11 = {cb.z, cb.w}, S12 = {cc.x, cc.y}, S22 = {cc.z, cc.w};
  const f2 S[3][3] = {{S00, S01, S02}, {S01, S11, S12}, {S02, S12, S22}};
  const float o = po.w;
  const bool opaque_enough = o >= kAlphaMin;
  const float r2 = opaque_enough ? fmaxf(2.f * logf(255.f * o), 0.f) : 0.f;
  const float nlo = opaque_enough ? -log2f(o) : 0.f;  // alpha = 2^-(|w|^2 - log2 o)

  // the block's share of the views
  const int v_end = static_cast<int>((blockIdx.y + 1) * n_views / gridDim.y);
  for (int v = static_cast<int>(blockIdx.y * n_views / gridDim.y); v < v_end; ++v) {
    const ViewParams& vp = views[v];
    const int64_t slot = static_cast<int64_t>(v) * n + i;
    const f2x2 txy = f2x2_dot3_add(vp.R_hi + 0, vp.R_lo + 0, vp.R_hi + 3, vp.R_lo + 3, po.x, po.y,
                                   po.z, make_float2(vp.t_hi[0], vp.t_hi[1]),
                                   make_float2(vp.t_lo[0], vp.t_lo[1]));
    const f2 tx = f2x2_first(txy), ty = f2x2_second(txy);
    const f2 tz = f2_dot3_add(vp.R_hi + 6, vp.R_lo + 6, po.x, po.y, po.z, vp.t_hi[2], vp.t_lo[2]);
    bool visible = opaque_enough && f2_greater(tz, vp.near_hi, vp.near_lo);
    float depth = 0.f, depth_l = 0.f;
    ProjRecord R;
    R.w_hi = R.w_lo = R.m = make_float4(0.f, 0.f, 0.f, 0.f);
    CompactRecord R16 = {0.f, 0.f, 0u, 0u, 0.f, 0.f, 0.f, 0.f};
    // misc.y: |w|^2 at which alpha falls to 1/255, log2(255 o), widened by
    // 0.1% + 1e-3 so the blend's sub-tile test stays conservative in FP32
    const float qcut = opaque_enough ? fmaxf(log2f(255.f * o), 0.f) * 1.001f + 1e-3f : 0.f;
    R.misc = make_float4(o, qcut, nlo, 0.f);
    R16.o = o;
    R16.q_cut = qcut;
    R16.nlo = nlo;
    Footprint F;
    F.mx = F.my = F.hy = F.syr = F.dys = F.a = F.b2 = 0.f;
    F.rows = 0x0000FFFFu;  // no tile row (first row 65535 > last row 0)
    uint32_t col_clip = kNoBox;       // 3-sigma coverage: no tile column
    TileBox bx = make_uint2(kNoBox, kNoBox);
    if (visible) {
      float sxx, sxy, syy, det32, mx32, my32;  // 2D covariance and mean for the footprint
      if constexpr (kFast) {
        // reduced-precision form: the record keeps an FP16 W and an FP32
        // mean, so the 2D covariance, its eigen-decomposition and W run in
        // plain FP32 (correctly rounded divisions and roots); the depth stays
        // a float pair for the order
        depth = tz.hi;
        depth_l = tz.lo;
        R16.depth = depth;
        const float iz = __fdiv_rn(1.f, tz.hi);
        const float uxf = __fmul_rn(tx.hi, iz), uyf = __fmul_rn(ty.hi, iz);
        mx32 = fmaf(vp.fx_hi, uxf, vp.cx_hi);
        my32 = fmaf(vp.fy_hi, uyf, vp.cy_hi);
        const float jx = vp.fx_hi * iz, jy = vp.fy_hi * iz;
        const float ucx = fminf(fmaxf(uxf, -vp.limx_hi), vp.limx_hi);
        const float ucy = fminf(fmaxf(uyf, -vp.limy_hi), vp.limy_hi);
        float T0[3], T1[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          T0[k] = jx * fmaf(-ucx, vp.R_hi[6 + k], vp.R_hi[k]);
          T1[k] = jy * fmaf(-ucy, vp.R_hi[6 + k], vp.R_hi[3 + k]);
        }
        float a = 0.f, b = 0.f, c = 0.f;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const float m0 = fmaf(T0[0], S[0][j].hi, fmaf(T0[1], S[1][j].hi, T0[2] * S[2][j].hi));
          const float m1 = fmaf(T1[0], S[0][j].hi, fmaf(T1[1], S[1][j].hi, T1[2] * S[2][j].hi));
          a = fmaf(m0, T0[j], a);
          c = fmaf(m1, T1[j], c);
          b = fmaf(m0, T1[j], b);
        }
        a += kLowPass;
        c += kLowPass;
        // a c - b^2 with the rounding error of b^2 put back (Kahan)
        const float bb = b * b;
        const float dt = fmaf(a, c, -bb) - fmaf(b, b, -bb);
        const float h = 0.5f * (a - c);
        const float rr = __fsqrt_rn(fmaf(h, h, bb));
        const float lam1 = 0.5f * (a + c) + rr;
        const float lam2 = __fdiv_rn(dt, lam1);
        float ex, ey;
        if (h >= 0.f) {
          ex = h + rr;
          ey = b;
        } else {
          ex = b;
          ey = rr - h;
        }
        const float en = __fsqrt_rn(fmaf(ex, ex, ey * ey));
        if (en > 0.f) {
          ex = __fdiv_rn(ex, en);
          ey = __fdiv_rn(ey, en);
        } else {
          ex = 1.f;
          ey = 0.f;
        }
        const float k1 = __fsqrt_rn(__fdiv_rn(kHalfLog2eHi, lam1));
        const float k2 = __fsqrt_rn(__fdiv_rn(kHalfLog2eHi, lam2));
        R16.mx = mx32;
        R16.my = my32;
        R16.w01 = static_cast<uint32_t>(__half_as_ushort(__float2half_rn(ex * k1))) |
                  (static_cast<uint32_t>(__half_as_ushort(__float2half_rn(ey * k1))) << 16);
        R16.w23 = static_cast<uint32_t>(__half_as_ushort(__float2half_rn(-ey * k2))) |
                  (static_cast<uint32_t>(__half_as_ushort(__float2half_rn(ex * k2))) << 16);
        sxx = a;
        sxy = b;
        syy = c;
        det32 = dt;
      } else {
        // one float-pair reciprocal of the depth, then (x, y) / z side by side
        const f2 iz = f2_rcp(tz);
        const f2x2 uxy = f2x2_mul(f2x2_pack(tx, ty), f2x2_pack(iz, iz));
        const f2 ux = f2x2_first(uxy), uy = f2x2_second(uxy);
        const f2 fx = {vp.fx_hi, vp.fx_lo}, fy = {vp.fy_hi, vp.fy_lo};
        // the x and y halves of the pinhole map run side by side (f2x2)
        const f2x2 fxy = f2x2_pack(fx, fy);
        const f2x2 mxy = f2x2_add(f2x2_mul(fxy, f2x2_pack(ux, uy)),
                                  f2x2_pack(f2{vp.cx_hi, vp.cx_lo}, f2{vp.cy_hi, vp.cy_lo}));
        const f2 mx = f2x2_first(mxy), my = f2x2_second(mxy);
        depth = tz.hi;
        depth_l = tz.lo;
        R.misc.w = depth;
        const f2x2 J = f2x2_mul(fxy, f2x2_pack(iz, iz));  // (fx / z, fy / z)
        const f2 uxc = f2_clamp(ux, vp.limx_hi, vp.limx_lo);
        const f2 uyc = f2_clamp(uy, vp.limy_hi, vp.limy_lo);
        const f2x2 U = f2x2_pack(uxc, uyc);
        // rows of J W side by side: T[k] = (T0[k], T1[k]) with
        // T0 = fx/z (W0 - ux W2), T1 = fy/z (W1 - uy W2)
        f2x2 T[3];
  #pragma unroll
        for (int k = 0; k < 3; ++k) {
          const f2 w0 = {vp.R_hi[k], vp.R_lo[k]}, w1 = {vp.R_hi[3 + k], vp.R_lo[3 + k]};
          const f2 w2 = {vp.R_hi[6 + k], vp.R_lo[6 + k]};
          T[k] = f2x2_mul(J, f2x2_sub(f2x2_pack(w0, w1), f2x2_mul(U, f2x2_pack(w2, w2))));
        }
        // Sigma' = T Sigma3D T^T: M = (m0, m1) = rows of T Sigma3D, then
        // (a, c) += (m0 T0[j], m1 T1[j]) side by side and b += m0 T1[j]
        f2x2 ac = f2x2_pack(f2_from(0.f), f2_from(0.f));
        f2 a, b = f2_from(0.f), c;
  #pragma unroll
        for (int j = 0; j < 3; ++j) {
          f2x2 M = f2x2_mul(T[0], f2x2_pack(S[0][j], S[0][j]));
          M = f2x2_fma(T[1], f2x2_pack(S[1][j], S[1][j]), M);
          M = f2x2_fma(T[2], f2x2_pack(S[2][j], S[2][j]), M);
          ac = f2x2_fma(M, T[j], ac);
          b = f2_fma(f2x2_first(M), f2x2_second(T[j]), b);
        }
        a = f2x2_first(ac);
        c = f2x2_second(ac);
        a = f2_add(a, f2_from(kLowPass));
        c = f2_add(c, f2_from(kLowPass));
        const f2 det = f2_sub(f2_mul(a, c), f2_mul(b, b));
        const f2 h = f2_scale(f2_sub(a, c), 0.5f);
        const f2 rr = f2_sqrt(f2_add(f2_mul(h, h), f2_mul(b, b)));
        const f2 lam1 = f2_add(f2_scale(f2_add(a, c), 0.5f), rr);
        // unit eigenvector of lambda1 from whichever form has no cancellation
        f2 ex, ey;
        if (h.hi >= 0.f) {
          ex = f2_add(h, rr);
          ey = b;
        } else {
          ex = b;
          ey = f2_sub(rr, h);
        }
        const f2 en2 = f2_add(f2_mul(ex, ex), f2_mul(ey, ey));
        f2 ien = f2_from(1.f);
        if (en2.hi > kRootMin) {
          ien = f2_rsqrt(en2);
        } else {
          ex = f2_from(1.f);
          ey = f2_from(0.f);
        }
        // axis scales sqrt(0.5 log2 e / lambda) as float pairs too: the FP64
        // near-tie re-check evaluates alpha from this record.  With lambda2 =
        // det / lambda1 they are c / sqrt(lambda1) and c sqrt(lambda1) /
        // sqrt(det), c = sqrt(0.5 log2 e); the eigenvector's norm goes in too.
        const f2 root_hl = {static_cast<float>(kRootHalfLog2e),
                            static_cast<float>(kRootHalfLog2e -
                                               static_cast<double>(static_cast<float>(kRootHalfLog2e)))};
        const f2 r1 = f2_rsqrt(lam1);
        const f2 rd = det.hi > 0.f ? f2_rsqrt(det) : f2_from(0.f);
        const f2 is = f2_mul(ien, root_hl);
        const f2x2 sc = f2x2_mul(f2x2_pack(r1, f2_mul(f2_mul(lam1, r1), rd)), f2x2_pack(is, is));
        const f2 s1 = f2x2_first(sc), s2 = f2x2_second(sc);
        const f2x2 W0 = f2x2_mul(f2x2_pack(ex, ey), f2x2_pack(s1, s1));
        const f2x2 W1 = f2x2_mul(f2x2_pack(f2_neg(ey), ex), f2x2_pack(s2, s2));
        const f2 W00 = f2x2_first(W0), W01 = f2x2_second(W0);
        const f2 W10 = f2x2_first(W1), W11 = f2x2_second(W1);
        R.w_hi = make_float4(W00.hi, W01.hi, W10.hi, W11.hi);
        R.w_lo = make_float4(W00.lo, W01.lo, W10.lo, W11.lo);
        R.m = make_float4(mx.hi, my.hi, mx.lo, my.lo);
        sxx = a.hi;
        sxy = b.hi;
        syy = c.hi;
        det32 = det.hi;
        mx32 = mx.hi;
        my32 = my.hi;
      }
      // binning footprint (FP32 is plenty: the binning keeps a pixel of margin)
      const float r2b = binning_r2(r2);
      F.mx = mx32;
      F.my = my32;
      F.syr = syy * r2b;
      F.hy = sqrt_approx(F.syr);
      F.dys = sxy * sqrt_approx(r2b * rcp_approx(sxx));
      const float isyy = rcp_approx(syy);
      F.a = sxy * isyy;
      F.b2 = det32 * isyy * isyy;
      const float hy = F.hy;
      const float py0 = ceilf(__fsub_rn(__fsub_rn(F.my, hy), 1.5f));
      const float py1 = floorf(__fadd_rn(__fadd_rn(F.my, hy), 0.5f));
      // visible when the widened bounding box meets the image; the exact
      // per-row tile spans are counted later, per depth chunk
      const float hx = sqrt_approx(sxx * r2b);
      const float px0 = ceilf(__fsub_rn(__fsub_rn(F.mx, hx), 1.5f));
      const float px1 = floorf(__fadd_rn(__fadd_rn(F.mx, hx), 0.5f));
      if (!(py1 >= 0.f && py0 <= vp.height - 1 && px1 >= 0.f && px0 <= vp.width - 1)) {
        visible = false;
      } else {
        int ty0 = static_cast<int>(fmaxf(py0, 0.f)) / kTile;
        int ty1 = static_cast<int>(fminf(py1, (float)(vp.height - 1))) / kTile;
        if (vp.cols) {
          // 3-sigma coverage: the tiles that the square of half side
          // r = ceil(3 sqrt(lambda_max)) around the mean overlaps, decided in
          // FP32 with every step rounded to nearest (no contraction)
          const float mid = __fmul_rn(0.5f, __fadd_rn(sxx, syy));
          const float hd = __fmul_rn(0.5f, __fsub_rn(sxx, syy));
          const float lmax =
              __fadd_rn(mid, __fsqrt_rn(__fadd_rn(__fmul_rn(hd, hd), __fmul_rn(sxy, sxy))));
          const float r = ceilf(__fmul_rn(3.f, __fsqrt_rn(lmax)));
          const float inv = 1.f / kTile;  // a power of two: the scaling is exact
          const float cx0 = fmaxf(floorf(__fmul_rn(__fsub_rn(F.mx, r), inv)), 0.f);
          const float cx1 = fminf(__fsub_rn(ceilf(__fmul_rn(__fadd_rn(F.mx, r), inv)), 1.f),
                                  static_cast<float>(vp.tiles_x - 1));
          const float cy0 = fmaxf(floorf(__fmul_rn(__fsub_rn(F.my, r), inv)), 0.f);
          const float cy1 = fminf(__fsub_rn(ceilf(__fmul_rn(__fadd_rn(F.my, r), inv)), 1.f),
                                  static_cast<float>(vp.tiles_y - 1));
          if (cx0 <= cx1 && cy0 <= cy1) {
            ty0 = max(ty0, static_cast<int>(cy0));
            ty1 = min(ty1, static_cast<int>(cy1));
            col_clip = static_cast<uint32_t>(cx0) | (static_cast<uint32_t>(cx1) << 16);
          } else {
            ty1 = ty0 - 1;
          }
        }
        if (ty0 <= ty1) {
          F.rows = static_cast<uint32_t>(ty0) | (static_cast<uint32_t>(ty1) << 16);
          // the spans of the rows stay within +-hx of the mean; one more pixel
          // on each side, and a little of hx, cover their rounding
          const float bxw = 1.00001f * hx;
          int c0 = static_cast<int>(fmaxf(ceilf(F.mx - bxw - 2.5f), 0.f)) / kTile;
          int c1 = static_cast<int>(fminf(floorf(F.mx + bxw + 1.5f),
                                          static_cast<float>(vp.width - 1))) / kTile;
          if (vp.cols) {
            c0 = max(c0, static_cast<int>(col_clip & 0xFFFFu));
            c1 = min(c1, static_cast<int>(col_clip >> 16));
          }
          if (c0 <= c1)
            bx = make_uint2(static_cast<uint32_t>(c0) | (static_cast<uint32_t>(c1) << 16), F.rows);
        } else {
          visible = false;
        }
      }
    }
    if (vp.cols) vp.cols[slot] = col_clip;
    if (visible) {  // records are read only through tile lists, which hold visible slots
      if constexpr (kFast)
        rec16[slot] = R16;
      else
        rec[slot] = R;
    }
    foot[slot] = F;
    box[slot] = bx;
    const uint32_t k = visible ? depth_key(depth) : 0xFFFFFFFFu;
    if (visible) {
      kmin = min(kmin, k);
      kmax = max(kmax, k);
      ++n_vis;
    }
    key[slot] = k;
    depth_lo[slot] = float_order_key(depth_l);
  }
  }
  if (key_range) {
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    n_vis = __reduce_add_sync(0xffffffffu, n_vis);
    if ((threadIdx.x & 31) == 0 && kmin <= kmax) {
      atomicMin(&key_range[0], kmin);
      atomicMax(&key_range[1], kmax);
      atomicAdd(&key_range[2], n_vis);
    }
  }
}

// The radix sort orders by the float depth key hi, stably by slot, so equal
// keys already come in (view, index) order.  Only elements of one view that
// share a key need another order: by the low word of the float-pair depth,
// then by slot -- the order of the full-precision depth with ties by index
// that the compositing of Eq. 1 walks.  A thread acts only where such a
// same-view run starts; the runs are short and sorted by insertion.
__device__ __forceinline__ void fix_tie_run(int64_t k, int64_t n_total, const SlotView& view_of,
                                            uint32_t kk, const uint32_t* __restrict__ key,
                                            uint32_t* __restrict__ val,
                                            const uint32_t* __restrict__ depth_lo) {
  const uint32_t view = view_of(val[k]);
  int64_t e = k + 2;
  while (e < n_total && key[e] == kk && view_of(val[e]) == view) ++e;
  for (int64_t a = k + 1; a < e; ++a) {
    const uint32_t va = val[a];
    const uint64_t ka = (static_cast<uint64_t>(depth_lo[va]) << 32) | va;
    int64_t b = a - 1;
    while (b >= k) {
      const uint32_t vb = val[b];
      const uint64_t kb = (static_cast<uint64_t>(depth_lo[vb]) << 32) | vb;
      if (kb <= ka) break;
      val[b + 1] = vb;
      --b;
    }
    val[b + 1] = va;
  }
}

// Each thread takes four consecutive positions, k0 .. k0 + 3.  Equal keys of
// different views are common (a batch holds many views of the same depths), so
// it compares keys and views of its positions' neighbours, k0 - 1 .. k0 + 5,
// from one 16-byte load each (when both arrays are 16-byte aligned) and the
// words around them.  Nearly every same-view run is a pair: the pairs' low
// words are gathered together, where walking each run as it is met costs a
// chain of gathers per run.  Longer runs are walked.  Bound by the latency of
// its loads and gathers: every sixth slot of a 10^6-Gaussian view shares its
// key.  4.8 10^7 slots of 48 views: 375 us with every run walked, 329 us with
// the pairs gathered, 313 us with the slots loaded beside the keys instead of
// after them, 249 us with blocks of 128, twelve to an SM (42 registers; 256
// threads, six: 268; 128, fourteen or sixteen: 281).
constexpr int kTieThreads = 128;
__global__ void __launch_bounds__(kTieThreads, 12) depth_tie_fix_kernel(
    int64_t n_total, int64_t n, const uint32_t* __restrict__ key, uint32_t* __restrict__ val,
    const uint32_t* __restrict__ depth_lo, const unsigned long long* __restrict__ counters) {
  const int64_t k0 = 4 * (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x);
  if (k0 + 1 >= n_total) return;
  // t[1 + i], w[1 + i]: key and slot of position k0 + i (key 0xFFFFFFFF where
  // there is none: never a run)
  uint32_t t[7], w[7];
  const bool full = k0 + 4 <= n_total &&
                    ((reinterpret_cast<uintptr_t>(key) | reinterpret_cast<uintptr_t>(val)) & 15u) == 0;
  auto load = [&](const uint32_t* src, uint32_t none, uint32_t* dst) {
    if (full) {
      const uint4 q = *reinterpret_cast<const uint4*>(src + k0);
      dst[1] = q.x;
      dst[2] = q.y;
      dst[3] = q.z;
      dst[4] = q.w;
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) dst[1 + i] = k0 + i < n_total ? src[k0 + i] : none;
    }
    dst[0] = k0 > 0 ? src[k0 - 1] : none;
    dst[5] = k0 + 4 < n_total ? src[k0 + 4] : none;
    dst[6] = k0 + 5 < n_total ? src[k0 + 5] : none;
  };
  load(key, 0xFFFFFFFFu, t);
  load(val, 0u, w);
  if (gave_up(counters)) return;
  bool any = false;  // an equal neighbour somewhere among the four
#pragma unroll
  for (int i = 1; i <= 4; ++i) any = any || (t[i] != 0xFFFFFFFFu && t[i + 1] == t[i]);
  if (!any) return;
  const SlotView view_of(n);
  bool tie[6];  // positions k0 + i - 1 and k0 + i: equal keys, one view
#pragma unroll
  for (int i = 0; i < 6; ++i)
    tie[i] = t[i] != 0xFFFFFFFFu && t[i + 1] == t[i] && view_of(w[i]) == view_of(w[i + 1]);
  uint32_t lo[4][2];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (tie[1 + i] && !tie[i] && !tie[2 + i]) {
      lo[i][0] = depth_lo[w[1 + i]];
      lo[i][1] = depth_lo[w[2 + i]];
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (!tie[1 + i] || tie[i]) continue;  // no run starts here
    if (!tie[2 + i]) {
      // slots of a pair ascend already: equal low words stay
      if (lo[i][0] > lo[i][1]) {
        val[k0 + i] = w[2 + i];
        val[k0 + i + 1] = w[1 + i];
      }
    } else {
      fix_tie_run(k0 + i, n_total, view_of, t[1 + i], key, val, depth_lo);
    }
  }
}

// ---------------------------------------------------------------------------
// Per depth chunk: count and emit the (tile, Gaussian) entries of sorted
// positions [p0, p0 + n_pos) on tiles not yet saturated.
// ---------------------------------------------------------------------------

// What the binning reads of a view, kept in shared memory: consecutive sorted
// positions belong to any of the batch's views, and 32 different views'
// parameters read through L1 take a line each.
struct BinView {
  int tile_base, tiles_x, width, cell;  // cell: the view's first prefix-table entry
};

struct RowJob {
  int row;         // tile row
  int owner;       // lane that holds the owning Gaussian
  bool ok;         // r < R
};

// Row r of the warp's 32 Gaussians' tile rows, in order: the owner is found by
// a binary search over the lanes' inclusive row counts.  Every lane of the
// warp must call this (it shuffles).
__device__ __forceinline__ RowJob row_job(int r, int R, uint32_t incl_rows, int ty0_lane) {
  // owner = number of lanes whose inclusive row count is <= r
  int lo = 0;
#pragma unroll
  for (int s = 16; s >= 1; s >>= 1) {
    const uint32_t v = __shfl_sync(0xffffffffu, incl_rows, lo + s - 1);
    if (v <= static_cast<uint32_t>(r)) lo += s;
  }
  const int owner = min(lo, 31);
  const uint32_t pi = __shfl_sync(0xffffffffu, incl_rows, max(owner - 1, 0));
  const int ty0 = __shfl_sync(0xffffffffu, ty0_lane, owner);
  RowJob j;
  j.ok = r < R;
  j.owner = owner;
  j.row = ty0 + (r - static_cast<int>(owner > 0 ? pi : 0u));
  return j;
}

// Number of tile rows of a slot's footprint (first row *ty0) -- none when every
// tile of the footprint's bounding box is already saturated, as is the case
// for most slots of later depth chunks.  Over the footprint x(dy) - mx stays
// within +-hx, hx^2 = syr (a^2 + b2); the box takes one more pixel on each
// side than the rows' spans, so it holds every span whatever their rounding.
__device__ __forceinline__ uint32_t live_rows(const Footprint& f, uint32_t slot, const BinView& vp,
                                              const uint32_t* __restrict__ cols,
                                              const uint32_t* __restrict__ free_tab,
                                              const uint64_t* __restrict__ sat, int* ty0) {
  int t0, t1;
  footprint_rows(f, &t0, &t1);
  *ty0 = t0;
  if (t1 < t0) return 0u;
  const float hx = sqrtf(f.syr * fmaf(f.a, f.a, f.b2));
  const float x0 = fmaxf(ceilf(f.mx - hx - 2.5f), 0.f);
  const float x1 = fminf(floorf(f.mx + hx + 1.5f), static_cast<float>(vp.width - 1));
  if (!(x0 <= x1)) return 0u;
  int c0 = static_cast<int>(x0) / kTile, c1 = static_cast<int>(x1) / kTile;
  if (cols) {  // 3-sigma coverage
    const uint32_t c = cols[slot];
    c0 = max(c0, static_cast<int>(c & 0xFFFFu));
    c1 = min(c1, static_cast<int>(c >> 16));
    if (c0 > c1) return 0u;
  }
  const uint32_t rows = static_cast<uint32_t>(t1 - t0 + 1);
  if (free_tab) return free_in_box(free_tab + vp.cell, vp.tiles_x, t0, t1, c0, c1) ? rows : 0u;
  for (int ty = t0; ty <= t1; ++ty) {
    const int base = vp.tile_base + ty * vp.tiles_x;
    if (any_free(sat, base + c0, base + c1)) return rows;
  }
  return 0u;
}

// Unsaturated tiles of one tile row of a footprint: [*a, *b] (global ids) and
// their number.
__device__ __forceinline__ uint32_t row_free(const Footprint& f, uint32_t slot, int row,
                                             const BinView& vp, const uint32_t* __restrict__ cols,
                                             const uint64_t* __restrict__ sat, int* a, int* b) {
  int tx0, tx1;
  if (!row_span(f, row, vp.width, &tx0, &tx1)) return 0;
  if (!clip_cols(cols, slot, &tx0, &tx1)) return 0;
  const int base = vp.tile_base + row * vp.tiles_x;
  *a = base + tx0;
  *b = base + tx1;
  return count_free(sat, *a, *b);
}

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t x, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// The k-th (from 0) unsaturated tile id from `a` on; there must be one.
__device__ __forceinline__ uint32_t nth_free(const uint64_t* __restrict__ sat, int a, int k) {
  int w = a >> 6;
  uint64_t bits = ~sat[w] & (~0ull << (a & 63));
  for (int c = __popcll(bits); k >= c; c = __popcll(bits)) {
    k -= c;
    bits = ~sat[++w];
  }
  for (; k > 0; --k) bits &= bits - 1;
  return static_cast<uint32_t>(w * 64 + __ffsll(static_cast<long long>(bits)) - 1);
}

// Count, offset and emit in one pass.  Blocks take virtual ids in launch
// order (a ticket), so every block's predecessors are running or done.  A
// block (4 warps: a short wait at its barriers) counts its 128 positions'
// entries, publishes the count, then adds up its predecessors' published words
// (decoupled look-back: a word is either a block's own count or the inclusive
// prefix up to it; the walk stops at the first prefix), publishes its own
// prefix and emits from its offset.  No block waits on a later one.  Entries
// at or past `capacity` are not written; *total receives the entry count
// either way, so the caller can grow the buffer and run the chunk again.  A
// look-back that polls a predecessor's word more than spin_limit times gives
// up, counts a time-out (kLookbackTimeout) and uses 0.
//
// With the positions' number read on the device (kDeviceRange) the blocks past
// it leave at once.  (One set of resident blocks that loops over the tickets
// measured slower, 7.06 ms against 5.25 for the 100-view, 10^6-Gaussian
// workload: its blocks advance in step and look back over each other.)  A warp
// spreads its 32 positions' tile rows over its lanes, one (slot, row)
// job per lane per round, so large footprints do not hold up small ones; the
// entries of a round are then spread over the lanes again, so that 32
// consecutive list places are written at a time.
constexpr int kBinThreads = 128, kBinWarps = kBinThreads / 32;

template <bool kDeviceRange>
__global__ void __launch_bounds__(kBinThreads, 12) bin_fused_kernel(
    int64_t p0, int64_t n_pos, SlotView sv, const ViewParams* __restrict__ views, int n_views,
    const uint32_t* __restrict__ sorted_val,
    const Footprint* __restrict__ foot, const uint64_t* __restrict__ sat,
    uint32_t* __restrict__ out_key, uint32_t* __restrict__ out_val, uint32_t capacity,
    unsigned long long* __restrict__ status, uint32_t* __restrict__ ticket,
    uint32_t* __restrict__ total, unsigned long long* __restrict__ counters, int spin_limit,
    const int64_t* __restrict__ range_dev) {
  __shared__ uint32_t s_vb, s_boff, s_wtot[kBinWarps];
  __shared__ BinView s_view[kMaxViewsPerBatch];
  if constexpr (kDeviceRange) {  // the chunk's positions [range_dev[0], range_dev[1])
    p0 = range_dev[0];
    n_pos = min(n_pos, range_dev[1] - range_dev[0]);  // the launch's scratch is sized for n_pos
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    const uint32_t t = atomicAdd(ticket, 1u);
    const bool off = gave_up(counters);  // the sorted slots may be incomplete
    s_vb = off ? kGaveUpTotal : t;
    if (off) *total = kGaveUpTotal;
  }
  const uint32_t* const cols = views[0].cols;
  const uint32_t* const free_tab = views[0].free_tab;
  for (int v = threadIdx.x; v < n_views; v += kBinThreads) {
    const ViewParams& vp = views[v];
    s_view[v] = {vp.tile_base, vp.tiles_x, vp.width,
                 free_tab ? static_cast<int>(vp.free_tab - free_tab) : 0};
  }
  __syncthreads();
  const uint32_t vb = s_vb;
  if (vb == kGaveUpTotal) return;
  const int64_t j = static_cast<int64_t>(vb) * kBinThreads + threadIdx.x;
  if (j - threadIdx.x >= n_pos) return;  // whole block: the grid was sized for more
  uint32_t g = 0u, nrows = 0u;
  int ty0 = 0;
  if (j < n_pos) {
    g = sorted_val[p0 + j];
    nrows = live_rows(foot[g], g, s_view[sv(g)], cols, free_tab, sat, &ty0);
  }
  const uint32_t incl = warp_incl_scan(nrows, lane);
  const int R = static_cast<int>(__shfl_sync(0xffffffffu, incl, 31));  // same for the whole warp
  // one round's job: the lane's tile range and its free tiles
  auto job = [&](int r, int* a, int* b, uint32_t* slot) -> uint32_t {
    const RowJob jb = row_job(r, R, incl, ty0);
    *slot = __shfl_sync(0xffffffffu, g, jb.owner);
    *a = 0;
    *b = -1;
    if (!jb.ok) return 0u;
    return row_free(foot[*slot], *slot, jb.row, s_view[sv(*slot)], cols, sat, a, b);
  };
  // count; the first kStash rounds' jobs are kept in registers for the emission
  constexpr int kStash = 3;
  int st_a[kStash], st_b[kStash];
  uint32_t st_fr[kStash], st_g[kStash];
  uint32_t wtot = 0;
#pragma unroll
  for (int k = 0; k < kStash; ++k) {
    st_a[k] = 0;
    st_b[k] = -1;
    st_fr[k] = 0;
    st_g[k] = 0;
    if (32 * k < R) {
      st_fr[k] = job(32 * k + lane, &st_a[k], &st_b[k], &st_g[k]);
      wtot += __reduce_add_sync(0xffffffffu, st_fr[k]);
    }
  }
  for (int r0 = 32 * kStash; r0 < R; r0 += 32) {
    int a, b;
    uint32_t slot;
    wtot += __reduce_add_sync(0xffffffffu, job(r0 + lane, &a, &b, &slot));
  }
  if (lane == 0) s_wtot[warp] = wtot;
  __syncthreads();
  // offset of the block
  if (warp == 0) {
    uint32_t btot = 0;
    for (int w = 0; w < kBinWarps; ++w) btot += s_wtot[w];
    if (lane == 0) atomicExch(&status[vb], (vb == 0 ? kLbPrefix : kLbCount) | btot);
    const uint32_t excl = look_back(status, vb, counters, spin_limit, lane);
    if (lane == 0) {
      if (vb > 0) atomicExch(&status[vb], kLbPrefix | add_sat(excl, btot));
      s_boff = excl;
      if (static_cast<int64_t>(vb + 1) * kBinThreads >= n_pos) *total = add_sat(excl, btot);
    }
  }
  __syncthreads();
  uint32_t o0 = s_boff;
  for (int w = 0; w < warp; ++w) o0 += s_wtot[w];
  const uint32_t wend = o0 + wtot;
  // one round's entries, from list place o0 on
  auto emit = [&](uint32_t fr, int a, int b, uint32_t slot) {
    const uint32_t sc = warp_incl_scan(fr, lane);
    const uint32_t T = __shfl_sync(0xffffffffu, sc, 31);
    const int n_tiles = b - a + 1;
    for (uint32_t e0 = 0; e0 < T; e0 += 32) {
      const uint32_t e = min(e0 + lane, T - 1);
      // owner of entry e: the number of lanes whose inclusive count is <= e
      int lo = 0;
#pragma unroll
      for (int s = 16; s >= 1; s >>= 1) {
        const uint32_t v = __shfl_sync(0xffffffffu, sc, lo + s - 1);
        if (v <= e) lo += s;
      }
      const int ow = min(lo, 31);
      const uint32_t fr_o = __shfl_sync(0xffffffffu, fr, ow);
      const uint32_t k = e - (__shfl_sync(0xffffffffu, sc, ow) - fr_o);
      const int a_o = __shfl_sync(0xffffffffu, a, ow), n_o = __shfl_sync(0xffffffffu, n_tiles, ow);
      const uint32_t slot_o = __shfl_sync(0xffffffffu, slot, ow);
      if (e0 + lane < T && o0 + e < capacity) {
        out_key[o0 + e] = fr_o == static_cast<uint32_t>(n_o)
                              ? static_cast<uint32_t>(a_o) + k  // no saturated tile among them
                              : nth_free(sat, a_o, static_cast<int>(k));
        out_val[o0 + e] = slot_o;
      }
    }
    o0 += T;
  };
  // emit, in the same (slot, row) order as the count
#pragma unroll
  for (int k = 0; k < kStash; ++k)
    if (32 * k < R) emit(st_fr[k], st_a[k], st_b[k], st_g[k]);
  for (int r0 = 32 * kStash; r0 < R; r0 += 32) {
    int a, b;
    uint32_t slot;
    const uint32_t fr = job(r0 + lane, &a, &b, &slot);
    emit(fr, a, b, slot);
  }
  if (lane == 0 && o0 != wend) atomicAdd(&counters[kBinningMismatch], 1ull);
}

// Bit i % 32 of word view * words_per_view + i / 32: an unsaturated tile lies
// in the tile box of Gaussian i in that view.  A block takes kLiveSlots
// consecutive slots of one view, whose prefix table it reads from shared
// memory (views of up to kTableCells cells): in depth order a slot's four
// table reads each fetch a sector of some other view's table.  Bound by the
// shared-memory gathers: with rows of an even number of words the slots'
// columns, crowded around the scene's middle, alone choose the banks, so rows
// are an odd number of words apart (4.8 10^7 slots of 1008x756 views: 182 us
// with rows of 64 entries, 154 us so).
constexpr int kTableCells = 10240;
constexpr int kLiveSlots = 16384;
__global__ void __launch_bounds__(256) slot_live_kernel(
    int64_t n, const ViewParams* __restrict__ views, const TileBox* __restrict__ box,
    int64_t words_per_view, uint32_t* __restrict__ live) {
  __shared__ uint16_t s_tab[kTableCells];
  const ViewParams& vp = views[blockIdx.y];
  const int w1 = vp.tiles_x + 1, w2 = 2 * (((w1 + 1) / 2) | 1);
  const uint32_t* __restrict__ tab = vp.free_tab;
  const bool shared = static_cast<int64_t>(w2) * (vp.tiles_y + 1) <= kTableCells;
  const int stride = shared ? w2 : w1;
  if (shared)
    for (int r = threadIdx.x >> 5; r <= vp.tiles_y; r += 8)
      for (int c = threadIdx.x & 31; c < w1; c += 32)
        s_tab[r * w2 + c] = static_cast<uint16_t>(tab[r * w1 + c]);
  __syncthreads();
  const int64_t i0 = static_cast<int64_t>(blockIdx.x) * kLiveSlots + threadIdx.x;
  const TileBox* __restrict__ vbox = box + static_cast<int64_t>(blockIdx.y) * n;
  uint32_t* const out = live + static_cast<int64_t>(blockIdx.y) * words_per_view;
#pragma unroll 4
  for (int k = 0; k < kLiveSlots / 256; ++k) {
    const int64_t i = i0 + 256 * k;
    bool any = false;
    if (i < n) {
      const TileBox b = vbox[i];
      if (box_visible(b)) {
        const int c0 = b.x & 0xFFFFu, c1 = (b.x >> 16) + 1;
        const int r0 = static_cast<int>(b.y & 0xFFFFu) * stride;
        const int r1 = static_cast<int>((b.y >> 16) + 1) * stride;
        any = shared ? s_tab[r1 + c1] + s_tab[r0 + c0] != s_tab[r0 + c1] + s_tab[r1 + c0]
                     : tab[r1 + c1] + tab[r0 + c0] != tab[r0 + c1] + tab[r1 + c0];
      }
    }
    const uint32_t bits = __ballot_sync(0xffffffffu, any);
    if ((threadIdx.x & 31) == 0 && i < n) out[i >> 5] = bits;
  }
}

// Per view of the batch (one block each), the 2-D prefix sums of its
// unsaturated tiles: free_tab[r * (tiles_x + 1) + c] = unsaturated tiles in
// rows < r and columns < c (row 0 and column 0 are zero).  A warp runs along a
// row 32 tiles at a time, a thread then down a column.  Views of up to
// kTableCells cells keep the table in shared memory until it is whole (a
// 1008x756 view: 17 us through global memory, 8 us so).
__global__ void __launch_bounds__(256) free_table_kernel(const ViewParams* __restrict__ views,
                                                         const uint64_t* __restrict__ sat) {
  __shared__ uint32_t s_tab[kTableCells];
  const ViewParams& vp = views[blockIdx.x];
  uint32_t* const out = vp.free_tab;
  if (!out) return;
  const int tx = vp.tiles_x, ty = vp.tiles_y, w1 = tx + 1, base = vp.tile_base;
  const int64_t cells = static_cast<int64_t>(w1) * (ty + 1);
  const bool shared = cells <= kTableCells;
  uint32_t* const tab = shared ? s_tab : out;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int c = threadIdx.x; c < w1; c += blockDim.x) tab[c] = 0u;
  for (int r = warp; r < ty; r += 8) {
    uint32_t* row = tab + static_cast<int64_t>(r + 1) * w1;
    if (lane == 0) row[0] = 0u;
    uint32_t run = 0;
    for (int c0 = 0; c0 < tx; c0 += 32) {
      const int g = base + r * tx + c0 + lane;
      const bool free = c0 + lane < tx && ((sat[g >> 6] >> (g & 63)) & 1ull) == 0ull;
      const uint32_t bits = __ballot_sync(0xffffffffu, free);
      if (c0 + lane < tx) row[c0 + lane + 1] = run + __popc(bits & (0xffffffffu >> (31 - lane)));
      run += __popc(bits);
    }
  }
  __syncthreads();
  for (int c = threadIdx.x + 1; c < w1; c += blockDim.x) {
    uint32_t acc = 0;
    for (int r = 1; r <= ty; ++r) {
      uint32_t* e = tab + static_cast<int64_t>(r) * w1 + c;
      acc += *e;
      *e = acc;
    }
  }
  if (!shared) return;
  __syncthreads();
  for (int k = threadIdx.x; k < static_cast<int>(cells); k += blockDim.x) out[k] = s_tab[k];
}

// [start, end) of every tile's run in the tile-sorted list.  Each thread
// takes four consecutive entries (one 16-byte load when the list is 16-byte
// aligned, as the library's buffers are) and the entries on either side.
__global__ void ranges_kernel(int64_t n_entries, const uint32_t* __restrict__ key,
                              uint2* __restrict__ ranges,
                              const unsigned long long* __restrict__ counters,
                              const uint32_t* __restrict__ n_dev) {
  if (n_dev) n_entries = min(n_entries, static_cast<int64_t>(*n_dev));
  const int64_t k0 = 4 * (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x);
  if (k0 >= n_entries) return;
  uint32_t t[6];  // entries k0 - 1 .. k0 + 4 (0xFFFFFFFF outside the list)
  t[0] = k0 > 0 ? key[k0 - 1] : 0xFFFFFFFFu;
  if (k0 + 4 <= n_entries && (reinterpret_cast<uintptr_t>(key) & 15u) == 0) {
    const uint4 q = *reinterpret_cast<const uint4*>(key + k0);
    t[1] = q.x;
    t[2] = q.y;
    t[3] = q.z;
    t[4] = q.w;
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) t[1 + i] = k0 + i < n_entries ? key[k0 + i] : 0xFFFFFFFFu;
  }
  t[5] = k0 + 4 < n_entries ? key[k0 + 4] : 0xFFFFFFFFu;
  if (gave_up(counters)) return;  // keys of the list may be missing
#pragma unroll
  for (int i = 1; i <= 4; ++i) {
    const int64_t k = k0 + i - 1;
    if (k >= n_entries) break;
    if (t[i - 1] != t[i]) ranges[t[i]].x = static_cast<uint32_t>(k);
    if (t[i + 1] != t[i]) ranges[t[i]].y = static_cast<uint32_t>(k + 1);
  }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------

cudaError_t launch_scene_prep(int64_t n, const float* mean, const void* quat, int quat_dtype,
                              const void* scale, int scale_dtype, const void* opacity,
                              int opacity_dtype, float4* pos_op, float4* cov, unsigned int* err,
                              cudaStream_t stream) {
  if (n == 0) return cudaSuccess;
  const int threads = 256;
  const int64_t blocks = (n + threads - 1) / threads;
  scene_prep_kernel<<<static_cast<unsigned>(blocks), threads, 0, stream>>>(
      n, mean, quat, quat_dtype, scale, scale_dtype, opacity, opacity_dtype, pos_op, cov, err);
  return cudaGetLastError();
}

cudaError_t launch_project(int64_t n, int n_views, const ViewParams* views, const float4* pos_op,
                           const float4* cov, ProjRecord* rec, CompactRecord* rec16,
                           Footprint* foot, TileBox* box, uint32_t* key, uint32_t* depth_lo,
                           uint32_t* key_range, cudaStream_t stream) {
  if (n == 0 || n_views == 0) return cudaSuccess;
  const int threads = 256;
  const int64_t blocks = (n + threads - 1) / threads;
  // two sets of resident blocks (three per SM of 152), if there are the views
  const int64_t share = std::max<int64_t>(1, std::min<int64_t>(n_views, 2 * 3 * 152 / blocks));
  const dim3 grid(static_cast<unsigned>(blocks), static_cast<unsigned>(share));
  // the reduced-precision form takes the FP32 projection
  if (rec16)
    project_kernel<true><<<grid, threads, 0, stream>>>(n, n_views, views, pos_op, cov, rec, rec16,
                                                       foot, box, key, depth_lo, key_range);
  else
    project_kernel<false><<<grid, threads, 0, stream>>>(n, n_views, views, pos_op, cov, rec, rec16,
                                                        foot, box, key, depth_lo, key_range);
  return cudaGetLastError();
}

cudaError_t launch_depth_tie_fix(int64_t n_total, int64_t n, const uint32_t* key, uint32_t* val,
                                 const uint32_t* depth_lo, const unsigned long long* counters,
                                 cudaStream_t stream) {
  if (n_total < 2) return cudaSuccess;
  const int64_t blocks = ((n_total + 3) / 4 + kTieThreads - 1) / kTieThreads;
  depth_tie_fix_kernel<<<static_cast<unsigned>(blocks), kTieThreads, 0, stream>>>(
      n_total, n, key, val, depth_lo, counters);
  return cudaGetLastError();
}

cudaError_t launch_bin_fused(int64_t p0, int64_t n_pos, int64_t n, const ViewParams* views,
                             int n_views, const uint32_t* sorted_val,
                             const Footprint* foot, const uint64_t* sat, uint32_t* out_key,
                             uint32_t* out_val, uint32_t capacity, void* lookback,
                             uint32_t* total, unsigned long long* counters, cudaStream_t stream,
                             const int64_t* range_dev) {
  if (n_pos <= 0) return cudaMemsetAsync(total, 0, sizeof(uint32_t), stream);
  const int64_t blocks = (n_pos + kBinThreads - 1) / kBinThreads;
  uint32_t* ticket = static_cast<uint32_t*>(lookback);
  unsigned long long* status = reinterpret_cast<unsigned long long*>(
      static_cast<char*>(lookback) + 256);
  cudaError_t e = cudaMemsetAsync(lookback, 0, 256 + static_cast<size_t>(blocks) * 8, stream);
  if (e == cudaSuccess && range_dev)  // a chunk may turn out empty
    e = cudaMemsetAsync(total, 0, sizeof(uint32_t), stream);
  if (e != cudaSuccess) return e;
  auto launch = [&](auto kernel) {
    kernel<<<static_cast<unsigned>(blocks), kBinThreads, 0, stream>>>(
        p0, n_pos, SlotView(n > 0 ? n : 1), views, n_views, sorted_val, foot, sat, out_key,
        out_val, capacity, status, ticket, total, counters, kLookbackSpinLimit, range_dev);
    return cudaGetLastError();
  };
  return range_dev ? launch(bin_fused_kernel<true>) : launch(bin_fused_kernel<false>);
}

cudaError_t launch_lookback_probe(void* lookback, uint32_t* total, unsigned long long* counters,
                                  const ViewParams* views, const uint32_t* sorted_val,
                                  const Footprint* foot, const uint64_t* sat, uint32_t* out_key,
                                  uint32_t* out_val, int spin_limit, cudaStream_t stream) {
  // one block whose ticket comes out as 1: its predecessor (block 0) never
  // runs, so its status word stays empty and the look-back must give up
  uint32_t* ticket = static_cast<uint32_t*>(lookback);
  unsigned long long* status = reinterpret_cast<unsigned long long*>(
      static_cast<char*>(lookback) + 256);
  cudaError_t e = cudaMemsetAsync(lookback, 0, 256 + 16, stream);
  if (e != cudaSuccess) return e;
  const uint32_t one = 1u;
  e = cudaMemcpyAsync(ticket, &one, sizeof(one), cudaMemcpyHostToDevice, stream);
  if (e != cudaSuccess) return e;
  // position 128 is the ticket's first and only one, sorted_val[0]
  bin_fused_kernel<false><<<1, kBinThreads, 0, stream>>>(
      -kBinThreads, kBinThreads + 1, SlotView(1), views, 1, sorted_val, foot, sat, out_key,
      out_val, 0u, status, ticket, total, counters, spin_limit, nullptr);
  return cudaGetLastError();
}

size_t bin_fused_temp_bytes(int64_t n_pos) {
  return 256 + static_cast<size_t>((n_pos + kBinThreads - 1) / kBinThreads) * 8;
}

int64_t live_words(int64_t n) { return (n + 31) / 32; }

cudaError_t launch_slot_live(int64_t n, const ViewParams* views, int n_views, const TileBox* box,
                             uint32_t* live, cudaStream_t stream) {
  if (n <= 0 || n_views <= 0) return cudaSuccess;
  const dim3 grid(static_cast<unsigned>((n + kLiveSlots - 1) / kLiveSlots),
                  static_cast<unsigned>(n_views));
  slot_live_kernel<<<grid, 256, 0, stream>>>(n, views, box, live_words(n), live);
  return cudaGetLastError();
}

namespace {
struct LiveSlots {
  SlotView sv;
  const uint32_t* sorted_val;
  const uint32_t* live;
  int64_t words_per_view;
  __device__ __forceinline__ uint32_t value(int64_t p) const { return sorted_val[p]; }
  __device__ __forceinline__ bool keep(uint32_t g) const {
    const uint32_t v = sv(g), k = g - v * sv.n;
    return (live[v * words_per_view + (k >> 5)] >> (k & 31)) & 1u;
  }
};
}  // namespace

cudaError_t launch_compact_live(int64_t p0, int64_t n_pos, int64_t n, const uint32_t* sorted_val,
                                const uint32_t* live, uint32_t* out, int64_t* range_out,
                                void* lookback, unsigned long long* counters, cudaStream_t stream,
                                const int64_t* range_in) {
  return launch_compact(LiveSlots{SlotView(n > 0 ? n : 1), sorted_val, live, live_words(n)}, p0,
                        n_pos, out, range_out, lookback, counters, stream, range_in);
}

cudaError_t launch_free_tables(const ViewParams* views, int n_views, const uint64_t* sat,
                               cudaStream_t stream) {
  if (n_views <= 0) return cudaSuccess;
  free_table_kernel<<<static_cast<unsigned>(n_views), 256, 0, stream>>>(views, sat);
  return cudaGetLastError();
}

cudaError_t launch_ranges(int64_t n_entries, const uint32_t* key, uint2* ranges,
                          const unsigned long long* counters, cudaStream_t stream,
                          const uint32_t* n_dev) {
  if (n_entries == 0) return cudaSuccess;
  const int threads = 256;
  const int64_t blocks = ((n_entries + 3) / 4 + threads - 1) / threads;
  ranges_kernel<<<static_cast<unsigned>(blocks), threads, 0, stream>>>(n_entries, key, ranges,
                                                                       counters, n_dev);
  return cudaGetLastError();
}

}  // namespace fs
