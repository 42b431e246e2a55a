// Double-float arithmetic: an unevaluated sum hi + lo of two floats per real
// (Dekker 1971; about 2^-46 relative), float4 {re_hi, re_lo, im_hi, im_lo} per
// complex number.  Products take the exact rounding error of hi * hi from an
// FMA (TwoProduct) plus the hi * lo cross terms; sums carry their exact
// rounding error by Knuth's TwoSum into the lo part (the accumulation of Ogita,
// Rump and Oishi's Dot2).  A float64 complex multiply-add (4 FMAs at GB300's
// 1/64 float64 rate) becomes 4 x 12 float32 operations.
#pragma once
#include "common.cuh"

namespace nne {

__device__ __forceinline__ float4 df_from_cd(cx<double> a) {
  const float rh = (float)a.re, ih = (float)a.im;
  return make_float4(rh, (float)(a.re - (double)rh), ih, (float)(a.im - (double)ih));
}
__device__ __forceinline__ double df_to_d(float hi, float lo) { return (double)hi + (double)lo; }
// (hi, lo) += x * y, x = xh + xl, y = yh + yl
__device__ __forceinline__ void df_mac(float& hi, float& lo, float xh, float xl, float yh, float yl) {
  const float ph = __fmul_rn(xh, yh);
  const float pe = fmaf(xh, yl, fmaf(xl, yh, fmaf(xh, yh, -ph)));
  const float s = __fadd_rn(hi, ph);
  const float bb = __fsub_rn(s, hi);
  const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(ph, bb));
  hi = s;
  lo = __fadd_rn(lo, __fadd_rn(e, pe));
}
// (hi, lo) += (bh, bl)
__device__ __forceinline__ void df_add(float& hi, float& lo, float bh, float bl) {
  const float s = __fadd_rn(hi, bh);
  const float bb = __fsub_rn(s, hi);
  const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(bh, bb));
  hi = s;
  lo = __fadd_rn(lo, __fadd_rn(e, bl));
}
// The same with the lo parts first: the bits do not depend on which addend is which (the
// rounding error of the hi parts is exact), so lanes that exchange partial sums agree.
__device__ __forceinline__ void df_add_sym(float& hi, float& lo, float bh, float bl) {
  const float s = __fadd_rn(hi, bh);
  const float bb = __fsub_rn(s, hi);
  const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(bh, bb));
  hi = s;
  lo = __fadd_rn(__fadd_rn(lo, bl), e);
}
__device__ __forceinline__ void df_norm(float& hi, float& lo) {
  const float s = __fadd_rn(hi, lo);
  lo = __fsub_rn(lo, __fsub_rn(s, hi));
  hi = s;
}
// acc (re, im) += a * v (conj_a: conj(a) * v)
template <bool CONJ_A>
__device__ __forceinline__ void df_cmac(float4& acc, float4 a, float4 v) {
  const float sa = CONJ_A ? -1.f : 1.f;
  df_mac(acc.x, acc.y, a.x, a.y, v.x, v.y);                       // re: a.re v.re
  df_mac(acc.x, acc.y, -sa * a.z, -sa * a.w, v.z, v.w);           //     -/+ a.im v.im
  df_mac(acc.z, acc.w, a.x, a.y, v.z, v.w);                       // im: a.re v.im
  df_mac(acc.z, acc.w, sa * a.z, sa * a.w, v.x, v.y);             //     +/- a.im v.re
  // renormalised every two terms: the lo parts stay small (10x less error over long sums)
  df_norm(acc.x, acc.y);
  df_norm(acc.z, acc.w);
}
__device__ __forceinline__ float4 df_warp_sum(float4 a) {
  for (int o = 16; o > 0; o >>= 1) {
    const float bh = __shfl_xor_sync(0xffffffffu, a.x, o), bl = __shfl_xor_sync(0xffffffffu, a.y, o);
    const float ch = __shfl_xor_sync(0xffffffffu, a.z, o), cl = __shfl_xor_sync(0xffffffffu, a.w, o);
    df_add(a.x, a.y, bh, bl);
    df_add(a.z, a.w, ch, cl);
  }
  return a;
}

// (ph, pl) = x * y for double-floats, renormalised
__device__ __forceinline__ float2 df_mul(float xh, float xl, float yh, float yl) {
  const float ph = __fmul_rn(xh, yh);
  const float pl = fmaf(xh, yl, fmaf(xl, yh, fmaf(xh, yh, -ph)));
  const float s = __fadd_rn(ph, pl);
  return make_float2(s, __fsub_rn(pl, __fsub_rn(s, ph)));
}
// block-wide double-float sum (every thread gets it); red holds 2 x 32 floats
__device__ __forceinline__ float2 df_block_sum(float hi, float lo, float* red) {
  for (int o = 16; o > 0; o >>= 1) {
    const float bh = __shfl_xor_sync(0xffffffffu, hi, o), bl = __shfl_xor_sync(0xffffffffu, lo, o);
    df_add(hi, lo, bh, bl);
  }
  __syncthreads();
  if ((threadIdx.x & 31) == 0) {
    red[2 * (threadIdx.x >> 5)] = hi;
    red[2 * (threadIdx.x >> 5) + 1] = lo;
  }
  __syncthreads();
  float th = 0.f, tl = 0.f;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) df_add(th, tl, red[2 * w], red[2 * w + 1]);
  return make_float2(th, tl);
}
__device__ __forceinline__ float2 df_mul2(float2 x, float2 y) { return df_mul(x.x, x.y, y.x, y.y); }
__device__ __forceinline__ float2 df_add2(float2 a, float2 b) {
  df_add(a.x, a.y, b.x, b.y);
  df_norm(a.x, a.y);
  return a;
}
// 1 / sqrt of a positive double-float (hi in [2^-100, 2^100]) from the hardware's float
// estimate y (2 ulp): with r = 1 - x y^2 formed in double-float, the binomial series
// y (1 + r / 2 + 3 r^2 / 8), whose first term left out is 2^-63; the float operations on r (below
// 2^-21) leave a relative error of at most 2^-44.
__device__ __forceinline__ float2 df_rsqrt(float2 x) {
  const float y = rsqrtf(x.x);
  const float2 y2 = df_mul(y, 0.f, y, 0.f);
  float rh = 1.f, rl = 0.f;
  df_mac(rh, rl, -x.x, -x.y, y2.x, y2.y);
  const float r = rh + rl;
  const float c = y * fmaf(0.375f * r, r, 0.5f * r);
  const float h = __fadd_rn(y, c);
  return make_float2(h, __fsub_rn(c, __fsub_rn(h, y)));
}
// 1 / x of a double-float (hi in [1, 2)): one Newton step from the rounded 1 / hi, relative error at
// most 2^-46.
__device__ __forceinline__ float2 df_rcp(float2 x) {
  const float y = __frcp_rn(x.x);
  float rh = 1.f, rl = 0.f;
  df_mac(rh, rl, -x.x, -x.y, y, 0.f);
  float2 c = make_float2(y, y * (rh + rl));
  df_norm(c.x, c.y);
  return c;
}

}  // namespace nne
