// Plan entries B(x,y) = exp(a(x) + b(y) - C(x,y)/eps) in double-float arithmetic
// (pairs of FP32 values with error-free transformations), shared by the FP64-grade
// check and the rounding kernels: the exponent is exact to ~1e-12 before one
// accurate expf of its high part, so every entry has ~1e-7 relative error with no
// systematic part, at FP32-pipe speed (FP64 runs at a small fraction of that here).
#pragma once
#include <cuda_runtime.h>

#include "internal.h"

namespace treeot {

struct DF {
  float hi, lo;
};

// The error-free transformations below use the _rn intrinsics, which the
// compiler never contracts into FMAs: a product fused into a neighbouring
// addition would no longer be the rounded value the error term was taken from.
__device__ __forceinline__ DF two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return {s, e};
}

// exact-ish square of (p - q) as a double-float
__device__ __forceinline__ DF sq_diff(float p, float q) {
  const DF d = two_sum(p, -q);
  const float h = __fmul_rn(d.hi, d.hi);
  const float e = fmaf(2.f * d.hi, d.lo, fmaf(d.hi, d.hi, -h));
  return {h, e};
}

__device__ __forceinline__ DF df_add(DF a, DF b) {
  const DF s = two_sum(a.hi, b.hi);
  return {s.hi, s.lo + a.lo + b.lo};
}

// lo back below half an ulp of hi (|hi| >= |lo|), so that adding to it stays exact to ~2^-48
__device__ __forceinline__ void df_renorm(DF& s) {
  const float t = __fadd_rn(s.hi, s.lo);
  s.lo = __fsub_rn(s.lo, __fsub_rn(t, s.hi));
  s.hi = t;
}

// Running sums as three floats: every rounding error of the first is summed in the second, the second's in the
// third.  A sum of n terms carries about n^2 2^-72 relative, less than one FP64 addition (2^-53) for any support
// here, where pairs of floats would leave n 2^-48; FP64 itself runs at 1/70 of the FP32 rate.
struct TF {
  float a, b, c;
};
__device__ __forceinline__ void tf_acc(TF& s, float v) {  // s += v
  const DF t = two_sum(s.a, v), u = two_sum(s.b, t.lo);
  s = {t.hi, u.hi, s.c + u.lo};
}
__device__ __forceinline__ void tf_acc(TF& s, float p, float m) {  // s += p + m
  const DF t = two_sum(s.a, p), u = two_sum(s.b, t.lo), v = two_sum(u.hi, m);
  s = {t.hi, v.hi, s.c + (u.lo + v.lo)};
}
__device__ __forceinline__ void tf_acc(TF& s, TF v) {
  tf_acc(s, v.a, v.b);
  s.c += v.c;
}
__device__ __forceinline__ double tf_to(TF s) { return (double)s.a + ((double)s.b + (double)s.c); }
__device__ __forceinline__ TF tf_of(double v) {
  const float a = (float)v;
  const double r = v - (double)a;
  const float b = (float)r;
  return {a, b, (float)(r - (double)b)};
}
// x v as three floats, x v.a exactly (as long as it neither overflows nor falls below 2^-102)
__device__ __forceinline__ TF tf_mul(float x, TF v) {
  const float p = __fmul_rn(x, v.a), q = __fmul_rn(x, v.b);
  const DF m = two_sum(fmaf(x, v.a, -p), q);
  return {p, m.hi, fmaf(x, v.c, m.lo + fmaf(x, v.b, -q))};
}
// finite: no sum on the way to it overflowed (an overflow leaves inf or NaN in every part that follows)
__device__ __forceinline__ bool tf_finite(TF s) { return fabsf(s.a) <= 3.4028235e38f; }

// Sums of eight per-lane values across the warp: the lanes trade halves of their values, so that each step adds half
// as many; every lane ends with the sum of value lane / 4.
__device__ __forceinline__ TF warp_rows_sum(TF (&v)[8]) {
  const int lane = threadIdx.x & 31;
  auto trade = [](TF keep, TF give, int o) {
    tf_acc(keep, TF{__shfl_xor_sync(0xffffffffu, give.a, o), __shfl_xor_sync(0xffffffffu, give.b, o),
                    __shfl_xor_sync(0xffffffffu, give.c, o)});
    return keep;
  };
#pragma unroll
  for (int h = 4; h >= 1; h >>= 1) {
    const int o = 4 * h;
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < h; ++i) v[i] = trade(up ? v[i + h] : v[i], up ? v[i] : v[i + h], o);
  }
  v[0] = trade(v[0], v[0], 2);
  return trade(v[0], v[0], 1);
}

// squared distance of two D-dimensional FP32 points (D <= 3) as a double-float
__device__ __forceinline__ DF sq_dist_df(int D, const float* pa, const float* pb) {
  DF c = sq_diff(pa[0], pb[0]);
  if (D > 1) c = df_add(c, sq_diff(pa[1], pb[1]));
  if (D > 2) c = df_add(c, sq_diff(pa[2], pb[2]));
  return c;
}

// C(x,y) as a double-float (rows x of the stored matrix); dense costs are exact FP32 values
__device__ __forceinline__ DF cost_df(const EdgeD& e, const ProbD& P, int x, int y, const float* pa,
                                     const float* pb) {
  if (P.cost_kind == 0) return {e.C[(int64_t)x * e.ld + y], 0.f};
  return sq_dist_df(P.dim, pa, pb);
}

// B = exp(a + b - C * k), k = scale / eps as (kh, kl); returns B and, in cost_out,
// C / scale rounded to FP32
__device__ __forceinline__ float plan_entry(float ah, float al, float bh, float bl, DF c, float kh, float kl,
                                            float& cost_out) {
  const DF s = two_sum(ah, bh);
  const float p = __fmul_rn(c.hi, kh);  // the rounded product; pe holds what it lost
  const float pe = fmaf(c.hi, kl, fmaf(c.lo, kh, fmaf(c.hi, kh, -p)));
  const DF d = two_sum(s.hi, -p);
  const float lo = (s.lo + d.lo) + (al + bl) - pe;
  cost_out = c.hi + c.lo;
  const float E = expf(d.hi);
  return E == 0.f ? 0.f : E * (1.f + lo);
}

}  // namespace treeot
