// Pairs of FP32 values (head + tail, about 48 significant bits) for the kernels that turn FP64
// fields into FP32-arithmetic populations and back.  GB300 issues FP64 at 1/64 of its FP32 rate
// (two lanes per SM and cycle), so those kernels, a few FP64 operations per population, were
// bound by the FP64 pipe and not by memory.  Sums by Knuth's two-sum, products by a fused
// multiply-add for the rounding error (Dekker 1971; Ogita, Rump & Oishi 2005); every rounding is
// explicit, so nothing is contracted.  The same templates run in plain FP64 for FP64 storage.
// Measured on a 128x128x512 box: initial fields + macroscopic fields 8.6 -> 1.6 ms (packed half),
// 9.4 -> 1.3 ms (FP32); FP64 storage gains from the smaller operation counts alone.
#pragma once
#include <cuda_runtime.h>

namespace lbmk {

struct DF {
  float h, l;
};

template <typename T>
__device__ __forceinline__ T wide_(double c);  // a constant, or one FP64 input
template <>
__device__ __forceinline__ double wide_<double>(double c) { return c; }
template <>
__device__ __forceinline__ DF wide_<DF>(double c) {
  const float h = (float)c;
  return {h, (float)(c - (double)h)};
}
__device__ __forceinline__ double narrow_(double a) { return a; }
__device__ __forceinline__ float narrow_(DF a) { return __fadd_rn(a.h, a.l); }
__device__ __forceinline__ double to_f64(double a) { return a; }
__device__ __forceinline__ double to_f64(DF a) { return (double)a.h + (double)a.l; }

// s + e = a + b exactly
__device__ __forceinline__ DF two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ DF renorm(float h, float l) {  // |h| >= |l|
  const float s = __fadd_rn(h, l);
  return {s, __fsub_rn(l, __fsub_rn(s, h))};
}
__device__ __forceinline__ double add_(double a, double b) { return a + b; }
__device__ __forceinline__ DF add_(DF a, DF b) {
  const DF s = two_sum(a.h, b.h);
  return renorm(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ double neg_(double a) { return -a; }
__device__ __forceinline__ DF neg_(DF a) { return {-a.h, -a.l}; }
__device__ __forceinline__ double sub_(double a, double b) { return a - b; }
__device__ __forceinline__ DF sub_(DF a, DF b) { return add_(a, neg_(b)); }
__device__ __forceinline__ double mul_(double a, double b) { return a * b; }
__device__ __forceinline__ DF mul_(DF a, DF b) {
  const float p = __fmul_rn(a.h, b.h);
  return renorm(p, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p))));
}
__device__ __forceinline__ double mad_(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ DF mad_(DF a, DF b, DF c) {
  const float p = __fmul_rn(a.h, b.h);
  const float e = __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p)));
  const DF s = two_sum(c.h, p);
  return renorm(s.h, __fadd_rn(s.l, __fadd_rn(c.l, e)));
}
// a / b: quotient of the heads, corrected once by the remainder (a few units of 2^-46)
__device__ __forceinline__ double div_(double a, double b) { return a / b; }
__device__ __forceinline__ DF div_(DF a, DF b) {
  const float q = __fdiv_rn(a.h, b.h);
  const float r = __fmaf_rn(-q, b.h, a.h);  // exact
  return renorm(q, __fdiv_rn(__fadd_rn(r, __fmaf_rn(-q, b.l, a.l)), b.h));
}
// running sums: the tail is not renormalised
__device__ __forceinline__ void acc_(double& a, double x) { a += x; }
__device__ __forceinline__ void acc_(DF& a, float x) {
  const DF s = two_sum(a.h, x);
  a = {s.h, __fadd_rn(a.l, s.l)};
}
__device__ __forceinline__ void acc_(DF& a, DF b) {
  const DF s = two_sum(a.h, b.h);
  a = {s.h, __fadd_rn(__fadd_rn(a.l, b.l), s.l)};
}

// the wide type of a storage's compute type
template <typename R>
struct WideOf { using type = double; };
template <>
struct WideOf<float> { using type = DF; };

}  // namespace lbmk
