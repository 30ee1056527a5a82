// Pairs of FP32 values (head + tail, about 48 significant bits) for the kernel that turns FP64
// fields into FP32-arithmetic populations, and lossless sums of FP32 values for the one that turns
// those back.  GB300 issues FP64 at 1/64 of its FP32 rate (two lanes per SM and cycle), so those
// kernels, a few FP64 operations per population, were bound by the FP64 pipe and not by memory.  Sums
// by Knuth's two-sum, products by a fused multiply-add for the rounding error (Dekker 1971; Ogita,
// Rump & Oishi 2005); every rounding is explicit, so nothing is contracted.  FP64 storage runs the same
// templates in plain FP64.  Measured on a 128x128x512 box: initial fields + macroscopic fields
// 8.6 -> 1.6 ms (packed half), 9.4 -> 1.3 ms (FP32); FP64 storage gains from the smaller operation counts alone.
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
// Running sums of FP32 values without loss: head, middle and tail, 72 bits, so that the sum rounded to FP64
// is as good as one carried in FP64 (a sum in pairs is 2^-48 of its terms off).  The parts overlap; only
// their sum counts.
struct TF {
  float h, m, l;
};
__device__ __forceinline__ void acc_(double& a, double x) { a += x; }
__device__ __forceinline__ void acc_(TF& a, float x) {
  const DF s = two_sum(a.h, x), q = two_sum(a.m, s.l);
  a = {s.h, q.h, __fadd_rn(a.l, q.l)};
}
__device__ __forceinline__ void acc_(TF& a, TF b) {
  const DF s = two_sum(a.h, b.h), p = two_sum(a.m, b.m), q = two_sum(p.h, s.l);
  a = {s.h, q.h, __fadd_rn(__fadd_rn(a.l, b.l), __fadd_rn(p.l, q.l))};
}
__device__ __forceinline__ void sum2_(double& a, double x, double y) { a = x + y; }  // a = x + y
__device__ __forceinline__ void sum2_(TF& a, float x, float y) {
  const DF s = two_sum(x, y);
  a = {s.h, s.l, 0.f};
}
__device__ __forceinline__ TF neg_(TF a) { return {-a.h, -a.m, -a.l}; }
__device__ __forceinline__ double to_f64(double a) { return a; }
// a normal float or zero, times 2^e, as FP64 by integer operations (the conversion instruction issues at the FP64
// rate)
__device__ __forceinline__ double wide_bits(float v, int e = 0) {
  const unsigned b = __float_as_uint(v);
  const int hi = (int)((((b & 0x7fffffffu) >> 3) + (unsigned)((896 + e) << 20)) | (b & 0x80000000u));
  return (b << 1) == 0u ? 0.0 : __hiloint2double(hi, (int)(b << 29));
}
__device__ __forceinline__ double to_f64(TF a) {
  // the parts of a small sum are lifted by 2^80 on the way, so that none that counts is subnormal
  const bool small = fabsf(a.h) < 1e-18f;
  const float s = small ? 0x1p80f : 1.0f;
  const int e = small ? -80 : 0;
  return wide_bits(a.h * s, e) + (wide_bits(a.m * s, e) + wide_bits(a.l * s, e));
}
// a sum that met no overflow, infinity or NaN
__device__ __forceinline__ bool whole_(double) { return true; }
__device__ __forceinline__ bool whole_(TF a) { return fabsf(a.h) < 1e37f; }

// the type of a storage's wide arithmetic and of its sums, by its compute type
template <typename R>
struct WideOf { using type = double; };
template <>
struct WideOf<float> { using type = DF; };
template <typename R>
struct SumOf { using type = double; };
template <>
struct SumOf<float> { using type = TF; };

}  // namespace lbmk
