// dfloat.cuh - FP64 work done on the FP32 pipe.
//
// GB300 issues one FP64 instruction per 64 cycles and SM sub-partition, an FP32
// one every cycle, so sums and products whose error is carried along exactly
// in FP32 (Knuth's TwoSum, Dekker's Fast2Sum, the fused multiply-add form of
// TwoProduct) cost a tenth of the FP64 operations they stand for.
//
// DF: an unevaluated sum hi + lo of two floats, relative error about 2^-46
// per operation: for results that are rounded to FP32 in the end.  F3: a sum
// of floats in three terms, beyond FP64's precision: for sums that end in FP64.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace mrtlb {

// s + e = a + b exactly
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
  const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return s;
}

struct DF {
  float hi, lo;
};
__device__ __forceinline__ DF df_norm(float s, float e) {  // |s| >= |e|
  const float h = __fadd_rn(s, e);
  return DF{h, __fsub_rn(e, __fsub_rn(h, s))};
}
__device__ __forceinline__ DF df_add(DF a, DF b) {
  float e;
  const float s = two_sum(a.hi, b.hi, e);
  return df_norm(s, __fadd_rn(e, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ DF df_neg(DF a) { return DF{-a.hi, -a.lo}; }
__device__ __forceinline__ DF df_sub(DF a, DF b) { return df_add(a, df_neg(b)); }
__device__ __forceinline__ DF df_scale(DF a, float p) { return DF{a.hi * p, a.lo * p}; }  // p: a power of two
__device__ __forceinline__ DF df_mul(DF a, DF b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  return df_norm(p, __fmaf_rn(a.lo, b.hi, e));
}
__device__ __forceinline__ DF df_mul(DF a, float b) {
  const float p = __fmul_rn(a.hi, b);
  return df_norm(p, __fmaf_rn(a.lo, b, __fmaf_rn(a.hi, b, -p)));
}
// s + c += k x, c the running sum of the errors (not normalised)
__device__ __forceinline__ void df_accumulate(DF& a, DF k, DF x) {
  const float p = __fmul_rn(k.hi, x.hi);
  float ep = __fmaf_rn(k.hi, x.hi, -p), e;
  ep = __fmaf_rn(k.lo, x.hi, __fmaf_rn(k.hi, x.lo, ep));
  a.hi = two_sum(a.hi, p, e);
  a.lo = __fadd_rn(a.lo, __fadd_rn(e, ep));
}
__device__ __forceinline__ DF df_first(DF k, DF x) {
  const float p = __fmul_rn(k.hi, x.hi);
  return DF{p, __fmaf_rn(k.lo, x.hi, __fmaf_rn(k.hi, x.lo, __fmaf_rn(k.hi, x.hi, -p)))};
}
__device__ __forceinline__ DF df_join(DF a, DF b) {
  float e;
  const float s = two_sum(a.hi, b.hi, e);
  return DF{s, __fadd_rn(e, __fadd_rn(a.lo, b.lo))};
}
// Zero or a magnitude in [2^-60, 2^60): what df_of takes (products of such
// values may still pass FP32's range).
__device__ __forceinline__ bool df_fits(double x) {
  const uint32_t h = (uint32_t)__double2hiint(x) & 0x7fffffffu;
  return x == 0.0 || (h >= (uint32_t)(1023 - 60) << 20 && h < (uint32_t)(1023 + 60) << 20);
}
// The leading 24 bits of x, cut, and what they leave, by its bits (a
// conversion instruction runs on the FP64 pipe).
__device__ __forceinline__ DF df_of(double x) {
  const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
  const uint32_t sign = h & 0x80000000u;
  const uint32_t mag = __funnelshift_l(l, h & 0x7fffffffu, 3) - (896u << 23);
  const float unit = __uint_as_float(sign | ((mag & 0x7f800000u) - (52u << 23)));
  const DF r{__uint_as_float(sign | mag), (float)(l & 0x1fffffffu) * unit};
  return (x == 0.0) ? DF{0.0f, 0.0f} : r;
}

// A sum of floats: a + b + c, every error of a's additions in b and of b's in
// c (whose own errors, 2^-72 of the sum, are dropped).
struct F3 {
  float a, b, c;
};
__device__ __forceinline__ F3 f3_of(float x, float y) {
  F3 s;
  s.a = two_sum(x, y, s.b);
  s.c = 0.0f;
  return s;
}
__device__ __forceinline__ void f3_add(F3& s, float x) {
  float e, e2;
  s.a = two_sum(s.a, x, e);
  s.b = two_sum(s.b, e, e2);
  s.c = __fadd_rn(s.c, e2);
}
// The value of a float as a double by its bits; zeros, subnormals, infinities
// and NaNs by the conversion.
__device__ __forceinline__ double wide(float x) {
  const uint32_t u = __float_as_uint(x), m = u & 0x7fffffffu;
  if (m - 0x00800000u >= 0x7f000000u) return (double)x;
  return __hiloint2double((int)((u & 0x80000000u) | ((m >> 3) + (896u << 20))), (int)(m << 29));
}
__device__ __forceinline__ double f3_value(const F3& s) {
  // (floats of nearly one size leave c empty, and a + b is then rounded once)
  const double v = wide(s.a) + wide(s.b);
  return (s.c == 0.0f) ? v : v + wide(s.c);
}

}  // namespace mrtlb
