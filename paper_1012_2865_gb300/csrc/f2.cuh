// f2.cuh -- double-float arithmetic: a value carried as an unevaluated sum
// of two FP32 numbers (hi, lo) with |lo| <= ulp(hi)/2, about 48 significant
// bits.  Error-free transformations after Knuth (two_sum), Dekker
// (fast_two_sum, |a| >= |b|) and the FMA product error (two-product).
#pragma once
#include <cuda_runtime.h>
#include <math.h>

namespace rtg {

struct F2 {
  float hi, lo;
};
__device__ __forceinline__ F2 two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  const float err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return {s, err};
}
__device__ __forceinline__ F2 fast_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, e));
  return fast_two_sum(p, e);
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
  F2 s = two_sum(a.hi, b.hi);
  return fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
// a - b as FP32 (both pairs), accurate to ~2^-44 |a|
__device__ __forceinline__ float f2_diff(F2 a, F2 b) {
  const F2 d = two_sum(a.hi, -b.hi);
  return __fadd_rn(d.hi, __fadd_rn(d.lo, __fsub_rn(a.lo, b.lo)));
}
__device__ __forceinline__ bool f2_eq(F2 a, F2 b) { return a.hi == b.hi && a.lo == b.lo; }
// 1 / (n.hi + n.lo) as a pair: the approximate reciprocal (2^-23), one Newton
// step in FP32, one for the low part (|n| in the normal range's middle, as
// direction components are)
__device__ __forceinline__ F2 f2_recip(F2 n) {
  const float q0 = __fdividef(1.0f, n.hi);
  const float q = fmaf(fmaf(-n.hi, q0, 1.0f), q0, q0);
  float e = fmaf(-n.hi, q, 1.0f);
  e = fmaf(-n.lo, q, e);
  return fast_two_sum(q, __fmul_rn(e, q));
}
__device__ __forceinline__ int f2_floor(F2 u) {
  const float f = floorf(u.hi);
  if (u.hi == f && u.lo < 0.0f) return (int)f - 1;
  return (int)f;
}

// a - b as a pair
__device__ __forceinline__ F2 f2_sub(F2 a, F2 b) { return f2_add(a, F2{-b.hi, -b.lo}); }
// pair times an FP32 number
__device__ __forceinline__ F2 f2_mul_f(F2 a, float b) {
  const float p = __fmul_rn(a.hi, b);
  const float e = fmaf(a.lo, b, fmaf(a.hi, b, -p));
  return fast_two_sum(p, e);
}
// nearest pair to an FP64 value (v - hi is exact in FP64)
__device__ __forceinline__ F2 f2_from_double(double v) {
  const float hi = __double2float_rn(v);
  return {hi, __double2float_rn(__dsub_rn(v, (double)hi))};
}

// That conversion and the one back with the format changes done in integer
// arithmetic (IEEE-754 binary64 / binary32 fields), for kernels where the
// FP64 pipe, a small fraction of the FP32 one, would otherwise bound them.
//
// Nearest pair to v: hi = v rounded to 24 bits (ties to even; a carry moves
// into the exponent as it should), lo the FP32 rounding of v - hi, an integer
// of at most 2^28 units of v's last place.  Equal to f2_from_double for zeros
// and 2^-74 <= |v| < 2^125, which it handles this way (hi and lo stay normal
// FP32 numbers); other values take f2_from_double.  All in 32-bit words:
// 64-bit integer additions share the FP64 pipe here, and it bound the kernels
// that convert a field (a 256^3 read of the rates: 102 -> 71 us without them).
// The rare operands of these conversions go through functions that are
// never inlined, so the compiler cannot predicate their FP64 instructions
// into the common path.
static __device__ __noinline__ F2 f2_from_double_call(double v) { return f2_from_double(v); }
static __device__ __noinline__ double f32_widen_call(float f) { return (double)f; }
__device__ __forceinline__ F2 f2_from_double_bits(double v) {
  const unsigned uh = (unsigned)__double2hiint(v), ul = (unsigned)__double2loint(v);
  const unsigned mh = uh & 0x7fffffffu, sign = uh & 0x80000000u;
  if (mh - (949u << 20) >= (199u << 20)) {  // outside 2^-74 .. 2^125
    if ((mh | ul) == 0u) return {__uint_as_float(sign), 0.0f};  // signed zero
    return f2_from_double_call(v);
  }
  unsigned m = ((mh - (896u << 20)) << 3) | (ul >> 29);
  const unsigned rem = ul & 0x1fffffffu;
  const bool up = rem > 0x10000000u - (m & 1u);
  m += up;
  const int d = (int)rem - (up ? 0x20000000 : 0);  // |v| - |hi|, units of 2^(e - 1075)
  const float lo = __fmul_rn(__int2float_rn(d), __uint_as_float(((mh >> 20) - 948u) << 23));  // |d| <= 2^28
  return {__uint_as_float(sign | m), sign ? -lo : lo};
}
// An FP32 number widened to binary64 exactly by moving its fields (normal
// numbers and zeros; others take the conversion instruction).
__device__ __forceinline__ double f32_widen_bits(float f) {
  const unsigned b = __float_as_uint(f);
  const unsigned ex = (b >> 23) & 0xffu;
  if (ex == 0u || ex == 0xffu) {
    if ((b << 1) == 0u) return __longlong_as_double((long long)((unsigned long long)b << 32));
    return f32_widen_call(f);
  }
  const unsigned hi = (b & 0x80000000u) | ((ex + 896u) << 20) | ((b & 0x7fffffu) >> 3);
  return __hiloint2double((int)hi, (int)(b << 29));
}
// hi + lo rounded to binary64 with one FP64 addition.
__device__ __forceinline__ double f2_to_double_bits(F2 a) { return __dadd_rn(f32_widen_bits(a.hi), f32_widen_bits(a.lo)); }
// 1 / v and 1 / sqrt(v) to ~2^-23, v in the normal range (no fix-up of
// subnormal operands)
__device__ __forceinline__ float rcp_approx(float v) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}
__device__ __forceinline__ float rsqrt_approx(float v) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}
// Chopped FP32 value of a double (relative error below 2^-23; below the FP32
// normal range: 0), and an FP32 number as a double (subnormals: 0), by moving
// the fields: for corrections that are themselves only good to FP32.
__device__ __forceinline__ float f32_chop(double v) {
  const int hi = __double2hiint(v);
  const int e = ((hi >> 20) & 0x7ff) - 896;
  const unsigned m = ((unsigned)e << 23) | ((unsigned)(hi & 0xfffff) << 3) | ((unsigned)__double2loint(v) >> 29);
  return __uint_as_float(((unsigned)hi & 0x80000000u) | (e > 0 ? m : 0u));
}
__device__ __forceinline__ double f64_wide(float f) {
  const unsigned b = __float_as_uint(f);
  const unsigned hi = (b & 0x80000000u) | ((((b >> 23) & 0xffu) + 896u) << 20) | ((b & 0x7fffffu) >> 3);
  return (b & 0x7f800000u) ? __hiloint2double((int)hi, (int)(b << 29)) : 0.0;
}

}  // namespace rtg
