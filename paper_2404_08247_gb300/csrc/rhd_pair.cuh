// rhd_pair.cuh -- arithmetic on unevaluated sums of two floats.
//
// A pair hi + lo carries about 48 bits (|lo| <= ulp(hi)/2), with float's
// exponent range.  The error-free sum is Knuth's two-sum, the error-free
// product uses the fused multiply-add (Dekker 1971; Knuth, The Art of
// Computer Programming, vol. 2, Sec. 4.2.2; Hida, Li & Bailey 2001).  The
// single-precision pipe of this GPU has 64 times the throughput of the
// double-precision one, so an operation on pairs (4 to 11 instructions) costs
// a fraction of a double-precision one's pipe time.  Sums are renormalised (a
// cancellation may leave everything in lo); products, reciprocals and roots
// are not, their lo being a few ulps of hi at most.  Results are good to a few
// 2^-47 of the operands: enough to bring an iteration next to its fixed point,
// which a double-precision pass then settles.
#pragma once

#include <cuda_runtime.h>

namespace rhd {

struct Pair {
  float hi, lo;
};

__device__ __forceinline__ Pair pair_of(float a) { return {a, 0.f}; }
// hi + lo with |hi| >= |lo|, renormalised
__device__ __forceinline__ Pair pair_norm(float a, float b) {
  const float s = __fadd_rn(a, b);
  return {s, __fadd_rn(b, -__fadd_rn(s, -a))};
}
__device__ __forceinline__ Pair operator-(Pair a) { return {-a.hi, -a.lo}; }
__device__ __forceinline__ Pair operator+(Pair a, Pair b) {
  const float s = __fadd_rn(a.hi, b.hi);
  const float t = __fadd_rn(s, -a.hi);
  const float e = __fadd_rn(__fadd_rn(a.hi, -__fadd_rn(s, -t)), __fadd_rn(b.hi, -t));
  return pair_norm(s, __fadd_rn(e, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ Pair operator-(Pair a, Pair b) { return a + (-b); }
__device__ __forceinline__ Pair operator*(Pair a, Pair b) {
  const float p = __fmul_rn(a.hi, b.hi);
  const float e = __fmaf_rn(a.lo, b.hi, __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.hi, b.hi, -p)));
  return {p, e};
}
__device__ __forceinline__ Pair operator*(Pair a, float b) {
  const float p = __fmul_rn(a.hi, b);
  return {p, __fmaf_rn(a.lo, b, __fmaf_rn(a.hi, b, -p))};
}
// product with a power of two (exact)
__device__ __forceinline__ Pair scaled(Pair a, float s) { return {a.hi * s, a.lo * s}; }
__device__ __forceinline__ Pair operator+(Pair a, float b) {
  const float s = __fadd_rn(a.hi, b);
  const float t = __fadd_rn(s, -a.hi);
  const float e = __fadd_rn(__fadd_rn(a.hi, -__fadd_rn(s, -t)), __fadd_rn(b, -t));
  return pair_norm(s, __fadd_rn(e, a.lo));
}
// 1/a: a float reciprocal r and the first two terms of r (1 + e + e^2 + ..),
// e = 1 - a r
__device__ __forceinline__ Pair recip(Pair a) {
  const float r = __fdividef(1.f, a.hi);
  const float e = __fmaf_rn(-a.lo, r, __fmaf_rn(-a.hi, r, 1.f));
  return {r, __fmul_rn(r, __fmaf_rn(e, e, e))};
}
// sqrt(a), a > 0: s = a rsqrt(a) and one Newton correction
__device__ __forceinline__ Pair root(Pair a) {
  const float y = rsqrtf(a.hi);
  const float s = __fmul_rn(a.hi, y);
  const float t = __fadd_rn(__fmaf_rn(-s, s, a.hi), a.lo);
  return {s, __fmul_rn(t, 0.5f * y)};
}

// x 2^-s as a pair, by integer operations and one 32-bit conversion: hi is x
// with its mantissa cut to 24 bits, lo the next 29 rounded to 24.  Below 2^-70
// the pair is zero; false (and zero) where x 2^-s exceeds the float range or x
// is not finite.  s > -953, so that a zero or subnormal x counts as below 2^-70.
__device__ __forceinline__ bool split_scaled(double x, int s, Pair& p) {
  const long long b = __double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ff) - s;  // biased exponent of x 2^-s
  p.hi = p.lo = 0.f;
  if (e > 1023 + 126) return false;
  if (e < 1023 - 70) return true;
  const unsigned sign = (unsigned)((b >> 32) & 0x80000000ll);
  p.hi = __uint_as_float(sign | ((unsigned)(e - 896) << 23) | (unsigned)((b >> 29) & 0x7fffff));
  // lo = (low 29 bits) 2^(e - 1023 - 52), with the sign of x
  const float u = (float)(unsigned)(b & 0x1fffffffll);
  p.lo = u * __uint_as_float(sign | ((unsigned)(e - 896 - 52) << 23));
  return true;
}

// hi + lo as a double times 2^s, |s| <= 895 (a double addition; the widening by
// integer operations, a float below the normal range counting as zero)
__device__ __forceinline__ double widened(float f, int s) {
  const unsigned u = __float_as_uint(f);
  if ((u & 0x7f800000u) == 0u) return 0.0;
  const long long m = ((long long)(u & 0x7fffffffu) << 29) + ((long long)(896 + s) << 52);
  return __longlong_as_double(m | ((long long)(u & 0x80000000u) << 32));
}
__device__ __forceinline__ double widened(Pair p, int s) {
  return widened(p.hi, s) + widened(p.lo, s);
}

}  // namespace rhd
