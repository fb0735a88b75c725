// FP64 operations that keep off the FP64 pipe.  On this part a scheduler's FP64 pipe takes one warp
// instruction per 64 clocks, whatever the number of active lanes, and the kernels around the sweeps
// are bound by it (ncu: FP64 pipe active 70-85 % of the active cycles in every one of them).
// Conversions between FP32 and FP64 and comparisons of FP64 values count as such instructions; the
// integer pipe takes one per two clocks.  So exact conversions are done on the bit patterns, and a
// reciprocal is four FP64 instructions (a quotient with it three more) instead of the nine of an IEEE division.
#pragma once
#include <cuda_runtime.h>

namespace fasw {

// (double)x, exactly.  Subnormals, infinities and NaNs take the conversion instruction.
__device__ __forceinline__ double f2d(float x) {
  const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
  if (m - 0x00800000u >= 0x7f000000u && m != 0u) return (double)x;
  const unsigned hi = m ? (m >> 3) + 0x38000000u : 0u;
  return __hiloint2double((int)(hi | (b & 0x80000000u)), (int)(b << 29));
}

// (float)x, rounded to nearest even.  Results that are not normal numbers (zero, subnormal, values
// that round past the largest float, infinities, NaNs) take the conversion instruction.
__device__ __forceinline__ float d2f(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x), m = hi & 0x7fffffffu;
  if (m - 0x38100000u >= 0x0fd00000u) return (float)x;
  unsigned f = ((m - 0x38000000u) << 3) | (lo >> 29);
  const unsigned rest = lo & 0x1fffffffu;
  f += rest > 0x10000000u || (rest == 0x10000000u && (f & 1u)) ? 1u : 0u;  // a carry moves into the exponent
  return __uint_as_float(f | (hi & 0x80000000u));
}

// 1/x: two Newton steps y <- y (2 - x y) from the hardware's approximation (relative error below 2^-18),
// which leave a truncation error of 2^-72 before the last rounding: the bits of the division but for a few
// arguments in a million whose reciprocal lies next to a tie.  Zero, subnormals, infinities, NaNs and 2^1021
// and above (whose reciprocals the approximation flushes to zero) take the division, out of line (inline it
// costs the 256x64 FP64 W-cycle 0.8 %, out of line 0.5: 6.93 -> 6.97 ms).
static __device__ __noinline__ double rcp64_rare(double x) { return 1.0 / x; }
__device__ __forceinline__ double rcp64(double x) {
  if (__builtin_expect(((unsigned)__double2hiint(x) & 0x7fffffffu) - 0x00100000u >= 0x7fb00000u, 0)) return rcp64_rare(x);
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  y = fma(fma(-x, y, 1.0), y, y);
  return fma(fma(-x, y, 1.0), y, y);
}

// a / b, rb = rcp64(b): the product with the reciprocal and one correction by its remainder (Markstein, IBM J. Res.
// Dev. 34, 1990), which give the division's rounding where the product alone is off by up to one and a half units in
// the last place.  Where there is no remainder (zero or infinite b, overflow) the product stands.
__device__ __forceinline__ double div64(double a, double b, double rb) {
  const double q = a * rb, c = fma(fma(-q, b, a), rb, q);
  return ((unsigned)__double2hiint(c) & 0x7fffffffu) > 0x7ff00000u ? q : c;
}

// x in the precision of T
template <typename T>
__device__ __forceinline__ T from64(double x);
template <>
__device__ __forceinline__ double from64<double>(double x) {
  return x;
}
template <>
__device__ __forceinline__ float from64<float>(double x) {
  return d2f(x);
}
__device__ __forceinline__ double to64(double x) { return x; }
__device__ __forceinline__ double to64(float x) { return f2d(x); }

// fmax of two non-negative values, fmin of x and a positive c: on the bit patterns, whose order as signed
// integers is that of the values.  As with fmax and fmin a NaN gives way to the other (a cell of negative
// pressure has a NaN for its sound speed; its faces take their neighbours' radii).  The upper word of a
// NaN that an operation returns is above that of infinity, with either sign.
__device__ __forceinline__ double max_nn(double a, double b) {
  const bool nan = (unsigned)__double2hiint(a) > 0x7ff00000u, other = (unsigned)__double2hiint(b) > 0x7ff00000u;
  return !nan && (other || __double_as_longlong(a) > __double_as_longlong(b)) ? a : b;
}
__device__ __forceinline__ double min_pos(double x, double c) {
  const bool nan = (unsigned)__double2hiint(x) > 0xfff00000u;  // a negative one; a positive one is above c
  return !nan && __double_as_longlong(x) < __double_as_longlong(c) ? x : c;
}
// fmax(x, 0)
__device__ __forceinline__ double relu64(double x) { return (unsigned)__double2hiint(x) > 0x7ff00000u ? 0.0 : x; }
__device__ __forceinline__ bool is_zero(double x) { return ((__double2hiint(x) << 1) | __double2loint(x)) == 0; }

}  // namespace fasw
