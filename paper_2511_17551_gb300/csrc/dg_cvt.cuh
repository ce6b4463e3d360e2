// FP64 <-> FP32 conversions by integer work, bit for bit the conversion instructions' results
// (round to nearest even).  Those run at the rate of the FP64 pipe, a sixtieth of the integer
// rate, and bounded the kernels that split or merge the compensated FP32 state (85 % of the pipe).
// Zeros and finite values in FP32's normal range take about ten integer operations, as do doubles that
// round to zero (the low part of a value that FP32 holds); FP32's subnormals take about twenty
// more, and values out of range, infinities and NaN the instruction, in functions of their own: inline
// it is predicated and takes its time on the pipe for every value.  10.5 M values: split 78 -> 27 us,
// merge 62 -> 26 us (168 MB: 25 us at the copy bandwidth).  A state of zeros, 32^3 elements, N = 3:
// 40 us a call to set and 55 to get, as any other; with the instruction for zeros 93 and 90, and one of
// FP32 values (low parts zero) 56 and 77.
#pragma once

// |x| < 2^-126 or not finite in FP32
static __device__ __noinline__ float f64_to_f32_any(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)(b >> 52) & 0x7ff;
  if (e > 0x380) return (float)x;
  const int s = 29 + (0x381 - e);  // below the last bit of a subnormal, 2^-149; e > 0x368: s < 54
  const unsigned long long m = (b & 0xfffffffffffffull) | 0x10000000000000ull, half = 1ull << (s - 1);
  const unsigned q = (unsigned)(m >> s), r = (m & (2 * half - 1)) + (q & 1u) > half;
  return __uint_as_float((q + r) | ((unsigned)(b >> 32) & 0x80000000u));
}
// subnormal, infinite, NaN
static __device__ __noinline__ double f32_to_f64_any(float x) {
  const unsigned b = __float_as_uint(x), a = b & 0x7fffffffu;
  if (a >= 0x7f800000u) return (double)x;
  const int p = __clz((int)a) - 8;  // to the leading bit's place, 1 to 23
  const unsigned m = (a << p) & 0x7fffffu;
  return __hiloint2double((int)((((unsigned)(0x381 - p) << 20) + (m >> 3)) | (b & 0x80000000u)), (int)(m << 29));
}
__device__ __forceinline__ float f64_to_f32(double x) {
  const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x), a = h & 0x7fffffffu;
  const bool zero = a < 0x36900000u;  // |x| < 2^-150
  if (a - 0x38100000u >= 0x47f00000u - 0x38100000u && !zero) return f64_to_f32_any(x);  // not 2^-126 <= |x| < 2^128
  // exponent and 23 bits of the mantissa, then the 29 bits below them; a carry of the rounding runs
  // into the exponent, up to that of infinity
  unsigned m = __funnelshift_l(l, a - 0x38000000u, 3);
  m += ((l << 3) + (m & 1u)) > 0x80000000u;
  return __uint_as_float((zero ? 0u : m) | (h & 0x80000000u));
}
__device__ __forceinline__ double f32_to_f64(float x) {
  const unsigned b = __float_as_uint(x), a = b & 0x7fffffffu;
  if (a - 0x00800000u >= 0x7f800000u - 0x00800000u && a) return f32_to_f64_any(x);
  return __hiloint2double((int)((a ? (a >> 3) + 0x38000000u : 0u) | (b & 0x80000000u)), (int)(a << 29));
}

template <typename T> __device__ __forceinline__ T narrow(double x);
template <> __device__ __forceinline__ double narrow<double>(double x) { return x; }
template <> __device__ __forceinline__ float narrow<float>(double x) { return f64_to_f32(x); }
// x = hi + lo, hi = fl32(x), lo = fl32(x - hi)
__device__ __forceinline__ void split_f64(double x, float& hi, float& lo) {
  hi = f64_to_f32(x);
  lo = f64_to_f32(x - f32_to_f64(hi));
}
__device__ __forceinline__ double merge_f64(float hi, float lo) { return f32_to_f64(hi) + f32_to_f64(lo); }

// Without a slow path, for the middle of heavier kernels (the call would cost them registers):
// magnitudes below 2^-126 become zeros, and a double of 2^128 and more becomes NaN.
__device__ __forceinline__ float f64_to_f32_mid(double x) {
  const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x), a = h & 0x7fffffffu;
  unsigned m = __funnelshift_l(l, a - 0x38000000u, 3);
  m += ((l << 3) + (m & 1u)) > 0x80000000u;
  m = a < 0x38100000u ? 0u : m;
  m = a >= 0x47f00000u ? 0x7fffffffu : m;
  return __uint_as_float(m | (h & 0x80000000u));
}
__device__ __forceinline__ double f32_to_f64_mid(float x) {
  const unsigned b = __float_as_uint(x), a = b & 0x7fffffffu;
  const bool tiny = a < 0x00800000u;
  unsigned h = tiny ? 0u : (a >> 3) + 0x38000000u;
  h = a >= 0x7f800000u ? h | 0x7ff00000u : h;  // infinite, NaN
  return __hiloint2double((int)(h | (b & 0x80000000u)), tiny ? 0 : (int)(a << 29));
}
