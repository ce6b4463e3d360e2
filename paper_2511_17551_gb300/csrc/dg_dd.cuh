// Double-FP32 arithmetic: a number is the unevaluated sum h + l of two FP32 values,
// |l| <= ulp(h) / 2, about 48 significant bits.  The FP64 pipe of this GPU does about one
// sixtieth of the FP32 pipe's operations (1.26 against 76.5 TFLOP/s measured with FMA
// chains), so an operation in this form, 6 to 20 FP32 instructions, costs a fraction of the
// FP64 one it stands for.  The error-free transformations are Knuth's and Dekker's (T. J.
// Dekker, "A floating-point technique for extending the available precision", 1971), with
// the fused multiply-add for the product's error.  Every operation goes through the rounding
// intrinsics, so that the compiler neither contracts nor reorders them and a function gives
// the same bits in every kernel it is inlined into.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>
#include "dg_cvt.cuh"

namespace dgdd {

struct dd {
  float h, l;
};

#ifdef __CUDACC__
#define DG_HD __host__ __device__ __forceinline__
#else
#define DG_HD inline
#endif

DG_HD float fadd(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fadd_rn(a, b);
#else
  return a + b;
#endif
}
DG_HD float fsub(float a, float b) { return fadd(a, -b); }
DG_HD float fmul(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  return a * b;
#endif
}
DG_HD float ffma(float a, float b, float c) {
#ifdef __CUDA_ARCH__
  return __fmaf_rn(a, b, c);
#else
  return fmaf(a, b, c);
#endif
}
// 1 / x to within an ulp or so; every use corrects it by its residual
DG_HD float frcp(float x) {
#ifdef __CUDA_ARCH__
  return __frcp_rn(x);
#else
  return 1.0f / x;
#endif
}

DG_HD dd make(float h, float l) {
  dd r;
  r.h = h;
  r.l = l;
  return r;
}
// conversions between the two (dg_cvt.cuh: integer work on the device)
DG_HD float narrow(double x) {
#ifdef __CUDA_ARCH__
  return f64_to_f32_mid(x);
#else
  return (float)x;
#endif
}
DG_HD double widen(float x) {
#ifdef __CUDA_ARCH__
  return f32_to_f64_mid(x);
#else
  return (double)x;
#endif
}
// the FP64 number as a pair
DG_HD dd from_double(double x) {
  const float h = narrow(x);
  return make(h, narrow(x - widen(h)));
}
DG_HD double to_double(dd a) { return widen(a.h) + widen(a.l); }
DG_HD dd neg(dd a) { return make(-a.h, -a.l); }

DG_HD dd two_sum(float a, float b) {
  const float s = fadd(a, b), t = fsub(s, a);
  return make(s, fadd(fsub(a, fsub(s, t)), fsub(b, t)));
}
DG_HD dd quick_two_sum(float a, float b) {  // |a| >= |b|
  const float s = fadd(a, b);
  return make(s, fsub(b, fsub(s, a)));
}
DG_HD dd two_prod(float a, float b) {
  const float p = fmul(a, b);
  return make(p, ffma(a, b, -p));
}
// error at most a few 2^-48 (|a| + |b|)
DG_HD dd add(dd a, dd b) {
  const dd s = two_sum(a.h, b.h);
  return quick_two_sum(s.h, fadd(s.l, fadd(a.l, b.l)));
}
DG_HD dd add(dd a, float b) {
  const dd s = two_sum(a.h, b);
  return quick_two_sum(s.h, fadd(s.l, a.l));
}
DG_HD dd mul(dd a, dd b) {
  const float p = fmul(a.h, b.h);
  return quick_two_sum(p, ffma(a.l, b.h, ffma(a.h, b.l, ffma(a.h, b.h, -p))));
}
DG_HD dd mul(dd a, float b) {
  const float p = fmul(a.h, b);
  return quick_two_sum(p, ffma(a.l, b, ffma(a.h, b, -p)));
}
// running sums: the head by an exact sum, the tail collected; norm() once at the end
DG_HD void acc(dd& s, dd x) {
  const dd t = two_sum(s.h, x.h);
  s.h = t.h;
  s.l = fadd(s.l, fadd(t.l, x.l));
}
// s += a b
DG_HD void acc_mul(dd& s, dd a, dd b) {
  const float p = fmul(a.h, b.h);
  acc(s, make(p, ffma(a.l, b.h, ffma(a.h, b.l, ffma(a.h, b.h, -p)))));
}
// s += a b for a small integer (or any FP32 value) b
DG_HD void acc_mul(dd& s, dd a, float b) {
  const float p = fmul(a.h, b);
  acc(s, make(p, ffma(a.l, b, ffma(a.h, b, -p))));
}
DG_HD dd norm(dd a) { return quick_two_sum(a.h, a.l); }
// a b + c (Horner step)
DG_HD dd mul_add(dd a, dd b, dd c) {
  const float p = fmul(a.h, b.h);
  const float e = ffma(a.l, b.h, ffma(a.h, b.l, ffma(a.h, b.h, -p)));
  const dd s = two_sum(p, c.h);
  return quick_two_sum(s.h, fadd(s.l, fadd(e, c.l)));
}
DG_HD dd rcp(dd a) {
  const float q = frcp(a.h);
  const float r = ffma(-q, a.l, ffma(-q, a.h, 1.0f));
  return quick_two_sum(q, fmul(q, r));
}
// a / b
DG_HD dd div(dd a, dd b) {
  const float i = frcp(b.h), q = fmul(a.h, i);
  const float r = fadd(ffma(-q, b.h, a.h), ffma(-q, b.l, a.l));
  return quick_two_sum(q, fmul(r, i));
}
DG_HD float bits(uint32_t u) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(u);
#else
  float f;
  memcpy(&f, &u, 4);
  return f;
#endif
}

// exp(t) 2^shift; t = h + l, the result flushed to zero below 2^-100 and made infinite above
// 2^126.  t = k ln2 / 128 + r with |r| <= 0.0028, ln2 / 128 in parts of 20, 9 and 24 bits (t - k L1 has
// at most 23 significant bits, so the FMA is exact; k L2 is exact for |t| up to 177, beyond
// which the result is out of range); exp(r) by its Taylor series, where r and r^2 / 2 are carried as pairs
// and the rest, below 4e-9, in FP32; 2^(j/128) from the table tab of EXP_TAB pairs.  A table
// of 32 entries (|r| <= 0.0109) costs an FMA more and leaves the rest at 3e-7, whose FP32
// rounding is then the largest error.
constexpr int EXP_TAB = 128;
DG_HD dd exp_scaled(dd t, int shift, const dd* tab) {
  const float kf = rintf(fmul(t.h, 184.6649627685547f));  // 128 / ln 2
  const int k = (int)kf;
  const float a = ffma(-kf, 0x1.62e42p-8f, t.h);  // exact
  const dd d = two_sum(a, fmul(-kf, 0x1.fdp-29f));
  const dd r = quick_two_sum(d.h, fadd(d.l, ffma(-kf, 0x1.e8e7bcp-38f, t.l)));
  const float p = fmul(r.h, r.h);
  const float e = ffma(r.h, r.h, -p);
  const float q = fmul(fmul(p, r.h), ffma(r.h, 1.0f / 24.0f, 1.0f / 6.0f));
  const dd s = quick_two_sum(r.h, fmul(0.5f, p));
  const float low = fadd(fadd(s.l, ffma(0.5f, e, ffma(r.h, r.l, r.l))), q);
  const dd T = tab[k & (EXP_TAB - 1)];
  const float m = fmul(T.h, s.h), me = ffma(T.h, s.h, -m);
  const dd z = quick_two_sum(T.h, m);
  const float lo = fadd(z.l, fadd(me, ffma(T.h, low, ffma(T.l, s.h, T.l))));
  const int ex = (k >> 7) + shift;
  const float sc = ex < -100 ? 0.0f : (ex > 126 ? bits(0x7f800000u) : bits((uint32_t)(ex + 127) << 23));
  return make(fmul(z.h, sc), ex > 126 ? 0.0f : fmul(lo, sc));
}

// exp(x) - 1 for |x| <= 1/16: x + x^2 (1/2 + x (1/6 + x r)), the Taylor series with r to x^4 in
// FP32; relative error below 2^-39
DG_HD dd expm1_small(dd x) {
  const float r = ffma(x.h, ffma(x.h, ffma(x.h, ffma(x.h, 1.0f / 40320.0f, 1.0f / 5040.0f), 1.0f / 720.0f), 1.0f / 120.0f),
                       1.0f / 24.0f);
  const float s6 = 1.0f / 6.0f;
  const dd s = add(make(s6, (float)(1.0 / 6.0 - (double)s6)), fmul(x.h, r));
  const dd q = add(mul(x, s), 0.5f);
  return add(mul(mul(x, x), q), x);
}

// ln(x) of a pair, x.h a normal positive number: y0 = logf, then ln x = y0 + ln(x exp(-y0)) with
// x exp(-y0) = 1 + z, |z| below 2^-16: z - z^2 / 2.  `sum64`, if given, gets it as an FP64 number (absolute
// error below 2^-45, where the pair itself is good to 2^-48 |ln x|) at the cost of three conversions
// and two additions in FP64.
DG_HD dd log_(dd x, const dd* tab, double* sum64 = nullptr) {
  const float y0 = logf(x.h);
  const dd E = exp_scaled(make(-y0, 0.0f), 0, tab);
  const float p = fmul(x.h, E.h);
  const float pe = ffma(x.l, E.h, ffma(x.h, E.l, ffma(x.h, E.h, -p)));
  const float z = fsub(p, 1.0f), t = ffma(fmul(-0.5f, z), z, pe);
  if (sum64) *sum64 = widen(y0) + (widen(z) + widen(t));
  const dd s = two_sum(y0, z);
  return quick_two_sum(s.h, fadd(s.l, t));
}

}  // namespace dgdd
