// Device arithmetic shared by the FP64 and float-float kernels: FP64 <-> FP32
// conversions on the integer pipes and float-float numbers.
#pragma once
#include <cuda_runtime.h>

namespace qed {
namespace {

// FP64 -> FP32 with round-to-nearest-even, done on the integer pipes from the
// IEEE-754 formats (sign, rebiased exponent, top 23 of the 52 fraction bits,
// rounding on the 29 dropped bits; a carry out of the fraction bumps the
// exponent, up to infinity).  Magnitudes below the FP32 normal range become
// signed zero, NaN stays NaN.  GB300 runs FP64 instructions, conversions
// included, at a small fraction of its FP32 rate, so the FP32 grouped GEMM
// converts its FP64 operands this way.
__device__ __forceinline__ float d2f_bits(double d) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(d);
  const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
  const int e = (int)((b >> 52) & 0x7ff);
  const unsigned long long frac = b & 0xFFFFFFFFFFFFFull;
  if (e == 0x7ff) return __uint_as_float(sign | 0x7f800000u | (frac ? 0x400000u : 0u));
  const int fe = e - 1023 + 127;
  if (fe <= 0) return __uint_as_float(sign);
  if (fe >= 255) return __uint_as_float(sign | 0x7f800000u);
  unsigned r = sign | ((unsigned)fe << 23) | (unsigned)(frac >> 29);
  const unsigned rem = (unsigned)(frac & 0x1FFFFFFFull);
  if (rem > 0x10000000u || (rem == 0x10000000u && (r & 1u))) r += 1u;
  return __uint_as_float(r);
}

static __device__ __noinline__ float d2f_edge(double d) { return d2f_bits(d); }

// FP32 -> FP64, exact, on the integer pipes (FP32 subnormals become zero).
__device__ __forceinline__ double f2d_bits(float f) {
  const unsigned u = __float_as_uint(f);
  const unsigned long long sign = (unsigned long long)(u & 0x80000000u) << 32;
  const int e = (int)((u >> 23) & 0xff);
  const unsigned long long frac = u & 0x7FFFFFu;
  if (e == 0) return __longlong_as_double((long long)sign);
  if (e == 0xff) return __longlong_as_double((long long)(sign | 0x7FF0000000000000ull | (frac << 29)));
  return __longlong_as_double((long long)(sign | ((unsigned long long)(e - 127 + 1023) << 52) | (frac << 29)));
}

// FP64 -> FP32 as the cast does it, FP32 subnormals and signed zeros kept, on
// the integer pipes in the normal range: the exponent rebiased, the top 23
// fraction bits, a carry from the other 29.
static __device__ __noinline__ float d2f_cast(double d) { return (float)d; }
__device__ __forceinline__ float d2f_rn(double d) {
  const unsigned h = (unsigned)__double2hiint(d), l = (unsigned)__double2loint(d);
  if ((h & 0x7fffffffu) - (897u << 20) >= (253u << 20))   // outside 2^-126 .. 2^127
    return ((h << 1) | l) == 0u ? __uint_as_float(h) : d2f_cast(d);
  const unsigned t = (__funnelshift_l(l, h, 3) - (384u << 23)) & 0x7fffffffu;
  return __uint_as_float((t + (((l & 0x1fffffffu) + 0x0fffffffu + (t & 1u)) >> 29)) | (h & 0x80000000u));
}

// FP32 -> FP64, exact, subnormals too (brought into the normal range first).
__device__ __forceinline__ double f2d_exact(float f) {
  const bool small = fabsf(f) < 0x1p-126f;
  const double d = f2d_bits(small ? f * 0x1p24f : f);
  return __hiloint2double(__double2hiint(d) - (small && f != 0.f ? 24 << 20 : 0), __double2loint(d));
}

// ---- float-float arithmetic: a value hi + lo held in two FP32 numbers
// (about 48 significant bits), with products and sums made error-free by
// FMA (Dekker's TwoProduct) and Knuth's TwoSum.  GB300 runs FP32 at many
// times its FP64 rate, so a float-float multiply-add (about a dozen FP32
// instructions) outruns one FP64 FMA while keeping FP64-level accuracy for
// these contractions.
struct ff {
  float hi, lo;
  __device__ __forceinline__ ff() {}
  __device__ __forceinline__ explicit ff(float h) : hi(h), lo(0.f) {}
  __device__ __forceinline__ ff(float h, float l) : hi(h), lo(l) {}
};

__device__ __forceinline__ ff ff_norm(float s, float e) {
  const float h = s + e;
  return ff(h, e - (h - s));
}

__device__ __forceinline__ ff operator*(ff a, ff b) {
  const float p = a.hi * b.hi;
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, e);
  e = fmaf(a.lo, b.hi, e);
  return ff_norm(p, e);
}

__device__ __forceinline__ ff operator+(ff a, ff b) {
  const float s = a.hi + b.hi;
  const float bb = s - a.hi;
  const float err = (a.hi - (s - bb)) + (b.hi - bb) + a.lo + b.lo;
  return ff_norm(s, err);
}

__device__ __forceinline__ ff& operator*=(ff& a, ff b) { a = a * b; return a; }
__device__ __forceinline__ ff& operator+=(ff& a, ff b) { a = a + b; return a; }

// c + a b with the product's error and the sum's error kept in lo
__device__ __forceinline__ ff kc_fma(ff a, ff b, ff c) {
  const float p = a.hi * b.hi;
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, e);
  e = fmaf(a.lo, b.hi, e);
  const float s = c.hi + p;
  const float bb = s - c.hi;
  const float err = (c.hi - (s - bb)) + (p - bb);
  return ff(s, c.lo + e + err);
}

__device__ __forceinline__ double kc_fma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float kc_fma(float a, float b, float c) { return fmaf(a, b, c); }

// FP64 -> float-float on the integer pipes: hi = the double cut to 24
// significant bits, lo = the remaining 29 fraction bits (rounded to 24)
__device__ __forceinline__ ff d2ff(double d);

template <typename T>
__device__ __forceinline__ T to_t(double v);
template <>
__device__ __forceinline__ double to_t<double>(double v) { return v; }
template <>
__device__ __forceinline__ float to_t<float>(double v) { return d2f_bits(v); }

// hi rounded to nearest: the lo lo product that a multiply-add drops is then
// a quarter of what two truncated parts leave, and of either sign.
template <>
__device__ __forceinline__ ff to_t<ff>(double v) {
  const ff t = d2ff(v);
  return ff_norm(t.hi, t.lo);
}

// Operands as they come, hi cut and not rounded: coefficients, and vectors whose
// sums round above what to_t would save.
template <typename T>
__device__ __forceinline__ T raw_t(double v) { return to_t<T>(v); }
template <>
__device__ __forceinline__ ff raw_t<ff>(double v) { return d2ff(v); }

// Values outside the range of the short form below: zeros, magnitudes below
// 2^-103 (whose lo part nears the FP32 subnormals) or past the FP32 range,
// infinities and NaN.
static __device__ __noinline__ ff d2ff_edge(double d) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(d);
  const float hi = d2f_bits(__longlong_as_double((long long)(b & ~((1ull << 29) - 1ull))));
  const int e = (int)((b >> 52) & 0x7ff);
  const unsigned low = (unsigned)(b & ((1ull << 29) - 1ull));
  if (e == 0x7ff && low) return ff(__uint_as_float(0x7fc00000u), 0.f);
  float lo = 0.f;
  if (e != 0 && e != 0x7ff && low) {
    // low x 2^(e - 1075): convert the integer, then move its exponent
    const float f = (float)low;
    const int ex = (int)((__float_as_uint(f) >> 23) & 0xff) + (e - 1075);
    if (ex > 0) lo = __uint_as_float((__float_as_uint(f) & 0x807fffffu) | ((unsigned)ex << 23));
    if (b >> 63) lo = -lo;
  }
  return ff(hi, lo);
}

// hi: the sign, the exponent rebiased by 896 and the top 23 fraction bits; lo:
// the other 29 bits as an integer, rounded to 24, times 2^-29 of hi's last
// place (a power of two taken from hi's own exponent field).
__device__ __forceinline__ ff d2ff(double d) {
  const unsigned h = (unsigned)__double2hiint(d), l = (unsigned)__double2loint(d);
  const unsigned top = h & 0x7fffffffu;
  if (top - (920u << 20) >= (230u << 20)) return top == 0u && l == 0u ? ff(0.f) : d2ff_edge(d);   // 920 <= e < 1150
  const unsigned hb = ((__funnelshift_l(l, h, 3) - (384u << 23)) & 0x7fffffffu) | (h & 0x80000000u);
  const float ulp = __uint_as_float((hb & 0xff800000u) - (23u << 23));
  return ff(__uint_as_float(hb), ((float)(l & 0x1fffffffu) * 0x1p-29f) * ulp);
}

template <typename T>
__device__ __forceinline__ double to_d(T v);
template <>
__device__ __forceinline__ double to_d<double>(double v) { return v; }
template <>
__device__ __forceinline__ double to_d<float>(float v) { return f2d_bits(v); }
template <>
__device__ __forceinline__ double to_d<ff>(ff v) { return f2d_bits(v.hi) + f2d_bits(v.lo); }

}  // namespace
}  // namespace qed
