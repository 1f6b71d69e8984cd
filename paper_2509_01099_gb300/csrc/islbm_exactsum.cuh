// FP64 results of sums of FP32 values, formed on the integer units.
//
// The FP64 units of this GPU retire 2 operations per clock and SM (an FP32 or
// integer operation: 64 to 128), so a kernel that converts its FP32 inputs to
// FP64 and adds them there is bound by that pipe: the field output of the 1024^2
// FP32 cavity took 115 us at 83% FP64 pipe activity, against 14 us for its
// bytes.  Here the values of one group are aligned to the group's largest
// exponent as 64-bit integers, added as integers, and the sum is rounded once
// to FP64.  An aligned value drops bits below 2^-58 of the largest one, so a
// sum of up to 32 values is at least as close to the true sum as the chain of
// FP64 additions (each rounding at 2^-53 of its partial sum).
#pragma once

#include <cuda_runtime.h>

namespace islbm {

// Largest biased exponent of the group (at least 1, the exponent of subnormal
// values); 255 means that the group holds an infinity or a NaN.
template <int N>
__device__ __forceinline__ int group_exponent(const float (&f)[N]) {
  unsigned m = 1u << 23;
#pragma unroll
  for (int i = 0; i < N; ++i) m = max(m, __float_as_uint(f[i]) & 0x7FFFFFFFu);
  return (int)(m >> 23);
}

// f in units of 2^(E - 184): at most 58 bits for the group's largest exponent E.
__device__ __forceinline__ long long aligned(float f, int E) {
  const unsigned b = __float_as_uint(f);
  const int e = (int)((b >> 23) & 0xFFu);
  const int s = (int)b >> 31;
  int m = (int)((b & 0x7FFFFFu) | (min(e, 1) << 23));
  m = (m ^ s) - s;
  return ((long long)(m << 2) << 32) >> min(E - max(e, 1), 63);
}

// v units of 2^(E - 184), |v| < 2^63, rounded to the nearest FP64 (ties to even).
__device__ __forceinline__ double aligned_to_double(long long v, int E) {
  const long long s = v >> 63;
  const unsigned long long u = (unsigned long long)((v ^ s) - s);
  const int lz = __clzll((long long)u);
  unsigned long long t = u << (lz - 1);      // leading bit at 62 (lz >= 1; u = 0 below)
  t += 0x1FFull + ((t >> 10) & 1ull);
  // biased exponent 63 - lz + E + 839; the mantissa's leading bit adds one
  const unsigned long long r =
      ((unsigned long long)(unsigned)(63 - lz + E + 838) << 52) + (t >> 10);
  return u == 0 ? 0.0
                : __longlong_as_double((long long)(r | ((unsigned long long)s << 63)));
}

// FP32 value of a positive normal FP64 value inside FP32's range, truncated.
__device__ __forceinline__ float trunc_to_float(double d) {
  const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
  return __uint_as_float(((hi - (896u << 20)) << 3) | (lo >> 29));
}

// FP64 value of a positive normal FP32 value.
__device__ __forceinline__ double widen(float f) {
  const unsigned b = __float_as_uint(f);
  return __hiloint2double((int)((b >> 3) + (896u << 20)), (int)(b << 29));
}

// FP64 value of an FP32 value that is normal or zero.
__device__ __forceinline__ double widen_signed(float f) {
  const unsigned b = __float_as_uint(f);
  const unsigned hi = (b & 0x80000000u) | (((b & 0x7FFFFFFFu) >> 3) + (896u << 20));
  return f == 0.f ? 0.0 : __hiloint2double((int)hi, (int)(b << 29));
}

// Whether |d| < 1/2 (not so for a NaN).
__device__ __forceinline__ bool below_half(double d) {
  return ((unsigned)__double2hiint(d) & 0x7FFFFFFFu) < 0x3FE00000u;
}

// FP32 value of |d| < 2, truncated; 0 below 2^-30.
__device__ __forceinline__ float trunc_small(double d) {
  const unsigned hi = (unsigned)__double2hiint(d), m = hi & 0x7FFFFFFFu;
  const unsigned b = ((m - (896u << 20)) << 3) | ((unsigned)__double2loint(d) >> 29);
  return m < ((1023u - 30u) << 20) ? 0.f : __uint_as_float(b | (hi & 0x80000000u));
}

// 1 / (1 + d) = hi + lo for |d| < 1/2: hi the FP32 reciprocal (relative error below
// 2^-21; 1 - hi is exact), x = 1 - (1 + d) hi, lo = hi (x + x^2 + ...).  Divided by
// 1 + d, j is quotient(j): one rounding, and 2^-74 |j| from the small terms.  RMS
// error of a component over |d| < 1/200 in units of 2^-53: 0.43, as a division
// where 1 + d is exact (0.63 where it is rounded; the product with a rounded
// reciprocal 0.78).  3 FP64 operations, and 2 for a quotient.
struct Reciprocal {
  double hi, lo;
  __device__ __forceinline__ explicit Reciprocal(double d) {
    const float rf = __fdividef(1.0f, 1.0f + trunc_small(d));
    hi = widen(rf);
    const double x = fma(-d, hi, widen_signed(1.0f - rf));
    lo = hi * fma(x, x, x);
  }
  // j / (1 + d), and with c (small beside it) added before it is rounded
  __device__ __forceinline__ double quotient(double j) const { return fma(j, hi, j * lo); }
  __device__ __forceinline__ double quotient(double j, double c) const {
    return fma(j, hi, fma(j, lo, c));
  }
};

// sqrt(a) for a = 0 and 2^-100 .. 2^100, elsewhere the library's.  g = a y with
// the FP32 reciprocal root y (relative error e below 2^-20) and two Newton steps
// on the residual a - g^2, whose errors are 3/2 e^2 and below 2^-60: the result
// is the correctly rounded one but for some 10^-6 of the arguments.  5 FP64
// operations.
__device__ __forceinline__ double quick_sqrt(double a) {
  const unsigned e = ((unsigned)__double2hiint(a) >> 20);
  if (e - (1023u - 100u) > 200u) return sqrt(a);
  const float yf = rsqrtf(trunc_to_float(a));
  const double y = widen(yf), h = widen(0.5f * yf);
  const double g = a * y;
  const double s = fma(fma(-g, g, a), h, g);
  return fma(fma(-s, s, a), h, s);
}

}  // namespace islbm
