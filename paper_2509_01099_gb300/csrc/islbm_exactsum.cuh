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

// Whether a is a positive normal value between 2^-60 and 2^60.
__device__ __forceinline__ bool mid_range(double a) {
  return ((unsigned)__double2hiint(a) >> 20) - (1023u - 60u) <= 120u;
}

// 1 / a within one ulp for a value of mid_range: the FP32 reciprocal (relative
// error below 2^-21) and one third-order correction, 3 FP64 operations.
__device__ __forceinline__ double quick_rcp(double a) {
  const double r = widen(__fdividef(1.0f, trunc_to_float(a)));
  const double x = fma(-a, r, 1.0);
  return fma(r, fma(x, x, x), r);
}

// sqrt(a) within one ulp for a = 0 and 2^-100 .. 2^100 (5 FP64 operations);
// elsewhere the library's.
__device__ __forceinline__ double quick_sqrt(double a) {
  const unsigned e = ((unsigned)__double2hiint(a) >> 20);
  if (e - (1023u - 100u) > 200u) return sqrt(a);
  const double y = widen(rsqrtf(trunc_to_float(a)));
  const double g = a * y;                    // sqrt(a) = g (1 - x)^(-1/2),
  const double x = fma(-g, y, 1.0);          // x = 1 - a y^2, below 2^-20
  return fma(g, x * fma(x, 0.375, 0.5), g);
}

}  // namespace islbm
