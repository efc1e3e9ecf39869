// Conversions and a division with the results of the plain ones, bit for bit,
// off the FP64 pipe (one operation per 15 clocks and warp on an SM) or off a
// serial chain.
#pragma once

#include <cuda_bf16.h>

namespace tddft {

// float32 -> float64 in the integer pipe (a conversion would take the FP64
// pipe's time); subnormals, infinities and NaN convert.
__device__ __forceinline__ double to_f64(float x) {
  const unsigned int u = __float_as_uint(x), e = (u >> 23) & 0xFF;
  if (e == 0xFF || (e == 0 && (u << 1) != 0)) return (double)x;
  const unsigned int top = (u & 0x80000000u) | (e == 0 ? 0u : ((u & 0x7FFFFFFFu) >> 3) + 0x38000000u);
  return __hiloint2double((int)top, (int)(u << 29));
}
__device__ __forceinline__ double to_f64(double x) { return x; }

// The split of a float64 value as __double2bfloat16 gives it, hi = bf16(x) and
// lo = bf16(x - hi), to nearest even, in integer arithmetic on the mantissa
// (the conversions and the subtraction would run on the FP64 pipe, one
// operation per 15 clocks and warp on an SM).  Exponents far from 1, zeros,
// infinities and NaN take the conversions.
__device__ __forceinline__ void split_f64(double x, __nv_bfloat16 &hi, __nv_bfloat16 &lo) {
  const long long b = __double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7FF);
  if (e < 1023 - 64 || e > 1023 + 64) {
    hi = __double2bfloat16(x);
    lo = __double2bfloat16(x - (double)__bfloat162float(hi));
    return;
  }
  const unsigned int sign = (unsigned int)((unsigned long long)b >> 63) << 31;
  const long long m = (b & 0xFFFFFFFFFFFFFll) | (1ll << 52);   // |x| = m 2^(e - 1075)
  const long long h = (m + ((1ll << 44) - 1) + ((m >> 45) & 1)) >> 45;   // 128 .. 256
  const long long r = m - (h << 45);                           // |r| <= 2^44
  // float32(h) 2^(e - 1030): h has 8 significant bits
  const unsigned int fh = __float_as_uint((float)(int)h) + ((unsigned int)(e - 1030) << 23);
  hi = __ushort_as_bfloat16((unsigned short)((fh | sign) >> 16));
  const unsigned long long q = (unsigned long long)(r < 0 ? -r : r);
  const int sh = max(0, 63 - __clzll((long long)(q | 1)) - 7);   // bits below the 8 kept
  const unsigned int l = sh == 0 ? (unsigned int)q
                                 : (unsigned int)((q + ((1ull << (sh - 1)) - 1) + ((q >> sh) & 1)) >> sh);
  // float32(l) 2^(sh + e - 1075), zero for r = 0
  const unsigned int fl = __float_as_uint((float)(int)l) + ((unsigned int)(sh + e - 1075) << 23);
  lo = __ushort_as_bfloat16(
      (unsigned short)(l == 0 ? 0u : ((fl | (r < 0 ? sign ^ 0x80000000u : sign)) >> 16)));
}

// n / d, correctly rounded, from inv = 1 / d (itself correctly rounded):
// remainders correct the product n inv twice, first to within one unit in the
// last place, then to the rounded quotient (Markstein, IBM J. Res. Dev. 34,
// 1990); five dependent operations instead of a whole division.  The theorem
// needs its products clear of under- and overflow and a denominator whose
// significand is not all ones; others divide.
__device__ inline double quotient(double n, double d, double inv) {
  const unsigned en = (unsigned)(__double2hiint(n) >> 20) & 0x7FFu,
                 ed = (unsigned)(__double2hiint(d) >> 20) & 0x7FFu;
  const bool plain = en - 400u < 1247u && ed - 400u < 1247u &&
                     (__double_as_longlong(d) & 0xFFFFFFFFFFFFFll) != 0xFFFFFFFFFFFFFll;
  const int gap = (int)en - (int)ed;
  if (!plain || gap > 500 || gap < -500) return n / d;
  double q = n * inv;
  q = fma(fma(-q, d, n), inv, q);
  return fma(fma(-q, d, n), inv, q);
}

}  // namespace tddft
