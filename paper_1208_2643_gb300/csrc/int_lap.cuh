// sum_nb f - 4 f(c) of binary64 values on the integer pipes.
//
// GB300 issues a warp-wide FP64 instruction every 80 cycles per sub-partition and an integer
// one every two, so four additions and a multiply-add (400 cycles) cost more than the five
// values' significands shifted to the largest exponent among them, summed as 64-bit integers
// and converted back (about 90 integer instructions, 180 cycles).  The largest significand's
// leading bit sits at bit 59, so a value keeps all its bits down to 2^-6 of the largest and the
// sum's error before its one rounding is below 5 x 2^-59 of the largest value, where the FP64
// form rounds four partial sums of up to 2^-53 each: the result is the more exact one.
// Negative values enter as their bitwise complements, one unit (2^-59) off.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace mpfc {

__device__ __forceinline__ unsigned long long shr64(unsigned long long v, unsigned s) {   // 0 from 64 on
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
  return r;
}
__device__ __forceinline__ unsigned f64_exp(double x) { return ((unsigned)__double2hiint(x) >> 20) & 0x7FFu; }

// The significand with its leading bit at 59 - (emax - exponent), signed.
__device__ __forceinline__ long long f64_fixed(double x, unsigned e, unsigned emax) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned long long m = (b << 11) | 0x8000000000000000ull;
  const long long s = (long long)((int)(b >> 32) >> 31);
  return (long long)shr64(m, emax - e + 4u) ^ s;
}

// a 2^(emax - 1023 - 59), rounded to nearest (ties up in magnitude).
__device__ __forceinline__ double fixed_f64(long long a, unsigned emax) {
  const long long s = a >> 63;
  const unsigned long long u = (unsigned long long)((a ^ s) - s);
  if (u == 0ull) return 0.0;
  const int z = __clzll((long long)u);
  // significand with its leading bit at 63, rounded to 53 bits; the leading bit adds one to
  // the exponent field, as does a carry out of the rounding
  const unsigned long long n = u << z;
  const unsigned long long m = (n >> 11) + ((n >> 10) & 1ull);
  const unsigned long long e = (unsigned long long)(emax + 3u - (unsigned)z);
  return __longlong_as_double((long long)((m + (e << 52)) | ((unsigned long long)s & 0x8000000000000000ull)));
}

// The FP64 form, out of line: inlined, its four instructions are issued predicated off on every
// cell, which holds the FP64 pipe all the same (12 of 20 instructions of a residual).
static __noinline__ __device__ double lap5_f64_general(double w, double e, double s, double n, double c) {
  return fma(-4.0, c, (w + e) + (s + n));
}

__device__ __forceinline__ double lap5_f64(double w, double e, double s, double n, double c) {
  const unsigned ew = f64_exp(w), ee = f64_exp(e), es = f64_exp(s), en = f64_exp(n), ec = f64_exp(c);
  const unsigned emax = max(max(max(ew, ee), max(es, en)), ec);
  // infinities and NaN, overflow, and magnitudes below 2^-900 (zeros, subnormals): the FP64 form
  if (emax - 123u >= 2046u - 4u - 123u) return lap5_f64_general(w, e, s, n, c);
  const long long a = (f64_fixed(w, ew, emax) + f64_fixed(e, ee, emax)) + (f64_fixed(s, es, emax) + f64_fixed(n, en, emax));
  return fixed_f64(a - 4 * f64_fixed(c, ec, emax), emax);
}

}  // namespace mpfc
