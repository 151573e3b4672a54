// Float-float arithmetic: a value is an unevaluated sum h + l of two binary32 numbers,
// |l| at most a few ulps of h, so about 48 significant bits.  Sums use Knuth's TwoSum and
// Dekker's FastTwoSum, products the FMA error term (T. J. Dekker, Numer. Math. 18, 1971;
// Y. Hida, X. S. Li, D. H. Bailey, ARITH-15, 2001).  On GB300 a warp-wide FP64 instruction
// holds its sub-partition's FP64 pipe for about 80 cycles and an FP32 one for one, so a
// float-float addition (8 to 11 FP32 instructions) costs an eighth of an FP64 one.
//
// Every operation is written with the rounding intrinsics, so the compiler contracts and
// reorders nothing and a cell function gives the same bits in every kernel that inlines it.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "int_lap.cuh"
#include "mpfc_common.cuh"

namespace mpfc {

struct df {
  float h, l;
};

__device__ __forceinline__ float fadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ df mk(float2 v) { return df{v.x, v.y}; }
__device__ __forceinline__ float2 f2(df v) { return make_float2(v.h, v.l); }

// s + e = a + b exactly
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = fadd(a, b);
  const float bb = fadd(s, -a);
  e = fadd(fadd(a, -fadd(s, -bb)), fadd(b, -bb));
}
// the same for |a| >= |b|
__device__ __forceinline__ df norm(float a, float b) {
  const float s = fadd(a, b);
  return df{s, fadd(b, -fadd(s, -a))};
}
__device__ __forceinline__ df norm(df a) { return norm(a.h, a.l); }
__device__ __forceinline__ df neg(df a) { return df{-a.h, -a.l}; }
// Sum without the final normalisation: error at most about 2^-47 of |a| + |b|.
__device__ __forceinline__ df addu(df a, df b) {
  float s, e;
  two_sum(a.h, b.h, s, e);
  return df{s, fadd(e, fadd(a.l, b.l))};
}
__device__ __forceinline__ df add(df a, df b) { return norm(addu(a, b)); }
// Sums of three and four terms, normalised once.
__device__ __forceinline__ df sum3u(df a, df b, df c) {
  float s, e, t, f;
  two_sum(a.h, b.h, s, e);
  two_sum(s, c.h, t, f);
  return df{t, fadd(fadd(e, f), fadd(fadd(a.l, b.l), c.l))};
}
__device__ __forceinline__ df sum4u(df a, df b, df c, df d) {
  float s, e, t, f, u, g;
  two_sum(a.h, b.h, s, e);
  two_sum(c.h, d.h, t, f);
  two_sum(s, t, u, g);
  return df{u, fadd(fadd(fadd(e, f), g), fadd(fadd(a.l, b.l), fadd(c.l, d.l)))};
}
// Product, unnormalised: the error term drops a.l b.l (2^-46 relative).
__device__ __forceinline__ df mulu(df a, df b) {
  const float p = fmul(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, e);
  e = __fmaf_rn(a.l, b.h, e);
  return df{p, e};
}
__device__ __forceinline__ df mul(df a, df b) { return norm(mulu(a, b)); }
__device__ __forceinline__ df sqr(df a) {
  const float p = fmul(a.h, a.h);
  const float e = __fmaf_rn(fadd(a.h, a.h), a.l, __fmaf_rn(a.h, a.h, -p));
  return norm(p, e);
}
// Exact scaling by a power of two.
__device__ __forceinline__ df scale2(df a, float p2) { return df{fmul(a.h, p2), fmul(a.l, p2)}; }
// Reciprocal: the hardware approximation r (relative error e of a few 2^-24), then
// r (1 + (1 - x r)), whose relative error is e^2 plus the roundings, below 2^-44.
__device__ __forceinline__ df rcp(df x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x.h));
  const float e = __fmaf_rn(-x.l, r, __fmaf_rn(-x.h, r, 1.0f));
  return norm(r, fmul(r, e));
}
// sum_nb f - 4 f(c), normalised.
__device__ __forceinline__ df lap5(df w, df e, df s, df n, df c) {
  const df q = sum4u(w, e, s, n);
  float t, f;
  two_sum(q.h, fmul(-4.0f, c.h), t, f);
  return norm(t, fadd(f, __fmaf_rn(-4.0f, c.l, q.l)));
}

// binary64 -> float-float: the high part truncated (integer pipes), the 29 significand
// bits below it as the low part (converted to binary32: 24 of them, so 48 bits in all).
// Zero, magnitudes below 2^-74 (whose low part's scale leaves the normal binary32 range) and
// from 2^100 on keep one part only, the value rounded to nearest.
__device__ __forceinline__ df df_of(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned int hi = (unsigned int)(b >> 32), eb = (hi >> 20) & 0x7FFu;
  if (eb - (1023u - 74u) >= 174u) {
    if ((b << 1) == 0ull) return df{0.0f, 0.0f};
    return df{f64_to_f32_rn(x), 0.0f};
  }
  const unsigned int sg = hi & 0x80000000u, ef = (eb - 1023u + 127u) << 23;
  // low 29 bits times 2^(e - 52), with the sign of x
  return df{__uint_as_float(sg | ef | ((unsigned int)(b >> 29) & 0x7FFFFFu)),
            fmul(__uint2float_rn((unsigned int)b & 0x1FFFFFFFu), __uint_as_float(sg | (ef - (52u << 23))))};
}

// float-float -> binary64 (exact where h and l span at most 53 bits).
__device__ __forceinline__ double df_to_f64(df a) { return f32_to_f64(a.h) + f32_to_f64(a.l); }

}  // namespace mpfc
