// Quotients without FP64 divisions (GB300: about 2 FP64 lanes per SM and cycle): reciprocals and
// quotients to about one FP64 rounding from the FP32 reciprocal estimate, and the FP32 scaling by
// an FP64 eigenvalue from float pairs.
#pragma once

#include "qk_common.cuh"

namespace qk {

// Approximate reciprocal (PTX rcp.approx.ftz.f32, max 1 ulp; subnormals flush to 0): 1/0 = inf.
__device__ __forceinline__ float rcp_approx(float a) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}
// a / b in FP64 without the FP64 divide (GB300 has about two FP64 lanes per SM and cycle):
// from the FP32 reciprocal estimate r of b (its leading 24 bits, relative error e below
// 2^-22), q0 = a r, then q0 (1 + e + e^2) with e = 1 - b r rounded once: what is left is e^3,
// below 2^-66, so the result is within 2 ulp of the rounded quotient (checked against the
// divide by qk_ratio_selftest, as ratio_lean).  Four FP64 instructions.  False for b outside
// 2^-100 .. 2^100 in magnitude (zero, subnormal, inf and NaN included).
__device__ __forceinline__ bool ratio_fast(double a, double b, double &q) {
  const uint32_t hi = (uint32_t)__double2hiint(b), lo = (uint32_t)__double2loint(b);
  const uint32_t ex = (hi >> 20) & 0x7FFu;
  if (ex - 923u > 200u) return false;
  const uint32_t fb = (hi & 0x80000000u) | ((ex - 896u) << 23) | ((hi & 0xFFFFFu) << 3) | (lo >> 29);
  const double r = f2d_exact(rcp_approx(__uint_as_float(fb)));
  const double e = fma(-b, r, 1.0);
  const double q0 = a * r;
  q = fma(q0, fma(e, e, e), q0);
  return true;
}
__device__ __forceinline__ double ratio(double a, double b) {
  double q;
  return ratio_fast(a, b, q) ? q : a / b;
}

// a / b with three FP64 instructions: the FP32 estimate of 1 / b for b's leading 24 bits and its
// residual over all of b (about 2^-46 left) become one double r by integer operations, then
// q0 = a r and its residual, as in Markstein's division: the rounded quotient up to 2^-80 before
// the last rounding.  The mantissa of 1 / b lies in (1/2, 1); where the correction could carry
// it over either end (b within 2^-20 of a power of two), or b is outside 2^-100 .. 2^100, false.
__device__ __forceinline__ bool ratio_lean(double a, double b, double &q) {
  const uint32_t hi = (uint32_t)__double2hiint(b), lo = (uint32_t)__double2loint(b);
  const uint32_t ex = (hi >> 20) & 0x7FFu, mt = hi & 0xFFFFFu;
  if (ex - 923u > 200u || mt - 1u > 0xFFFFDu) return false;
  const float bh = __uint_as_float(0x3F800000u | (mt << 3) | (lo >> 29));
  const float bl = __fmul_rn(__uint2float_rn(lo & 0x1FFFFFFFu), 0x1p-52f);
  const float rm = rcp_approx(bh);  // in (1/2, 1)
  const float e = __fmaf_rn(-bl, rm, __fmaf_rn(-bh, rm, 1.f));
  const int32_t dl = __float2int_rn(__fmul_rn(__fmul_rn(e, rm), 0x1p52f));  // units of 2^-52
  const uint32_t u = __float_as_uint(rm);
  const uint32_t rh = ((u >> 3) + (896u << 20) - ((ex - 1023u) << 20)) | (hi & 0x80000000u);
  const double r = __longlong_as_double((long long)((((uint64_t)rh << 32) | (u << 29)) + (uint64_t)((int64_t)dl * 2)));
  const double q0 = a * r;
  q = fma(fma(-b, q0, a), r, q0);
  return true;
}

// The divide, out of line: predicated FP64 instructions take FP64 time.
static __device__ __noinline__ double divide_rare(double a, double b) { return a / b; }

// 1 / b for b in 2^-100 .. 2^100 as ratio_fast(1, b): one rounding, 3 FP64 instructions.
__device__ __forceinline__ double rcp64_mid(uint32_t hi, uint32_t lo, uint32_t ex) {
  const uint32_t fb = (hi & 0x80000000u) | ((ex - 896u) << 23) | ((hi & 0xFFFFFu) << 3) | (lo >> 29);
  const double r = f2d_normal(rcp_approx(__uint_as_float(fb)));
  const double e = fma(-__hiloint2double((int)hi, (int)lo), r, 1.0);
  return fma(r, fma(e, e, e), r);
}
__device__ __forceinline__ double rcp64(double b) {
  const uint32_t hi = (uint32_t)__double2hiint(b), ex = (hi >> 20) & 0x7FFu;
  if (ex - 923u > 200u) return divide_rare(1.0, b);
  return rcp64_mid(hi, (uint32_t)__double2loint(b), ex);
}

// 1 / b correctly rounded: one more Newton step, whose residual is exact and whose last operation
// is one rounding (Markstein 1990: correct unless b's mantissa is all ones).  5 FP64
// instructions.  False for that mantissa and for b outside 2^-100 .. 2^100: take the divide.
__device__ __forceinline__ bool rcp64_rounded(double b, double &r) {
  const uint32_t hi = (uint32_t)__double2hiint(b), lo = (uint32_t)__double2loint(b);
  const uint32_t ex = (hi >> 20) & 0x7FFu;
  if (ex - 923u > 200u || ((hi & 0xFFFFFu) == 0xFFFFFu && lo == 0xFFFFFFFFu)) return false;
  const double r0 = rcp64_mid(hi, lo, ex);
  r = fma(r0, fma(-b, r0, 1.0), r0);
  return true;
}
__device__ __forceinline__ double rcp64_exact(double b) {
  double r;
  return rcp64_rounded(b, r) ? r : divide_rare(1.0, b);
}
// v fac, fac a power of two, by the exponent field: v and the product normal.
__device__ __forceinline__ double times_pow2(double v, double fac) {
  return __hiloint2double(__double2hiint(v) + (__double2hiint(fac) - 0x3FF00000), __double2loint(v));
}
// fac / b, fac a power of two in 2^-64 .. 1, correctly rounded.
__device__ __forceinline__ double pow2_over(double fac, double b) {
  double r;
  return rcp64_rounded(b, r) ? times_pow2(r, fac) : divide_rare(fac, b);
}

// The MLL's step at one frequency, from |Y|^2, 1 / n and lambda: a = |Y|^2 / (n lambda) by the
// rounded reciprocal and one correction (the rounded quotient, as the divide gives it; 2 FP64
// instructions more than a product with the reciprocal, which is off by one more rounding),
// returns g = (a - 1) / (2 lambda).  The divides where lambda has no rounded reciprocal or the
// quotient's residual could underflow or overflow.
__device__ __forceinline__ double mll_step(double y2, double inv_n, double lam, double &a) {
  double r;
  if (((uint32_t)__double2hiint(y2) >> 20) - 400u > 1300u || !rcp64_rounded(lam, r)) {
    a = divide_rare(y2 * inv_n, lam);
    return divide_rare(0.5 * (a - 1.0), lam);
  }
  const double z = times_pow2(y2, inv_n), q = z * r, h = times_pow2(r, 0.5);
  a = fma(fma(-lam, q, z), r, q);
  return fma(a, h, -h);
}

// x / lambda fac (inverse) or x lambda fac, fac a power of two.
__device__ __forceinline__ double scale_lambda(double x, double lam, double fac, bool inverse) {
  return x * (inverse ? pow2_over(fac, lam) : fac * lam);
}
// FP32: the FP64 division (or product) rounded to FP32, bit for bit, without FP64 instructions.
// lambda as a float pair (its leading 24 bits and the rest, by integer operations) gives the
// result p + s to a relative 2^-43; where p + s -+ 2^-42 |p| round to one FP32 number, so does
// everything between them, the FP64 value (off by 2^-52) included.  The others (about one in
// 2^18) take FP64 out of line, and so do x or lambda outside a wide middle range.  The check is 5
// of some 25 FP32 instructions; with the FP64 form out of line the column, solve and product of
// 32 x 2^18 values take 533 -> 520 us.
static __device__ __noinline__ float scale_lambda_fp64(float x, double lam, double fac, bool inverse) {
  return (float)((double)x * (inverse ? fac / lam : fac * lam));
}
__device__ __forceinline__ float scale_lambda(float x, double lam, double fac, bool inverse) {
  const uint32_t hi = (uint32_t)__double2hiint(lam), lo = (uint32_t)__double2loint(lam);
  const uint32_t ex = (hi >> 20) & 0x7FFu, xe = (__float_as_uint(x) >> 23) & 0xFFu;
  const bool mid = ex - 983u <= 80u && !(hi & 0x80000000u);
  if (!mid || xe - 87u > 80u) return mid && x == 0.f ? x : scale_lambda_fp64(x, lam, fac, inverse);
  const float lh = __uint_as_float(((ex - 896u) << 23) | ((hi & 0xFFFFFu) << 3) | (lo >> 29));
  const float ll = __uint2float_rn(lo & 0x1FFFFFFFu) * __uint_as_float((ex - 948u) << 23);
  float a = lh, b = ll;
  if (inverse) {
    a = rcp_approx(lh);
    const float e = __fmaf_rn(-ll, a, __fmaf_rn(-lh, a, 1.f));
    b = __fmul_rn(a, __fmaf_rn(e, e, e));
  }
  const float p = __fmul_rn(x, a), s = __fmaf_rn(x, b, __fmaf_rn(x, a, -p)), del = __fmul_rn(fabsf(p), 0x1p-42f);
  const float v = __fadd_rn(p, __fsub_rn(s, del));
  if (v != __fadd_rn(p, __fadd_rn(s, del))) return scale_lambda_fp64(x, lam, fac, inverse);
  return v * (float)fac;
}

}  // namespace qk
