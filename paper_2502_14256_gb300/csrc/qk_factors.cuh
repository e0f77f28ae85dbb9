// One-dimensional kernel factors K_alpha of 32-bit words (SI here; DSI as coefficient rows in
// qk_column.cuh) and the product-minus-one recurrence for the first column.
//
// DSI (arXiv 2502.14256, Sec. 5.3, Theorem; x = Z 2^-32, beta(x) = -floor(log2 x),
// t_nu = 2^(-nu beta), beta(0) = t_nu(0) = 0):
//   K_1 = 1 - 3 t_1 (Z != 0), K_1(0) = 1    (first-order Walsh kernel; the paper
//                                            defers order 1 to Dick & Pillichshammer)
//   K_2 = -1 - beta x + 5/2 (1 - t_1)
//   K_3 = -1 + beta x^2 - 5 (1 - t_1) x + 43/18 (1 - t_2)
//   K_4 = -1 - 2/3 beta x^3 + 5 (1 - t_1) x^2 - 43/9 (1 - t_2) x + 701/294 (1 - t_3)
//         + beta (S/48 - 1/42),  S = sum_a wal_{2^a}(x) 8^-a.
// With 32 digits S = 8/7 - 2 S', S' = sum over set digits x_{a+1} of 8^-a, so the
// last term equals -beta S'/24 (no cancellation between S/48 and 1/42).  S' is
// read off the word by spreading its leading bits three apart (octal digits).
//
// SI (Sec. 5.2): K_alpha(x) = (2 pi)^(2 alpha) / ((-1)^(alpha+1) (2 alpha)!) B_2alpha(x):
//   K_1 = pi^2/3 - 2 pi^2 x (1 - x),   K_2 = pi^4/45 - 2 pi^4/3 (x (1 - x))^2.
#pragma once

#include "qk_common.cuh"

namespace qk {

// Exact small integer -> float by the mantissa trick (one add, no conversion unit).
__device__ __forceinline__ float small_int_to(float, uint32_t v) {
  return __int_as_float(0x4B000000 | (int)v) - 8388608.0f;  // v < 2^23
}

// v 2^-t as a double (RN) by integer operations: an FP64 add or conversion takes the issue time of
// 32 integer adds (qk_wht96.cuh) (t: binary places, |t| small).
__device__ __forceinline__ double u64_to_double(uint64_t v, int t) {
  const int c = __clzll((long long)v);
  const uint64_t x = v << (c & 63);                      // leading one at bit 63
  const uint32_t rem = (uint32_t)x & 0x7FFu;
  uint64_t mant = x >> 11;                               // 53 bits, the leading one at bit 52
  mant += (rem > 0x400u) | ((rem == 0x400u) & ((uint32_t)mant & 1u));
  const uint64_t bits = ((uint64_t)(uint32_t)(1085 - c - t) << 52) + mant;
  return __longlong_as_double(v ? (long long)bits : 0ll);
}
__device__ __forceinline__ double u32_to_double(uint32_t v, int t) {  // exact
  const int c = __clz(v);
  const uint32_t x = v << (c & 31);
  const uint32_t hi = ((uint32_t)(1053 - c - t) << 20) + (x >> 11);
  return __hiloint2double(v ? (int)hi : 0, (int)(x << 21));
}

// S' = sum_{a >= 0, bit (31-a) of Z set} 8^-a to FP32's precision: a = 0..9.
__device__ __forceinline__ float octal_tail(uint32_t Z) { return __uint2float_rn(spread3_10(Z >> 22)) * 0x1p-27f; }

template <typename T, int ALPHA>
__device__ __forceinline__ T si_factor(uint32_t W) {
  // x (1 - x) = W (2^32 - W) 2^-64: in FP64 the exact 64-bit product rounded once, without
  // FP64 instructions (the bits of fma(-x, x, x))
  T q;
  if constexpr (sizeof(T) == 8) {
    q = u64_to_double((uint64_t)W * (uint32_t)(0u - W), 64);
  } else {
    const T x = word_to_unit(W);
    q = x * (T(1) - x);
  }
  if constexpr (ALPHA == 1) {
    return T(3.2898681336964528729) - T(19.739208802178717238) * q;  // pi^2/3, 2 pi^2
  } else {
    static_assert(ALPHA == 2, "SI smoothness 1..2");
    return T(2.1646464674222763831) - T(64.939394022668291491) * (q * q);  // pi^4/45, 2pi^4/3
  }
}

// Fused multiply-add in the precision of the arguments (never promoted).
__device__ __forceinline__ float fmadd(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fmadd(double a, double b, double c) { return fma(a, b, c); }

// p <- (1 + p)(1 + a) - 1, keeping p = prod(1 + a_j) - 1 with relative precision.
template <typename T>
__device__ __forceinline__ T pm1_step(T p, T a) { return fmadd(p, a, p + a); }

}  // namespace qk
