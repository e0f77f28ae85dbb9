// FP64 Walsh-Hadamard butterflies in 96-bit integers (arXiv 2502.14256, Sec. 5.3).
//
// GB300 has about 2 FP64 lanes per SM and cycle: an FP64 instruction takes the issue time of 32
// integer adds with carry (measured on all SMs: 0.63e12 FP64, 20e12 add-with-carry and 35e12 FP32
// fma instructions per second).  The WHT only adds and subtracts, so a tile is carried as
// integers over the tile's largest exponent E: X = +-mantissa 2^30 >> (E - e), 96-bit two's
// complement.  The top mantissa bit of the largest element sits at bit 82; 12 stages grow it to
// bit 94; elements down to 2^-30 of the largest keep all 53 bits, smaller ones those from 2^-82
// of it up.  A tile of which a value has bits below that takes the FP64 butterflies, so no bit is
// lost: the butterflies are exact (three adds with carry each), and each output is the exact sum
// rounded to a double once, where FP64 butterflies round every value at every stage.  (Values
// far below the largest mostly come from cancellation and end in zero bits: n = 2^13 to 2^20,
// nuggets from 1e-8: 1 tile in some 500 falls back, nearly all of them the column tile with
// w = 0 of the spectral step's values; where 1 / lambda spans five decades and more, up to 1 in
// 8 of those.)
// Conversion in and out takes about 70 integer instructions per element, a stage 3 per element:
// 12 stages cost the issue time of some 3 FP64 instructions.
//
// The transforms of the first column (the eigenvalues) do not come here: with a small nugget the
// last bits of the small eigenvalues decide the outputs' digits, so they keep the FP64
// butterflies and their rounding.
//
// Tiles whose largest exponent lies outside [kW96MinExp, kW96MaxExp] (all zero, subnormal, near
// overflow, infinite or NaN) take the FP64 butterflies too.
#pragma once

#include "qk_common.cuh"

namespace qk {

constexpr uint32_t kW96MinExp = 128, kW96MaxExp = 1900;  // biased exponents

struct I96 {
  uint32_t a, b, c;  // least significant word first
};

__device__ __forceinline__ I96 i96_add(I96 x, I96 y) {
  I96 r;
  asm("add.cc.u32 %0, %3, %6;\n\taddc.cc.u32 %1, %4, %7;\n\taddc.u32 %2, %5, %8;"
      : "=&r"(r.a), "=&r"(r.b), "=&r"(r.c)
      : "r"(x.a), "r"(x.b), "r"(x.c), "r"(y.a), "r"(y.b), "r"(y.c));
  return r;
}
__device__ __forceinline__ I96 i96_sub(I96 x, I96 y) {
  I96 r;
  asm("sub.cc.u32 %0, %3, %6;\n\tsubc.cc.u32 %1, %4, %7;\n\tsubc.u32 %2, %5, %8;"
      : "=&r"(r.a), "=&r"(r.b), "=&r"(r.c)
      : "r"(x.a), "r"(x.b), "r"(x.c), "r"(y.a), "r"(y.b), "r"(y.c));
  return r;
}

// v as an integer over the biased exponent E >= that of v.
__device__ __forceinline__ I96 i96_from(double v, uint32_t E) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  const uint32_t e = (hi >> 20) & 0x7FFu;
  const uint32_t mh = (hi & 0xFFFFFu) | (e ? 0x100000u : 0u);
  uint32_t s = E - (e ? e : 1u);
  s = s > 95u ? 95u : s;
  uint32_t a = lo << 30, b = __funnelshift_r(lo, mh, 2), c = mh >> 2;
  if (s & 64u) a = c, b = 0u, c = 0u;
  if (s & 32u) a = b, b = c, c = 0u;
  a = __funnelshift_r(a, b, s & 31u), b = __funnelshift_r(b, c, s & 31u), c >>= (s & 31u);
  const uint32_t sg = (uint32_t)((int32_t)hi >> 31);
  return i96_sub(I96{a ^ sg, b ^ sg, c ^ sg}, I96{sg, sg, sg});  // negate: ~x + 1
}

// The integer over exponent E as a double, rounded to nearest even.
__device__ __forceinline__ double i96_to(I96 x, uint32_t E) {
  const uint32_t sg = (uint32_t)((int32_t)x.c >> 31);
  x = i96_sub(I96{x.a ^ sg, x.b ^ sg, x.c ^ sg}, I96{sg, sg, sg});
  uint32_t n = 0;
  if (x.c == 0u) n = 32, x.c = x.b, x.b = x.a, x.a = 0u;
  if (x.c == 0u) n += 32, x.c = x.b, x.b = x.a, x.a = 0u;  // a zero of 96 bits stays zero
  const uint32_t z = __clz((int)x.c) & 31u;
  n += z;
  const uint32_t h = __funnelshift_l(x.b, x.c, z), m = __funnelshift_l(x.a, x.b, z), l = x.a << z;
  const uint32_t rem = (m & 0x7FFu) << 1 | (l != 0u);
  uint32_t mlo = (m >> 11) | (h << 21), mhi = h >> 11;                    // 53 bits, leading one at bit 52
  const uint32_t up = rem + (mlo & 1u) > 0x800u ? 1u : 0u;                // round half to even
  asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, 0;" : "+r"(mlo), "+r"(mhi) : "r"(up));
  mhi += (E + 12u - n) << 20;                                             // the leading one adds 1
  return h ? __hiloint2double((int)(mhi | (sg & 0x80000000u)), (int)mlo) : 0.0;
}

// Whether v loses bits as an integer over E (its lowest set bit lies below 2^-82 of 2^E).
__device__ __forceinline__ bool i96_cut(double v, uint32_t E) {
  const uint32_t hi = (uint32_t)__double2hiint(v), e = (hi >> 20) & 0x7FFu;
  const uint64_t mant = ((uint64_t)((hi & 0xFFFFFu) | (e ? 0x100000u : 0u)) << 32) | (uint32_t)__double2loint(v);
  return (int)(E - (e ? e : 1u)) - 30 >= __ffsll((long long)mant) && mant;
}

// Range of the CTA's biased exponents from each thread's largest and smallest |high word|; red:
// 16 words of shared memory, free again after the caller's next barrier.
__device__ __forceinline__ void block_exp_range(uint32_t himax, uint32_t himin, uint32_t *red, uint32_t &E, uint32_t &En) {
  const uint32_t w = __reduce_max_sync(0xffffffffu, himax), u = __reduce_min_sync(0xffffffffu, himin);
  const uint32_t lane = threadIdx.x & 31, q = lane < (blockDim.x >> 5) ? lane : 0u;
  if (lane == 0) red[threadIdx.x >> 5] = w, red[8 + (threadIdx.x >> 5)] = u;
  __syncthreads();
  const uint32_t m = __reduce_max_sync(0xffffffffu, red[q]), n = __reduce_min_sync(0xffffffffu, red[8 + q]);
  E = m >> 20, En = n >> 20;
}

// The exponent E over which the CTA's values (16 per thread, `valid(l)` of them) become integers
// without losing a bit, 0 where a value may lose some or E is outside the range (then `far` is E
// or 0).  Every thread of the CTA calls it.
template <typename VF>
__device__ __forceinline__ uint32_t w96_exponent(const double (&v)[16], VF valid, uint32_t *red, uint32_t &far) {
  uint32_t hm = 0, hn = ~0u, E, En;
#pragma unroll
  for (int l = 0; l < 16; ++l)
    if (valid(l)) {
      const uint32_t h = (uint32_t)__double2hiint(v[l]) & 0x7FFFFFFFu;
      hm = h > hm ? h : hm;
      hn = h < hn ? h : hn;
    }
  block_exp_range(hm, hn, red, E, En);
  far = E < kW96MinExp || E > kW96MaxExp ? 0u : E;
  return E > En + 30u ? 0u : far;
}

}  // namespace qk
