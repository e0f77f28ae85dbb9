// FP64 Walsh-Hadamard butterflies in 96-bit integers (arXiv 2502.14256, Sec. 5.3).
//
// GB300 has about 2 FP64 lanes per SM and cycle, so an FP64 butterfly stage costs as much issue
// time as some 60 integer instructions per warp.  The WHT only adds and subtracts, so a tile is
// carried as integers over the tile's largest exponent E: X = +-mantissa 2^30 >> (E - e), 96-bit
// two's complement.  The top mantissa bit of the largest element sits at bit 82; 12 stages grow
// it to bit 94; elements down to 2^-30 of the largest keep all 53 bits and smaller ones are cut
// at 2^-82 of it.  The butterflies are exact (three adds with carry each), and each output is
// rounded to a double once: the error is one rounding per output instead of one per stage.
// Conversion in and out takes about 60 integer instructions per element, a stage 3 per
// element, so 12 stages cost about as much issue time as 2 FP64 instructions.
//
// The transforms of the first column (the eigenvalues) do not come here: with a small nugget the
// last bits of the small eigenvalues decide the outputs' digits, so they keep the FP64
// butterflies and their rounding.
//
// Tiles whose largest exponent lies outside [kW96MinExp, kW96MaxExp] (all zero, subnormal, near
// overflow, infinite or NaN) take the FP64 butterflies.
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

// Largest biased exponent of the CTA's values (each thread's largest |high word| given);
// red: 8 words of shared memory, free again after the caller's next barrier.
__device__ __forceinline__ uint32_t block_max_exp(uint32_t himax, uint32_t *red) {
  const uint32_t w = __reduce_max_sync(0xffffffffu, himax);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = w;
  __syncthreads();
  uint32_t m = 0;
  for (uint32_t q = 0; q < (blockDim.x >> 5); ++q) m = red[q] > m ? red[q] : m;
  return m >> 20;
}

}  // namespace qk
