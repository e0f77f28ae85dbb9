// Randomized QMC integration on top of the point sets (arXiv 2502.14256):
//   * the six test integrands of the numerical experiments (Sec. 6) evaluated at the points
//     of R randomizations, optionally through the baker transform x -> 1 - 2|x - 1/2|
//     (Sec. 4.2), without materialising the points;
//   * the RQMC estimate over R randomizations with its Student-t interval (Sec. 3.1);
//   * the squared worst-case error (generalized kernel discrepancy) of a cubature rule
//     (Sec. 3.2): closed forms for equal weights 1/n and the optimal weights K^-1 kappa,
//     and general weights through the spectrum (w^T K w = sum lambda |w~|^2, Sec. 5.4).
#include <cfloat>
#include <cmath>

#include "qk_column.cuh"
#include "qk_common.cuh"
#include "qk_internal.h"

namespace qk {

constexpr int kIntRL = 8;  // consecutive points per thread

template <typename T>
__device__ __forceinline__ T t_exp(T v) {
  if constexpr (sizeof(T) == 8) return exp(v);
  else return expf(v);
}
template <typename T>
__device__ __forceinline__ T t_cos(T v) {
  if constexpr (sizeof(T) == 8) return cos(v);
  else return cosf(v);
}

// Coordinate x = X 2^-32 of a word, or its baker transform 1 - 2|x - 1/2| = X' 2^-31 with
// X' = X (X < 2^31) or 2^32 - X, converted once to T.
__device__ __forceinline__ uint32_t baker_word(uint32_t X) { return (int32_t)X < 0 ? 0u - X : X; }
template <typename T>
__device__ __forceinline__ T coord(uint32_t X, bool baker) {
  if constexpr (sizeof(T) == 8) return baker ? u32_to_double(baker_word(X), 31) : u32_to_double(X, 32);
  else return baker ? __uint2float_rn(baker_word(X)) * 0x1p-31f : __uint2float_rn(X) * 0x1p-32f;
}

// Points of 64-bit mantissas: value m 2^(e - 63), m >= 2^63 or m = 0 (e then meaningless).
// A product keeps 63 bits; used where FP64 would spend its few lanes per SM on every dimension.
struct M64 {
  uint64_t m;
  int e;
};
__device__ __forceinline__ M64 m64_mul(M64 a, M64 b) {
  uint64_t p = __umul64hi(a.m, b.m);  // in [2^62, 2^64) for nonzero factors
  const int up = (p >> 63) ? 1 : 0;
  return {up ? p : p << 1, a.e + b.e + up};
}
__device__ __forceinline__ M64 m64_from(uint64_t v, int t) {  // v 2^-t
  const int c = __clzll((long long)v);
  return {v << (c & 63), 63 - c - t};
}
__device__ __forceinline__ double m64_to_double(M64 a) {  // rounded once; |a.e| below the FP64 range
  return u64_to_double(a.m, 63 - a.e);
}

// Per-dimension constants of the integrands, FP64 (d doubles), and for FP64 evaluation of the Genz
// functions the coefficients as fixed-point words (hi, lo): c = (hi 2^24 + lo) 2^-S.
struct FConst {
  double *cf;
  uint2 *fx;
};
constexpr int kGenzShiftOsc = 53, kGenzShiftCp = 57;  // sum c = 4.5 and 0.25: sum hi < 2^32

// Running state of one point over its dimensions: the first two coordinates, a product
// (G-function) and a linear form (Genz).  FP32: plain FP32 arithmetic.
template <typename T>
struct FState {
  T x1, x2, prod, lin;
};
// FP64: exact integers instead of FP64 sums and products (GB300: about 2 FP64 lanes per SM and
// cycle, a 32 x 32 + 64 bit multiply-add issues an order of magnitude faster).  Genz: sum c_j x_j
// from 57-bit fixed-point coefficients in two 64-bit accumulators (no rounding per
// dimension); G-function: |4x_j - 2| - a_j = N 2^-32 is an integer N, the product of the N
// keeps 63 bits.
template <>
struct FState<double> {
  uint32_t w1, w2;
  uint64_t hi, lo;
  M64 prod;
  uint32_t neg;
};

template <typename T>
__device__ __forceinline__ void fstate_init(FState<T> &s) {
  if constexpr (sizeof(T) == 8) {
    s.w1 = s.w2 = s.neg = 0, s.hi = s.lo = 0, s.prod = {1ull << 63, 0};
  } else {
    s = FState<T>{T(0), T(0), T(1), T(0)};
  }
}

__device__ __forceinline__ void fstate_add(FState<float> &s, int f, uint32_t j, uint32_t X, bool baker, const FConst &k) {
  const float x = coord<float>(X, baker);
  if (j == 0) s.x1 = x;
  if (j == 1) s.x2 = x;
  if (f == QK_F_GFUN) {
    const float a = (float)k.cf[j];
    s.prod *= (fabsf(4.f * x - 2.f) - a) / (1.f + a);
  } else if (f == QK_F_GENZ_OSC || f == QK_F_GENZ_CP) {
    s.lin = fmadd((float)k.cf[j], x, s.lin);
  }
}
__device__ __forceinline__ void fstate_add(FState<double> &s, int f, uint32_t j, uint32_t X, bool baker, const FConst &k) {
  if (j == 0) s.w1 = X;
  if (j == 1) s.w2 = X;
  if (f == QK_F_GFUN) {
    // |4x - 2| 2^32 (a multiple of 4 or 8, below 2^34) minus a_j 2^32 = (j - 1) 2^31 (0-based j)
    const int64_t v = baker ? ((int64_t)baker_word(X) << 3) - (1ll << 33) : ((int64_t)X << 2) - (1ll << 33);
    const int64_t N = (v < 0 ? -v : v) - (((int64_t)j - 1) << 31);
    s.neg ^= N < 0 ? 1u : 0u;
    s.prod = m64_mul(s.prod, m64_from((uint64_t)(N < 0 ? -N : N), 32));
  } else if (f == QK_F_GENZ_OSC || f == QK_F_GENZ_CP) {
    const uint2 c = k.fx[j];
    const uint32_t W = baker ? baker_word(X) : X;
    s.hi += (uint64_t)c.x * W;  // sum hi_j < 2^32, W < 2^32: no overflow
    s.lo += (uint64_t)c.y * W;  // 2^24 2^32 d, d <= 256
  }
}

template <typename T>
__device__ __forceinline__ T simple_value(int f, T x1, T x2) {
  if (f == QK_F_SIMPLE1) return x1 * t_exp(x1) - T(1);
  if (f == QK_F_SIMPLE2) return x2 * t_exp(x1 * x2) / T(0.71828182845904523536) - T(1);  // e - 2
  const T t1 = (x1 - T(0.5)) / T(50), t2 = (x2 - T(0.5)) / T(50);  // Oakley
  return T(5) + t1 + t2 + T(2) * t_cos(t1) + T(2) * t_cos(t2);
}
__device__ __forceinline__ float fstate_value(const FState<float> &s, int f, uint32_t d, bool, const M64 &) {
  if (f == QK_F_GFUN) return s.prod;
  if (f == QK_F_GENZ_OSC) return cosf(s.lin);  // cos(-s) = cos(s)
  if (f == QK_F_GENZ_CP) return powf(1.f + s.lin, -(float)(d + 1));
  return simple_value<float>(f, s.x1, s.x2);
}
__device__ __forceinline__ double fstate_value(const FState<double> &s, int f, uint32_t d, bool baker, const M64 &ginv) {
  const int wb = baker ? 31 : 32;
  if (f == QK_F_GFUN) {
    const double v = s.prod.m ? m64_to_double(m64_mul(s.prod, ginv)) : 0.0;
    return s.neg ? -v : v;
  }
  if (f == QK_F_GENZ_OSC)
    return cos(fma(u64_to_double(s.hi, 0), 0x1p24, u64_to_double(s.lo, 0)) * exp2neg(0.0, kGenzShiftOsc + wb));
  if (f == QK_F_GENZ_CP) {
    // (1 + s)^-(d + 1): 1 + s = m 2^-63 with s below 1/4, the power by squaring on 64-bit
    // mantissas (relative error below (d + 1) 2^-62), one FP64 reciprocal
    const int sh = kGenzShiftCp - 24 + wb - 63;  // hi 2^(24 - S - wb) in units of 2^-63
    M64 b{(1ull << 63) + ((s.hi + (s.lo >> 24)) >> sh), 0}, r{1ull << 63, 0};
    for (uint32_t k = d + 1;; k >>= 1) {
      if (k & 1u) r = m64_mul(r, b);
      if (k <= 1u) break;
      b = m64_mul(b, b);
    }
    return rcp64(m64_to_double(r));
  }
  return simple_value<double>(f, coord<double>(s.w1, baker), coord<double>(s.w2, baker));
}

// y[r][i] = f(x_i) for the points at positions i0 + [0, n) of randomization r0 + blockIdx.y.
// A CTA of NT threads covers NT kIntRL consecutive positions aligned to that; a thread makes
// kIntRL consecutive points dimension by dimension (nets: seeded from the XOR tables of the
// tile, lane and warp bits, then one XOR per point with a column known at compile time, as in
// point generation; lattices: brev(i) g + D).  NT = 64 where tiles of 2048 points would leave
// a wave partly empty (10 x 2^15 points: 160 tiles on 152 SMs).
template <typename T, bool NET, int NT>
__global__ void __launch_bounds__(NT) k_integrand(uint32_t d, int order, const uint32_t *__restrict__ Ct,
                                                  const uint32_t *__restrict__ g, const uint32_t *__restrict__ D,
                                                  uint32_t r0, uint64_t i0, uint64_t n, int f, int baker,
                                                  T *__restrict__ y) {
  constexpr int NP = NT * kIntRL, NW = NT / 32;
  extern __shared__ __align__(16) unsigned char ism[];
  __shared__ double sh[32];
  __shared__ double s_scale;
  __shared__ M64 s_ginv;
  FConst fc;
  fc.cf = reinterpret_cast<double *>(ism);                        // (d) coefficients
  fc.fx = reinterpret_cast<uint2 *>(fc.cf + d);                   // (d) fixed-point coefficients
  uint32_t *ztile = reinterpret_cast<uint32_t *>(fc.fx + d);      // (d) tile words, shift included
  uint32_t *zlane = ztile + d;                                    // (32 d) nets
  uint32_t *zwarp = zlane + 32 * d;                               // (NW d) nets
  uint32_t *steps = zwarp + NW * d;                               // (3 d) nets: step columns
  const uint32_t rl = blockIdx.y, r = r0 + rl;
  const uint64_t base = ((i0 / NP) + blockIdx.x) * NP;  // < 2^32
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  // coefficients (FP64): Genz oscillatory / corner peak (Sec. 6), G-function a_j = (j - 2)/2
  if (f == QK_F_GENZ_OSC || f == QK_F_GENZ_CP) {
    double sum = 0.0;
    for (uint32_t j = t; j < d; j += NT) {
      const double ct = f == QK_F_GENZ_OSC ? exp((double)(j + 1) * log(1e-8) / (double)d)
                                           : 1.0 / ((double)(j + 1) * (double)(j + 1));
      fc.cf[j] = ct;
      sum += ct;
    }
    sum = block_sum(sum, sh);
    if (t == 0) s_scale = (f == QK_F_GENZ_OSC ? 4.5 : 0.25) / sum;
    __syncthreads();
    const double fix = exp2neg(0.0, -(f == QK_F_GENZ_OSC ? kGenzShiftOsc : kGenzShiftCp));
    for (uint32_t j = t; j < d; j += NT) {
      const double c = fc.cf[j] * s_scale;
      const uint64_t q = (uint64_t)__double2ull_rn(c * fix);
      fc.cf[j] = c;
      fc.fx[j] = make_uint2((uint32_t)(q >> 24), (uint32_t)q & 0xFFFFFFu);
    }
  } else {
    for (uint32_t j = t; j < d; j += NT) fc.cf[j] = ((double)(j + 1) - 2.0) / 2.0;
    if (f == QK_F_GFUN && sizeof(T) == 8 && t == 0) {
      // 1 / prod_j (1 + a_j) = 2^d / d! : 64-bit mantissas, the reciprocal from a long division
      M64 p{1ull << 63, 0};
      for (uint32_t j = 2; j <= d; ++j) p = m64_mul(p, m64_from(j, 0));
      // floor(2^126 / m) for m in [2^63, 2^64): bit by bit
      uint64_t q = 0, rem = 1ull << 62;  // remainder of 2^62 after 0 quotient bits, then 64 steps of 2 rem
      for (int k = 0; k < 64; ++k) {
        const bool top = rem >> 63;
        rem <<= 1;
        q <<= 1;
        if (top || rem >= p.m) rem -= p.m, q |= 1;
      }
      const M64 inv = m64_from(q, 63);  // 2^63 / m in (1/2, 1]
      s_ginv = {inv.m, inv.e - p.e + (int)d};
    }
  }
  if constexpr (NET) {
    const uint32_t *Cr = Ct + (size_t)r * d * 32;
    for (uint32_t q = t; q < 32 * d; q += NT) {
      const uint32_t j = q >> 5, v = order_map(order, (q & 31) * kIntRL);
      uint32_t acc = 0;
#pragma unroll
      for (int k = 2; k < 8; ++k)  // digits 3..7 of the position (and 2 in Gray order): independent loads
        if ((v >> k) & 1u) acc ^= Cr[j * 32 + k];
      zlane[q] = acc;
    }
    for (uint32_t q = t; q < NW * d; q += NT) {
      const uint32_t w = q / d, j = q - w * d;
      zwarp[w * d + j] = xor_columns(Cr + j * 32, order_map(order, (w * 32) * kIntRL));
    }
    for (uint32_t j = t; j < d; j += NT) {
      const uint32_t v = order_map(order, (uint32_t)base);
      uint32_t acc = D ? D[(size_t)r * d + j] : 0u;
#pragma unroll
      for (int k = 0; k < 32; ++k)
        if ((v >> k) & 1u) acc ^= Cr[j * 32 + k];
      ztile[j] = acc;
      const uint32_t c0 = Cr[j * 32], c1 = Cr[j * 32 + 1], c2 = Cr[j * 32 + 2];
      steps[3 * j] = c0;
      steps[3 * j + 1] = order == QK_GRAY ? c1 : (c0 ^ c1);
      steps[3 * j + 2] = order == QK_GRAY ? c2 : (c0 ^ c1 ^ c2);
    }
  } else {
    for (uint32_t j = t; j < d; j += NT) ztile[j] = D ? D[(size_t)r * d + j] : 0u;
  }
  __syncthreads();
  FState<T> st[kIntRL];
#pragma unroll
  for (int k = 0; k < kIntRL; ++k) fstate_init<T>(st[k]);
  const uint32_t i_first = (uint32_t)base + (uint32_t)t * kIntRL;
  for (uint32_t j = 0; j < d; ++j) {
    uint32_t w[kIntRL];
    if constexpr (NET) {
      const uint32_t s0 = steps[3 * j], s1 = steps[3 * j + 1], s2 = steps[3 * j + 2];
      uint32_t x = ztile[j] ^ zlane[j * 32 + lane] ^ zwarp[warp * d + j];
      w[0] = x;
      x ^= s0, w[1] = x;
      x ^= s1, w[2] = x;
      x ^= s0, w[3] = x;
      x ^= s2, w[4] = x;
      x ^= s0, w[5] = x;
      x ^= s1, w[6] = x;
      x ^= s0, w[7] = x;
    } else {
      const uint32_t gj = g[j], dj = ztile[j];
#pragma unroll
      for (int k = 0; k < kIntRL; ++k) w[k] = __brev(i_first + k) * gj + dj;
    }
#pragma unroll
    for (int k = 0; k < kIntRL; ++k) fstate_add(st[k], f, j, w[k], baker != 0, fc);
  }
  T *yr = y + (size_t)rl * n;
  const M64 ginv = s_ginv;
#pragma unroll
  for (int k = 0; k < kIntRL; ++k) {
    const uint64_t i = (uint64_t)i_first + k;
    if (i >= i0 && i < i0 + n) yr[i - i0] = fstate_value(st[k], f, d, baker != 0, ginv);
  }
}

template <typename T, int NT>
static int launch_integrand_t(const qk_pointset *ps, uint32_t r0, uint32_t nr, uint64_t i0, uint64_t n, int f,
                              int baker, T *y, cudaStream_t st) {
  const uint32_t d = ps->d;
  constexpr int NP = NT * kIntRL;
  const uint64_t tiles = (i0 + n - 1) / NP - i0 / NP + 1;
  const size_t smem = 2 * sizeof(double) * d + sizeof(uint32_t) * ((size_t)d + 32 * d + (NT / 32) * d + 3 * d);
  const bool net = ps->kind == QK_NET_B2;
  if (net) smem_optin<k_integrand<T, true, NT>>(smem);
  else smem_optin<k_integrand<T, false, NT>>(smem);
  for (uint32_t rc = 0; rc < nr; rc += 65535) {  // grid.y limit
    const uint32_t cnt = nr - rc < 65535 ? nr - rc : 65535;
    dim3 grid((unsigned)tiles, cnt);
    T *yc = y + (size_t)rc * n;
    if (net)
      k_integrand<T, true, NT><<<grid, NT, smem, st>>>(d, ps->order, ps->Ct, nullptr, ps->D, r0 + rc, i0, n, f, baker, yc);
    else
      k_integrand<T, false, NT><<<grid, NT, smem, st>>>(d, ps->order, nullptr, ps->g, ps->D, r0 + rc, i0, n, f, baker, yc);
    int rc_ = check_launch("qk_integrand");
    if (rc_) return rc_;
  }
  return QK_OK;
}
template <typename T>
static int launch_integrand(const qk_pointset *ps, uint32_t r0, uint32_t nr, uint64_t i0, uint64_t n, int f, int baker,
                            T *y, cudaStream_t st) {
  // tiles of 2048 points from eight CTAs per SM on, of 512 below
  return (n / (256 * kIntRL)) * nr >= 8ull * sm_count() ? launch_integrand_t<T, 256>(ps, r0, nr, i0, n, f, baker, y, st)
                                                        : launch_integrand_t<T, 64>(ps, r0, nr, i0, n, f, baker, y, st);
}

// ------------------------------------------------------------- row sums and the RQMC estimate
// Sums of the rows of a (rows, n) array by a cluster of kRowCta CTAs per row (no scratch to
// leave partial sums in: they meet in the first CTA's shared memory).  One CTA per row took
// 14 us for 10 rows of 2^15 doubles; rows are many times longer than a CTA.
constexpr int kRowCta = 8, kRowNT = 512;

// Every thread of every CTA of the cluster calls both (release on arrival, acquire on return).
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait;" ::: "memory"); }

// FP64 sum over this cluster's row of f(i) for i < n; valid in thread 0 of the cluster's rank 0.
// Another CTA's shared memory exists once that CTA has started: each arrives at the cluster's
// barrier first thing and waits before its store, so the row's loads hide the wait (a CTA of
// rank k has no element of a row shorter than 512 k and would store at once).
template <typename F>
__device__ __forceinline__ double cluster_row_sum(uint64_t n, F f) {
  __shared__ double sh[32];
  __shared__ double part[kRowCta];
  cluster_arrive();
  uint32_t rank;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  double s0 = 0.0, s1 = 0.0;
  const uint64_t step = (uint64_t)kRowCta * kRowNT;
  uint64_t i = (uint64_t)rank * kRowNT + threadIdx.x;
  for (; i + step < n; i += 2 * step) s0 += f(i), s1 += f(i + step);
  if (i < n) s0 += f(i);
  const double s = block_sum(s0 + s1, sh);
  cluster_wait();
  if (threadIdx.x == 0) {
    uint32_t local = (uint32_t)__cvta_generic_to_shared(&part[rank]), remote;
    asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(remote) : "r"(local));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(remote), "d"(s) : "memory");
  }
  // the parts are in place, and no CTA has left before
  cluster_arrive();
  cluster_wait();
  double tot = 0.0;
  if (rank == 0 && threadIdx.x == 0)
    for (int k = 0; k < kRowCta; ++k) tot += part[k];
  return tot;
}
__device__ __forceinline__ bool cluster_first() {
  uint32_t rank;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  return rank == 0 && threadIdx.x == 0;
}

// launch(r0, cnt): rows r0 .. r0 + cnt - 1, cnt * kRowCta CTAs (kept below the grid limit).
template <typename F>
static void by_rows(uint64_t rows, F launch) {
  for (uint64_t r0 = 0; r0 < rows; r0 += 1u << 27) launch(r0, (unsigned)(rows - r0 < (1u << 27) ? rows - r0 : 1u << 27));
}

template <typename T>
__global__ void __cluster_dims__(kRowCta, 1, 1) __launch_bounds__(kRowNT) k_row_means(const T *__restrict__ y, uint64_t n,
                                                                                     double *__restrict__ mu_r) {
  const uint64_t row = blockIdx.x / kRowCta;
  const T *yr = y + row * n;
  const double tot = cluster_row_sum(n, [&](uint64_t i) { return f2d_exact(yr[i]); });
  if (cluster_first()) mu_r[row] = tot / (double)n;
}

// out = [mu, sigma, half width, t, mu_1 .. mu_R]: mu_r already in out[4 ..].  One warp.
__global__ void k_rqmc_final(uint32_t R, double t_star, double *__restrict__ out) {
  const double *mu_r = out + 4;
  const uint32_t lane = threadIdx.x;
  auto warp_total = [](double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  double mu = 0.0;
  for (uint32_t r = lane; r < R; r += 32) mu += mu_r[r];
  mu = warp_total(mu) / (double)R;
  double ss = 0.0;
  for (uint32_t r = lane; r < R; r += 32) ss += (mu_r[r] - mu) * (mu_r[r] - mu);
  ss = warp_total(ss);
  if (lane) return;
  const double sigma = sqrt(ss / (double)(R - 1));
  out[0] = mu;
  out[1] = sigma;
  out[2] = t_star * sigma / sqrt((double)R);
  out[3] = t_star;
}

// ------------------------------------------------ Student-t quantile (host)
// Regularised incomplete beta I_x(a, b) by its continued fraction (evaluated with the
// modified Lentz method), using I_x(a, b) = 1 - I_{1-x}(b, a) where the fraction converges
// slowly (x > (a + 1)/(a + b + 2)).
static double inc_beta_cf(double a, double b, double x) {
  const double tiny = 1e-300;
  double c = 1.0, dd = 1.0 - (a + b) * x / (a + 1.0);
  if (std::fabs(dd) < tiny) dd = tiny;
  dd = 1.0 / dd;
  double h = dd;
  for (int k = 1; k <= 400; ++k) {
    // even step: k (b - k) x / ((a + 2k - 1)(a + 2k))
    double num = k * (b - k) * x / ((a + 2.0 * k - 1.0) * (a + 2.0 * k));
    dd = 1.0 + num * dd;
    c = 1.0 + num / c;
    if (std::fabs(dd) < tiny) dd = tiny;
    if (std::fabs(c) < tiny) c = tiny;
    dd = 1.0 / dd;
    h *= dd * c;
    // odd step: -(a + k)(a + b + k) x / ((a + 2k)(a + 2k + 1))
    num = -(a + k) * (a + b + k) * x / ((a + 2.0 * k) * (a + 2.0 * k + 1.0));
    dd = 1.0 + num * dd;
    c = 1.0 + num / c;
    if (std::fabs(dd) < tiny) dd = tiny;
    if (std::fabs(c) < tiny) c = tiny;
    dd = 1.0 / dd;
    const double del = dd * c;
    h *= del;
    if (std::fabs(del - 1.0) < 1e-16) break;
  }
  return h;
}

static double inc_beta(double a, double b, double x) {
  if (x <= 0.0) return 0.0;
  if (x >= 1.0) return 1.0;
  const double lbeta = std::lgamma(a) + std::lgamma(b) - std::lgamma(a + b);
  const double front = std::exp(a * std::log(x) + b * std::log1p(-x) - lbeta);
  if (x < (a + 1.0) / (a + b + 2.0)) return front * inc_beta_cf(a, b, x) / a;
  return 1.0 - front * inc_beta_cf(b, a, 1.0 - x) / b;
}

// P(T <= t) for Student's t with df degrees of freedom: for t >= 0,
// 1 - I_{df/(df + t^2)}(df/2, 1/2) / 2, and symmetry for t < 0.
static double student_t_cdf(double t, double df) {
  const double tail = 0.5 * inc_beta(0.5 * df, 0.5, df / (df + t * t));
  return t >= 0.0 ? 1.0 - tail : tail;
}

// The quantile by bisection on the monotone CDF (to the last bit of the bracket).
static double student_t_quantile(double df, double p) {
  if (p == 0.5) return 0.0;
  const bool lower = p < 0.5;
  const double q = lower ? 1.0 - p : p;
  double lo = 0.0, hi = 1.0;
  while (student_t_cdf(hi, df) < q && hi < 1e300) hi *= 2.0;
  for (int it = 0; it < 2000; ++it) {
    const double mid = 0.5 * (lo + hi);
    if (mid <= lo || mid >= hi) break;
    if (student_t_cdf(mid, df) < q) lo = mid;
    else hi = mid;
  }
  const double v = 0.5 * (lo + hi);
  return lower ? -v : v;
}

// --------------------------------------------- squared worst-case error (Sec. 3.2)
// From the first column in form P (p = k_1/zeta - 1), per batch entry, with S = sum_i p_i
// (FP64 sums) and lambda_0 = zeta (n + S) for the kernel without nugget:
//   equal weights 1/n:        int int K - 2 zeta + 1^T K 1 / n^2 = zeta S / n
//   optimal weights K^-1 kappa = (zeta / lambda_0) 1:  zeta - zeta^2 n / lambda_0 = zeta S / (n + S)
// (kappa_i = int K(u, x_i) du = zeta and int int K = zeta: each one-dimensional K_alpha
// integrates to zero).  out (batch, 3) = [equal, optimal, optimal weight value].
template <typename T>
__global__ void __cluster_dims__(kRowCta, 1, 1) __launch_bounds__(kRowNT) k_discrepancy_closed(const T *__restrict__ col, int form,
                                                                                              uint64_t n, double zeta,
                                                                                              double *__restrict__ out) {
  const uint64_t row = blockIdx.x / kRowCta;
  const T *cr = col + row * n;
  const double S = form == QK_COL_P ? cluster_row_sum(n, [&](uint64_t i) { return f2d_exact(cr[i]); })
                                    : cluster_row_sum(n, [&](uint64_t i) { return (double)cr[i] / zeta - 1.0; });
  if (cluster_first()) {
    const double nn = (double)n;
    double *o = out + row * 3;
    o[0] = zeta * S / nn;
    o[1] = zeta * S / (nn + S);
    o[2] = 1.0 / (nn + S);  // zeta / lambda_0
  }
}

__device__ __forceinline__ double sq_abs(float v) { return (double)v * (double)v; }
__device__ __forceinline__ double sq_abs(double v) { return v * v; }
__device__ __forceinline__ double sq_abs(float2 v) { return (double)v.x * v.x + (double)v.y * v.y; }
__device__ __forceinline__ double sq_abs(double2 v) { return v.x * v.x + v.y * v.y; }

// General weights: per vector v the partial sums of lambda_w |W_w|^2 / n (W = the
// unnormalised transform of the weights, so sum lambda |W|^2 / n = w^T K w) and of w.
template <typename E>
__global__ void k_quad_lambda(const E *__restrict__ X, const double *__restrict__ lam, int m, uint32_t nw,
                              double *__restrict__ part) {
  __shared__ double sh[32];
  const uint64_t n = 1ull << m;
  const uint32_t v = blockIdx.y;
  const double *lr = lam + (uint64_t)(v / nw) * n;
  const E *xv = X + (uint64_t)v * n;
  double q = 0.0;
  for (uint64_t w = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; w < n; w += (uint64_t)gridDim.x * blockDim.x)
    q += lr[w] * sq_abs(xv[w]);
  const double sq = block_sum(q, sh);
  if (threadIdx.x == 0) part[(uint64_t)v * gridDim.x + blockIdx.x] = sq / (double)n;
}

template <typename T>
__global__ void __cluster_dims__(kRowCta, 1, 1) __launch_bounds__(kRowNT) k_weight_sums(const T *__restrict__ w, uint64_t n,
                                                                                       double *__restrict__ out) {
  const uint64_t row = blockIdx.x / kRowCta;
  const T *wr = w + row * n;
  const double tot = cluster_row_sum(n, [&](uint64_t i) { return f2d_exact(wr[i]); });
  if (cluster_first()) out[row] = tot;
}

__global__ void k_discrepancy_final(uint32_t nvec, uint32_t blocks, double zeta, const double *__restrict__ part,
                                    const double *__restrict__ wsum, double *__restrict__ out) {
  const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= nvec) return;
  double q = 0.0;
  for (uint32_t b = 0; b < blocks; ++b) q += part[(uint64_t)v * blocks + b];
  out[v] = zeta - 2.0 * zeta * wsum[v] + q;
}

constexpr uint32_t kDiscBlocks = 64;

template <typename T, typename E>
static int discrepancy_weights_t(int family, uint32_t m, uint32_t batch, uint32_t nw, const double *lam, const T *w,
                                 double zeta, double *out, void *ws, cudaStream_t st) {
  const uint32_t nvec = batch * nw;
  const uint64_t n = 1ull << m, cnt = (uint64_t)nvec << m;
  unsigned char *p = (unsigned char *)ws;
  E *X = (E *)p;
  p += align256(sizeof(E) * cnt);
  double *part = (double *)p;
  p += align256(sizeof(double) * nvec * kDiscBlocks);
  double *wsum = (double *)p;
  by_rows(nvec, [&](uint64_t r0, unsigned c) { k_weight_sums<T><<<c * kRowCta, kRowNT, 0, st>>>(w + r0 * n, n, wsum + r0); });
  int rc = check_launch("discrepancy weight sums");
  if (rc) return rc;
  // unnormalised forward transform of the weights (the solve's first half)
  if ((rc = op_forward_real(family, m, nvec, sizeof(T) == 8 ? QK_F64 : QK_F32, w, X, st))) return rc;
  const uint32_t blocks = n < 256 * kDiscBlocks ? (uint32_t)((n + 255) / 256) : kDiscBlocks;
  k_quad_lambda<E><<<dim3(blocks, nvec), 256, 0, st>>>(X, lam, (int)m, nw, part);
  if ((rc = check_launch("discrepancy quadratic form"))) return rc;
  // part holds `blocks` entries per vector; the final sums that many
  k_discrepancy_final<<<(nvec + 127) / 128, 128, 0, st>>>(nvec, blocks, zeta, part, wsum, out);
  return check_launch("discrepancy final");
}

size_t ws_discrepancy(int family, uint32_t m, uint32_t batch, uint32_t nw, int dtype) {
  const uint64_t nvec = (uint64_t)batch * nw;
  return ws_matvec(family, m, batch, nw, dtype) + align256(sizeof(double) * nvec * kDiscBlocks) +
         align256(sizeof(double) * nvec);
}

}  // namespace qk

using namespace qk;

#define QK_TRY(x)        \
  do {                   \
    int rc_ = (x);       \
    if (rc_) return rc_; \
  } while (0)

extern "C" {

int qk_student_t_quantile(double df, double p, double *q) {
  set_error("%s", "");
  if (!q) return fail(QK_EINVAL, "qk_student_t_quantile: q is NULL");
  if (!(df > 0.0) || !std::isfinite(df)) return fail(QK_EINVAL, "degrees of freedom must be finite and > 0");
  if (!(p > 0.0 && p < 1.0)) return fail(QK_EINVAL, "p must lie in (0, 1)");
  *q = student_t_quantile(df, p);
  return QK_OK;
}

int qk_integrand(const qk_pointset *ps, uint32_t r0, uint32_t nr, uint64_t i0, uint64_t n, int32_t f, int32_t baker,
                 int32_t dtype, void *y, qk_stream stream) {
  set_error("%s", "");
  QK_TRY(check_pointset(ps, r0, nr));
  if (dtype != QK_F64 && dtype != QK_F32) return fail(QK_EINVAL, "dtype must be QK_F64 or QK_F32");
  if (f < QK_F_SIMPLE1 || f > QK_F_GENZ_CP) return fail(QK_EINVAL, "unknown integrand %d", f);
  if (f == QK_F_SIMPLE1 && ps->d != 1) return fail(QK_EINVAL, "the simple d = 1 integrand needs d = 1");
  if ((f == QK_F_SIMPLE2 || f == QK_F_OAKLEY) && ps->d != 2)
    return fail(QK_EINVAL, "this integrand is defined for d = 2 (point set has d = %u)", ps->d);
  if (i0 + n > (1ull << 32)) return fail(QK_EINVAL, "positions beyond 2^32");
  if (n == 0 || nr == 0) return QK_OK;
  if (!y) return fail(QK_EINVAL, "qk_integrand: y is NULL");
  const cudaStream_t st = (cudaStream_t)stream;
  return dtype == QK_F64 ? launch_integrand<double>(ps, r0, nr, i0, n, f, baker, (double *)y, st)
                         : launch_integrand<float>(ps, r0, nr, i0, n, f, baker, (float *)y, st);
}

int qk_rqmc(uint32_t R, uint64_t n, int32_t dtype, const void *y, double tau, double *out, qk_stream stream) {
  set_error("%s", "");
  if (dtype != QK_F64 && dtype != QK_F32) return fail(QK_EINVAL, "dtype must be QK_F64 or QK_F32");
  if (R < 2) return fail(QK_EINVAL, "the interval needs R >= 2 randomizations");
  if (n == 0) return fail(QK_EINVAL, "n must be >= 1");
  if (!(tau > 0.0 && tau < 1.0)) return fail(QK_EINVAL, "tau must lie in (0, 1)");
  if (!y || !out) return fail(QK_EINVAL, "qk_rqmc: NULL array");
  const double t_star = student_t_quantile((double)(R - 1), 1.0 - 0.5 * tau);
  const cudaStream_t st = (cudaStream_t)stream;
  by_rows(R, [&](uint64_t r0, unsigned c) {
    if (dtype == QK_F64) k_row_means<double><<<c * kRowCta, kRowNT, 0, st>>>((const double *)y + r0 * n, n, out + 4 + r0);
    else k_row_means<float><<<c * kRowCta, kRowNT, 0, st>>>((const float *)y + r0 * n, n, out + 4 + r0);
  });
  QK_TRY(check_launch("rqmc means"));
  k_rqmc_final<<<1, 32, 0, st>>>(R, t_star, out);
  return check_launch("rqmc interval");
}

int qk_discrepancy(int32_t family, uint32_t m, uint32_t batch, int32_t dtype, int32_t form, const void *col,
                   double zeta, double *out, qk_stream stream) {
  set_error("%s", "");
  if (family != QK_DSI && family != QK_SI) return fail(QK_EINVAL, "family must be QK_DSI or QK_SI");
  if (dtype != QK_F64 && dtype != QK_F32) return fail(QK_EINVAL, "dtype must be QK_F64 or QK_F32");
  if (m > QK_MAX_M) return fail(QK_EINVAL, "m = %u exceeds QK_MAX_M = %d", m, QK_MAX_M);
  if (form != QK_COL_K1 && form != QK_COL_P) return fail(QK_EINVAL, "form must be QK_COL_K1 or QK_COL_P");
  if (!(zeta > 0.0)) return fail(QK_EINVAL, "zeta must be > 0");
  if (batch == 0) return QK_OK;
  if (!col || !out) return fail(QK_EINVAL, "qk_discrepancy: NULL array");
  const cudaStream_t st = (cudaStream_t)stream;
  const uint64_t n = 1ull << m;
  by_rows(batch, [&](uint64_t r0, unsigned c) {
    if (dtype == QK_F64)
      k_discrepancy_closed<double><<<c * kRowCta, kRowNT, 0, st>>>((const double *)col + r0 * n, form, n, zeta, out + 3 * r0);
    else
      k_discrepancy_closed<float><<<c * kRowCta, kRowNT, 0, st>>>((const float *)col + r0 * n, form, n, zeta, out + 3 * r0);
  });
  return check_launch("qk_discrepancy");
}

int qk_discrepancy_weights(int32_t family, uint32_t m, uint32_t batch, uint32_t nw, int32_t dtype, const double *lam,
                           const void *w, double zeta, double *out, void *ws, size_t ws_bytes, qk_stream stream) {
  set_error("%s", "");
  if (family != QK_DSI && family != QK_SI) return fail(QK_EINVAL, "family must be QK_DSI or QK_SI");
  if (dtype != QK_F64 && dtype != QK_F32) return fail(QK_EINVAL, "dtype must be QK_F64 or QK_F32");
  if (m > QK_MAX_M) return fail(QK_EINVAL, "m = %u exceeds QK_MAX_M = %d", m, QK_MAX_M);
  if (!(zeta > 0.0)) return fail(QK_EINVAL, "zeta must be > 0");
  if (batch == 0 || nw == 0) return QK_OK;
  if ((uint64_t)batch * nw > 0xFFFFFFFFull) return fail(QK_EINVAL, "batch x nw exceeds 2^32");
  if (!lam || !w || !out) return fail(QK_EINVAL, "qk_discrepancy_weights: NULL array");
  QK_TRY(check_ws(ws, ws_bytes, ws_discrepancy(family, m, batch, nw, dtype)));
  const cudaStream_t st = (cudaStream_t)stream;
  if (family == QK_DSI)
    return dtype == QK_F64 ? discrepancy_weights_t<double, double>(family, m, batch, nw, lam, (const double *)w, zeta, out, ws, st)
                           : discrepancy_weights_t<float, float>(family, m, batch, nw, lam, (const float *)w, zeta, out, ws, st);
  return dtype == QK_F64 ? discrepancy_weights_t<double, double2>(family, m, batch, nw, lam, (const double *)w, zeta, out, ws, st)
                         : discrepancy_weights_t<float, float2>(family, m, batch, nw, lam, (const float *)w, zeta, out, ws, st);
}

}  // extern "C"
