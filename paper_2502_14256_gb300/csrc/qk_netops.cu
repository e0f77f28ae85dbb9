// Standalone spectral operations of nets (arXiv 2502.14256, Sec. 5.4) in as few passes over
// memory as the transform needs: eigenvalues, K^-1 y and K y, and the MLL's forward and
// adjoint transforms, with the loads, the spectral step and the stores inside the transform's
// passes.
//
//   n = 2^m up to one tile (2^13 FP32, 2^12 FP64): ONE kernel, one CTA per vector, the vector
//     in shared memory between a load and a store;
//   up to 2^21 (FP32) / 2^20 (FP64): contiguous tiles of the low bits, column tiles of the high
//     bits with the spectral step inside (forward high bits, scale, inverse high bits), and
//     contiguous tiles again: 3 kernels for K^-1 y, 2 for the eigenvalues and their doubling.
//
// FP64 transforms of data run in 96-bit integers (qk_wht96.cuh).  The eigenvalues' transforms and
// all FP32 ones keep the butterflies of the multi-pass transform, bits upwards: with a small
// nugget the last bits of the small eigenvalues decide the outputs' digits, and an FP32
// spectrum's rounding shows in every FP64 sum over it.  K^-1 y and K y run their inverse from
// the high bits down.
#include <type_traits>

#include "qk_common.cuh"
#include "qk_fused.cuh"
#include "qk_internal.h"
#include "qk_netops.h"

namespace qk {

// lambda = zmul x + dc [w = 0] + eta with the floor and the sign test of qk_eigs, and the doubling
// update lambda' = lambda +- t, t = zmul x + dc [w = 0].  The common form costs one FP64 fma per
// value: eta > 0, x zero or normal; the floor compares as integers (the order of positive
// doubles; a value below eta, negative or NaN becomes eta, and is then positive).  A thread that
// holds w = 0 or a special x, and every thread where eta <= 0, repeats its elements in the
// general form behind a branch: an FP64 instruction that a predicate turns off still takes its
// time on GB300 (measured: 6 instead of 2 per element and update).
struct LamArgs {
  double zmul, dc, eta;
  uint32_t *status;
};
__device__ __forceinline__ double lam_floor_int(double v, double eta, bool &floored) {
  const long long b = __double_as_longlong(v);
  if (b >= __double_as_longlong(eta) && b <= 0x7FF0000000000000ll) return v;
  floored = true;
  return eta;
}
template <typename T>
__device__ __forceinline__ double lam_fast(T x, const LamArgs &a, bool &rare, bool &floored) {
  rare |= f2d_special(x);
  return lam_floor_int(fma(a.zmul, f2d_normal(x), a.eta), a.eta, floored);
}
template <typename T>
__device__ __forceinline__ void lam_pair_fast(T x, double old, const LamArgs &a, double (&v)[2], bool &rare, bool &floored) {
  const double xd = f2d_normal(x);
  rare |= f2d_special(x);
  v[0] = lam_floor_int(fma(a.zmul, xd, old), a.eta, floored);
  v[1] = lam_floor_int(fma(-a.zmul, xd, old), a.eta, floored);
}
__device__ __forceinline__ double lam_floor(double v, const LamArgs &a, bool &bad, bool &floored) {
  if (a.eta > 0.0 && !(v >= a.eta)) {  // K + eta I has no eigenvalue below eta: rounding
    v = a.eta;
    floored = true;
  }
  bad |= !(v > 0.0);
  return v;
}
template <typename T>
__device__ __forceinline__ double lam_value(T x, bool w0, const LamArgs &a, bool &bad, bool &floored) {
  double v = fma(a.zmul, f2d_exact(x), a.eta);
  if (w0) v += a.dc;
  return lam_floor(v, a, bad, floored);
}
template <typename T>
__device__ __forceinline__ void lam_pair(T x, double old, bool w0, const LamArgs &a, double (&v)[2], bool &bad, bool &floored) {
  const double t = fma(a.zmul, f2d_exact(x), w0 ? a.dc : 0.0);
  v[0] = lam_floor(old + t, a, bad, floored), v[1] = lam_floor(old - t, a, bad, floored);
}
__device__ __forceinline__ void lam_flags(const LamArgs &a, bool bad, bool floored) {
  if (bad && a.status) atomicOr(a.status, (uint32_t)QK_STATUS_NOTPD);
  if (floored && a.status) atomicOr(a.status, (uint32_t)QK_STATUS_FLOOR);
}

// Data into the transform's precision, and back.
template <typename T, typename TIO>
__device__ __forceinline__ T widen(TIO v) {
  if constexpr (sizeof(T) == 8) return f2d_int(v);
  else return v;
}
template <typename TIO, typename T>
__device__ __forceinline__ TIO narrow(T v) {
  if constexpr (sizeof(TIO) == 4 && sizeof(T) == 8) return d2f_int(v);
  else return v;
}

// MLL spectral step of one frequency: adds to the quadratic form and to sum g, returns g.
__device__ __forceinline__ double mll_g(double Y, double lam, double inv_n, double &quad, double &gs) {
  double a;
  const double g = mll_step(Y * Y, inv_n, lam, a);
  quad += a;
  gs += g;
  return g;
}

// What is stored for a result v where `prev` is the value there (NET_ADD) or y's (NET_RESIDUAL).
__device__ __forceinline__ float op_value(float v, float prev, int op) {
  return op == NET_SET ? v : prev + v;  // residuals are formed by FP64 transforms
}
__device__ __forceinline__ float op_value(double v, float prev, int op) {
  if (op == NET_RESIDUAL) return d2f_int(f2d_int(prev) - v);
  const float f = d2f_int(v);
  return op == NET_SET ? f : prev + f;
}
__device__ __forceinline__ double op_value(double v, double prev, int op) {
  return op == NET_SET ? v : op == NET_ADD ? prev + v : prev - v;
}

// ------------------------------------------------------------ one CTA per vector
// The vector in shared memory, radix-16 rounds upwards, element e at e + (e >> 4).  FP64
// vectors are 96-bit integers (12 bytes each; an odd stride, conflict-free), or doubles where
// the exponent range asks for it.
template <typename V>
__device__ __forceinline__ V v_add(V a, V b) { return a + b; }
template <typename V>
__device__ __forceinline__ V v_sub(V a, V b) { return a - b; }
template <>
__device__ __forceinline__ I96 v_add<I96>(I96 a, I96 b) { return i96_add(a, b); }
template <>
__device__ __forceinline__ I96 v_sub<I96>(I96 a, I96 b) { return i96_sub(a, b); }

template <typename V, int R>
__device__ __forceinline__ void small_round(V *sm, int m, int b) {
  const int G = 1 << (m - R);
  for (int g = threadIdx.x; g < G; g += blockDim.x) {
    const int e0 = (g & ((1 << b) - 1)) | ((g >> b) << (b + R));
    V v[1 << R];
#pragma unroll
    for (int q = 0; q < (1 << R); ++q) {
      const int e = e0 | (q << b);
      v[q] = sm[e + (e >> 4)];
    }
#pragma unroll
    for (int h = 0; h < R; ++h)
#pragma unroll
      for (int q = 0; q < (1 << R); ++q)
        if (!(q & (1 << h))) {
          const V a = v[q], c = v[q | (1 << h)];
          v[q] = v_add(a, c), v[q | (1 << h)] = v_sub(a, c);
        }
#pragma unroll
    for (int q = 0; q < (1 << R); ++q) {
      const int e = e0 | (q << b);
      sm[e + (e >> 4)] = v[q];
    }
  }
  __syncthreads();
}
template <typename V>
__device__ __forceinline__ void small_rounds(V *sm, int m) {
  for (int b = 0; b < m; b += 4) {
    switch (m - b) {
      case 1: small_round<V, 1>(sm, m, b); break;
      case 2: small_round<V, 2>(sm, m, b); break;
      case 3: small_round<V, 3>(sm, m, b); break;
      default: small_round<V, 4>(sm, m, b); break;
    }
  }
}

// x[i] (element t + i NT, i < per) <- its WHT.  sm: net_small_smem bytes.
// KEEP: FP64 butterflies (eigenvalues).
template <typename T, int PER, bool KEEP = false>
__device__ __forceinline__ void small_wht(T (&x)[PER], int m, unsigned char *smem) {
  const int NT = blockDim.x, n = 1 << m, t = threadIdx.x;
  if constexpr (sizeof(T) == 4) {
    float *sm = reinterpret_cast<float *>(smem);
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const int e = t + i * NT;
      if (e < n) sm[e + (e >> 4)] = x[i];
    }
    __syncthreads();
    small_rounds<float>(sm, m);
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const int e = t + i * NT;
      if (e < n) x[i] = sm[e + (e >> 4)];
    }
    __syncthreads();
  } else {
    __shared__ uint32_t red[16];
    uint32_t E = 0, far;
    if constexpr (!KEEP) E = w96_exponent(x, [&](int i) { return t + i * NT < n; }, red, far);
    if (E) {
      I96 *sm = reinterpret_cast<I96 *>(smem);
#pragma unroll
      for (int i = 0; i < PER; ++i) {
        const int e = t + i * NT;
        if (e < n) sm[e + (e >> 4)] = i96_from(x[i], E);
      }
      __syncthreads();
      small_rounds<I96>(sm, m);
#pragma unroll
      for (int i = 0; i < PER; ++i) {
        const int e = t + i * NT;
        if (e < n) x[i] = i96_to(sm[e + (e >> 4)], E);
      }
    } else {
      double *sm = reinterpret_cast<double *>(smem);
#pragma unroll
      for (int i = 0; i < PER; ++i) {
        const int e = t + i * NT;
        if (e < n) sm[e + (e >> 4)] = x[i];
      }
      __syncthreads();
      small_rounds<double>(sm, m);
#pragma unroll
      for (int i = 0; i < PER; ++i) {
        const int e = t + i * NT;
        if (e < n) x[i] = sm[e + (e >> 4)];
      }
    }
    __syncthreads();
  }
}

template <typename T>
static size_t net_small_smem(uint32_t m) {
  const size_t n = (size_t)1 << m;
  return (n + (n >> 4) + 1) * (sizeof(T) == 8 ? sizeof(I96) : sizeof(float));
}
// Threads: 16 elements each (one radix-16 group), at least a warp; FP32 tiles of 2^13 take 512.
static unsigned net_small_threads(uint32_t m) {
  const unsigned nt = m > 4 ? 1u << (m - 4) : 1u;
  return nt < 32u ? 32u : nt;
}

template <typename T>
__global__ void __launch_bounds__(sizeof(T) == 8 ? 256 : 512) k_net_eigs_small(const T *__restrict__ col,
                                                                               const double *__restrict__ old,
                                                                               double *__restrict__ lam, int m, LamArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int NT = blockDim.x, n = 1 << m, t = threadIdx.x;
  const uint64_t off = (uint64_t)blockIdx.x << m;
  T x[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) x[i] = t + i * NT < n ? col[off + t + i * NT] : T(0);
  small_wht<T, 16, true>(x, m, smem);
  bool rare = t == 0 || !(a.eta > 0.0), bad = false, floored = false;  // t == 0: w = 0
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const int e = t + i * NT;
    if (e >= n) continue;
    if (old) {
      double v[2];
      lam_pair_fast(x[i], old[off + e], a, v, rare, floored);
      lam[2 * off + e] = v[0], lam[2 * off + n + e] = v[1];
    } else {
      lam[off + e] = lam_fast(x[i], a, rare, floored);
    }
  }
  if (!rare) {
    lam_flags(a, false, floored);
    return;
  }
  floored = false;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const int e = t + i * NT;
    if (e >= n) continue;
    if (old) {
      double v[2];
      lam_pair(x[i], old[off + e], e == 0, a, v, bad, floored);
      lam[2 * off + e] = v[0], lam[2 * off + n + e] = v[1];
    } else {
      lam[off + e] = lam_value(x[i], e == 0, a, bad, floored);
    }
  }
  lam_flags(a, bad, floored);
}

// out <- op(H (H in (.) lambda^-+1) / n), core precision T.
template <typename T, typename TIO>
__global__ void __launch_bounds__(sizeof(T) == 8 ? 256 : 512) k_net_apply_small(const TIO *in, const TIO *y, TIO *out,
                                                                                const double *__restrict__ lam, int m,
                                                                                uint32_t nrhs, int inverse, int op) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int NT = blockDim.x, n = 1 << m, t = threadIdx.x;
  const uint64_t off = (uint64_t)blockIdx.x << m;
  const double *lr = lam + ((uint64_t)(blockIdx.x / nrhs) << m);
  const double fac = 1.0 / (double)n;
  T x[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) x[i] = t + i * NT < n ? widen<T>(in[off + t + i * NT]) : T(0);
  small_wht<T, 16>(x, m, smem);
#pragma unroll
  for (int i = 0; i < 16; ++i)
    if (t + i * NT < n) x[i] = scale_lambda(x[i], lr[t + i * NT], fac, inverse != 0);
  small_wht<T, 16>(x, m, smem);
#pragma unroll
  for (int i = 0; i < 16; ++i)
    if (t + i * NT < n) {
      const uint64_t j = off + t + i * NT;
      out[j] = op_value(x[i], op == NET_SET ? TIO(0) : op == NET_ADD ? out[j] : y[j], op);
    }
}

// The MLL's transforms: quadratic form, sum g and sum y (one partial sum per vector), u = H g.
template <typename T, typename TIO>
__global__ void __launch_bounds__(sizeof(T) == 8 ? 256 : 512) k_net_mll_small(const TIO *__restrict__ y, const double *__restrict__ lam,
                                                                              int m, uint32_t nrhs, double *__restrict__ part,
                                                                              double *__restrict__ ysum, TIO *__restrict__ u) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double sh[32];
  const int NT = blockDim.x, n = 1 << m, t = threadIdx.x;
  const uint64_t off = (uint64_t)blockIdx.x << m;
  const double *lr = lam + ((uint64_t)(blockIdx.x / nrhs) << m);
  const double inv_n = 1.0 / (double)n;
  T x[16];
  double sd = 0.0;  // FP32 data: their sum (one FP64 addition each; the conversion is integer)
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const TIO v = t + i * NT < n ? y[off + t + i * NT] : TIO(0);
    x[i] = widen<T>(v);
    if constexpr (sizeof(TIO) == 4) sd += f2d_int(v);
  }
  small_wht<T, 16>(x, m, smem);
  if constexpr (sizeof(TIO) == 4) sd = block_sum(sd, sh);
  else sd = x[0];  // element 0 of the transform (thread 0): the sum rounded once
  if (t == 0) ysum[blockIdx.x] = sd;
  double quad = 0.0, gs = 0.0;
#pragma unroll
  for (int i = 0; i < 16; ++i)
    if (t + i * NT < n) x[i] = narrow<T>(mll_g(f2d_int(x[i]), lr[t + i * NT], inv_n, quad, gs));
  quad = block_sum(quad, sh);
  gs = block_sum(gs, sh);
  if (t == 0) part[2 * blockIdx.x] = quad, part[2 * blockIdx.x + 1] = gs;
  if (!u) return;
  small_wht<T, 16>(x, m, smem);
#pragma unroll
  for (int i = 0; i < 16; ++i)
    if (t + i * NT < n) u[off + t + i * NT] = narrow<TIO>(x[i]);
}

// --------------------------------------------------------------- two tile passes
// FP32 low bits upwards from bit 0, layout L0 in and out (three transposes).
__device__ __forceinline__ void xwht_full_up(float (&v)[32], float *sm) {
  xw_L0_to_L1w(v, sm);
  reg_stages<float>(v, 0, 0, 5);
  xw_L1w_to_L2(v, sm);
  reg_stages<float>(v, 5, 5, 8);
  xw_L2_to_L1w(v, sm);
  xw_L1w_to_L0(v, sm);
  reg_stages<float>(v, 8, 8, 13);
}

__device__ __forceinline__ void xwht_full_up(double (&v)[16], double *sm) {
  xpose<double>(v, sm, 0, 1);
  reg_stages<double>(v, 0, 0, 4);
  xpose<double>(v, sm, 1, 2);
  reg_stages<double>(v, 4, 4, 8);
  xpose<double>(v, sm, 2, 0);
  reg_stages<double>(v, 8, 8, 12);
}

// UP: bits upwards in FP64 / FP32 butterflies (all FP32 transforms, and FP64 ones of first
// columns); otherwise integers, whose order does not matter.
template <typename T, bool KEEP> constexpr bool kUp = sizeof(T) == 4 || KEEP;

template <typename T, typename TIO, bool KEEP>
__global__ void __launch_bounds__(kFNT, sizeof(T) == 8 ? 3 : 4) k_net_low_in(const TIO *in, T *X,
                                                                             double *__restrict__ ysum) {
  constexpr int LOGT = FCfg<T>::LOGT, L = FCfg<T>::L;
  extern __shared__ __align__(16) unsigned char smem[];
  T *sm = reinterpret_cast<T *>(smem);
  const uint64_t base = (uint64_t)blockIdx.x << LOGT;
  const int t = threadIdx.x;
  T v[L];
  double s = 0.0;
#pragma unroll
  for (int l = 0; l < L; ++l) {
    const TIO a = in[base + t + (l << kLOGNT)];
    v[l] = widen<T>(a);
    if constexpr (sizeof(TIO) == 4)
      if (ysum) s += f2d_int(a);
  }
  if constexpr (sizeof(TIO) == 4) {
    if (ysum) {
      __shared__ double sh[32];
      const double sd = block_sum(s, sh);
      if (t == 0) ysum[blockIdx.x] = sd;
    }
  }
  if constexpr (kUp<T, KEEP>) xwht_full_up(v, sm);
  else xwht_full<T>(v, sm, 0);
  if (sizeof(TIO) == 8 && ysum && t == 0) ysum[blockIdx.x] = f2d_exact(v[0]);  // element 0: the tile's sum
#pragma unroll
  for (int l = 0; l < L; ++l) X[base + e_of<T>(kUp<T, KEEP> ? 0 : 2, t, l)] = v[l];
}

template <typename T, typename TIO>
__global__ void __launch_bounds__(kFNT, 3) k_net_low_out(const T *X, const TIO *y, TIO *out, int op) {
  constexpr int LOGT = FCfg<T>::LOGT, L = FCfg<T>::L;
  extern __shared__ __align__(16) unsigned char smem[];
  T *sm = reinterpret_cast<T *>(smem);
  const uint64_t base = (uint64_t)blockIdx.x << LOGT;
  const int t = threadIdx.x;
  T v[L];
#pragma unroll
  for (int l = 0; l < L; ++l) v[l] = X[base + t + (l << kLOGNT)];
  TIO prev[L];  // read before the transform where the registers allow (FP32 data)
  const TIO *src = op == NET_ADD ? out : y;
#pragma unroll
  for (int l = 0; l < L; ++l) prev[l] = sizeof(TIO) == 4 && op != NET_SET ? src[base + e_of<T>(2, t, l)] : TIO(0);
  xwht_full<T>(v, sm, 0);
  if (sizeof(TIO) == 8 && op != NET_SET) {
#pragma unroll
    for (int l = 0; l < L; ++l) prev[l] = src[base + e_of<T>(2, t, l)];
  }
#pragma unroll
  for (int l = 0; l < L; ++l) out[base + e_of<T>(2, t, l)] = op_value(v[l], prev[l], op);
}

// The high bits of one column tile with the operation on the transform's values inside.
enum { MID_EIGS = 0, MID_APPLY = 1, MID_MLL = 2, MID_STORE = 3, MID_EXTEND = 4 };
struct MidArgs {
  int m, c;              // c: contiguous column bits (2 LOGT - m)
  uint32_t nrhs;
  int inverse;           // APPLY: by 1 / lambda (1) or lambda (0)
  int back;              // MLL: inverse high bits of g (FP64 transforms); 0: g is stored as it is
  const double *lam;     // APPLY, MLL: eigenvalues; EXTEND: those of the first half
  double *lam_out, *part;
  LamArgs la;
};
// The eigenvalues a tile needs (EXTEND, APPLY, MLL) are copied to shared memory asynchronously
// behind the transform tile while the transform runs, each thread reading back what it copied:
// loaded into registers four or eight at a time the kernel waited on them (long_scoreboard 13
// per issue; 32 x 2^19 doubling: 164 us, now 145).
template <typename T, int MODE>
constexpr size_t mid_smem() {
  return xtile_bytes<T>() + (MODE == 4 || MODE == 1 || MODE == 2 ? sizeof(double) << FCfg<T>::LOGT : 0);
}
template <typename T, typename TIO, int MODE>
__global__ void __launch_bounds__(kFNT, MODE == 0 || MODE == 3 ? 3 : 2) k_net_mid(T *X, TIO *out, MidArgs a) {
  constexpr int LOGT = FCfg<T>::LOGT, L = FCfg<T>::L;
  constexpr bool KEEP = MODE == MID_EIGS || MODE == MID_EXTEND, UP = kUp<T, KEEP>;
  constexpr int LIN = UP ? 2 : 0, LMID = 2 - LIN, DF = UP ? 1 : 0;  // bits upwards: L2 then L0
  extern __shared__ __align__(16) unsigned char smem[];
  T *sm = reinterpret_cast<T *>(smem);
  const int t = threadIdx.x, c = a.c;
  const uint32_t tau = blockIdx.x, v = blockIdx.y, tcol = tau << c;
  const uint64_t n = 1ull << a.m;
  auto widx = [&](uint32_t e) -> uint32_t { return ((e >> c) << LOGT) | tcol | (e & ((1u << c) - 1)); };
  T *xv = X + (uint64_t)v * n;
  T x[L];
#pragma unroll
  for (int l = 0; l < L; ++l) x[l] = xv[widx(e_of<T>(LIN, t, l))];
  // with_lam(f): f(l, w, lambda_w) for every element of layout LMID
  constexpr bool NEEDS = MODE == MID_EXTEND || MODE == MID_APPLY || MODE == MID_MLL;
  const double *lr = NEEDS ? a.lam + (uint64_t)(MODE == MID_EXTEND ? v : v / a.nrhs) * n : nullptr;
  double *sl = reinterpret_cast<double *>(smem + xtile_bytes<T>());  // element (t, l) at t + 256 l
  if constexpr (NEEDS) {
#pragma unroll
    for (int l = 0; l < L; ++l) cp_async8(&sl[t + (l << kLOGNT)], &lr[widx(e_of<T>(LMID, t, l))]);
  }
  auto with_lam = [&](auto f) {
    cp_async_wait();
#pragma unroll
    for (int l = 0; l < L; ++l) f(l, widx(e_of<T>(LMID, t, l)), sl[t + (l << kLOGNT)]);
  };
  if constexpr (KEEP) xwht_col_fp<T>(x, sm, c, DF);  // LIN -> LMID
  else xwht_col<T>(x, sm, c, DF);
  if constexpr (MODE == MID_EIGS) {
    double *dst = a.lam_out + (uint64_t)v * n;
    bool rare = (tau == 0 && t == 0) || !(a.la.eta > 0.0);  // w = 0: element 0 of every layout
    bool bad = false, floored = false;
#pragma unroll
    for (int l = 0; l < L; ++l) dst[widx(e_of<T>(LMID, t, l))] = lam_fast(x[l], a.la, rare, floored);
    if (rare) {  // through the thread's own slots of the tile: a rolled loop, no registers held for it
      floored = false;
#pragma unroll
      for (int l = 0; l < L; ++l) sm[t + (l << kLOGNT)] = x[l];
#pragma unroll 1
      for (int l = 0; l < L; ++l) {
        const uint32_t w = widx(e_of<T>(LMID, t, l));
        dst[w] = lam_value(sm[t + (l << kLOGNT)], w == 0, a.la, bad, floored);
      }
    }
    lam_flags(a.la, bad, floored);
  } else if constexpr (MODE == MID_EXTEND) {
    double *dst = a.lam_out + (uint64_t)v * 2 * n;
    bool rare = (tau == 0 && t == 0) || !(a.la.eta > 0.0), bad = false, floored = false;
    with_lam([&](int l, uint32_t w, double old) {
      double p[2];
      lam_pair_fast(x[l], old, a.la, p, rare, floored);
      dst[w] = p[0], dst[n + w] = p[1];
    });
    if (rare) {
      floored = false;
#pragma unroll
      for (int l = 0; l < L; ++l) sm[t + (l << kLOGNT)] = x[l];
#pragma unroll 1
      for (int l = 0; l < L; ++l) {
        const uint32_t w = widx(e_of<T>(LMID, t, l));
        double p[2];
        lam_pair(sm[t + (l << kLOGNT)], lr[w], w == 0, a.la, p, bad, floored);
        dst[w] = p[0], dst[n + w] = p[1];
      }
    }
    lam_flags(a.la, bad, floored);
  } else if constexpr (MODE == MID_APPLY) {
    const double fac = 1.0 / (double)n;
    with_lam([&](int l, uint32_t, double lam) { x[l] = scale_lambda(x[l], lam, fac, a.inverse != 0); });
    xwht_col<T>(x, sm, c, 1 - DF);
#pragma unroll
    for (int l = 0; l < L; ++l) xv[widx(e_of<T>(LIN, t, l))] = x[l];
  } else if constexpr (MODE == MID_MLL) {
    __shared__ double sh[32];
    const double inv_n = 1.0 / (double)n;
    double quad = 0.0, gs = 0.0;
    with_lam([&](int l, uint32_t, double lam) { x[l] = narrow<T>(mll_g(f2d_int(x[l]), lam, inv_n, quad, gs)); });
    if (a.back) xwht_col<T>(x, sm, c, 1 - DF);
#pragma unroll
    for (int l = 0; l < L; ++l) xv[widx(a.back ? e_of<T>(LIN, t, l) : e_of<T>(LMID, t, l))] = x[l];
    quad = block_sum(quad, sh);
    gs = block_sum(gs, sh);
    if (t == 0) {
      a.part[((uint64_t)v * gridDim.x + tau) * 2] = quad;
      a.part[((uint64_t)v * gridDim.x + tau) * 2 + 1] = gs;
    }
  } else {
#pragma unroll
    for (int l = 0; l < L; ++l) out[(uint64_t)v * n + widx(e_of<T>(LMID, t, l))] = (TIO)x[l];
  }
}

// ------------------------------------------------------------------ host side
template <typename T>
static bool one_tile(uint32_t m) { return (int)m <= FCfg<T>::LOGT; }
template <typename T>
static bool two_pass(uint32_t m) { return (int)m > FCfg<T>::LOGT && (int)m <= two_pass_max_m<T>(); }

bool net_ops_supported(uint32_t m, uint64_t nvec, bool fp64) {
  const uint32_t top = (uint32_t)(fp64 ? two_pass_max_m<double>() : two_pass_max_m<float>());
  return m <= top && nvec <= 65535;
}

template <typename T>
static unsigned tiles_of(uint32_t m) { return 1u << (m - FCfg<T>::LOGT); }

uint32_t net_mll_blocks(uint32_t m, bool fp64) {
  if (fp64) return one_tile<double>(m) ? 1u : tiles_of<double>(m);
  return one_tile<float>(m) ? 1u : tiles_of<float>(m);
}

template <typename T, typename TIO, int MODE>
static int launch_mid(T *X, TIO *out, uint32_t m, uint32_t nvec, MidArgs a, cudaStream_t st) {
  a.m = (int)m, a.c = 2 * FCfg<T>::LOGT - (int)m;
  constexpr size_t sm = mid_smem<T, MODE>();
  smem_optin<k_net_mid<T, TIO, MODE>>(sm);
  k_net_mid<T, TIO, MODE><<<dim3(tiles_of<T>(m), nvec), kFNT, sm, st>>>(X, out, a);
  return check_launch("net transform: high bits");
}
template <typename T, typename TIO, bool KEEP = false>
static int launch_low_in(const TIO *in, T *X, uint32_t m, uint32_t nvec, double *ysum, cudaStream_t st) {
  smem_optin<k_net_low_in<T, TIO, KEEP>>(xtile_bytes<T>());
  k_net_low_in<T, TIO, KEEP><<<tiles_of<T>(m) * nvec, kFNT, xtile_bytes<T>(), st>>>(in, X, ysum);
  return check_launch("net transform: low bits");
}

template <typename T>
int net_eigs(uint32_t m, uint32_t batch, const T *col, T *X, double zmul, double dc, double eta, const double *old,
             double *lam, uint32_t *status, cudaStream_t st) {
  const LamArgs la{zmul, dc, eta, status};
  if (one_tile<T>(m)) {
    const size_t sm = net_small_smem<T>(m);
    smem_optin<k_net_eigs_small<T>>(sm);
    k_net_eigs_small<T><<<batch, net_small_threads(m), sm, st>>>(col, old, lam, (int)m, la);
    return check_launch("net eigenvalues");
  }
  int rc = launch_low_in<T, T, true>(col, X, m, batch, nullptr, st);
  if (rc) return rc;
  MidArgs a{};
  a.nrhs = 1, a.lam = old, a.lam_out = lam, a.la = la;
  if (old) return launch_mid<T, T, MID_EXTEND>(X, nullptr, m, batch, a, st);
  return launch_mid<T, T, MID_EIGS>(X, nullptr, m, batch, a, st);
}

template <typename T, typename TIO>
int net_apply(uint32_t m, uint32_t nvec, uint32_t nrhs, const double *lam, const TIO *in, const TIO *y, TIO *out, T *X,
              int inverse, int op, cudaStream_t st) {
  if (one_tile<T>(m)) {
    const size_t sm = net_small_smem<T>(m);
    smem_optin<k_net_apply_small<T, TIO>>(sm);
    k_net_apply_small<T, TIO><<<nvec, net_small_threads(m), sm, st>>>(in, y, out, lam, (int)m, nrhs, inverse, op);
    return check_launch("net solve");
  }
  int rc = launch_low_in<T, TIO>(in, X, m, nvec, nullptr, st);
  if (rc) return rc;
  MidArgs a{};
  a.nrhs = nrhs, a.lam = lam, a.inverse = inverse;
  if ((rc = launch_mid<T, TIO, MID_APPLY>(X, nullptr, m, nvec, a, st))) return rc;
  smem_optin<k_net_low_out<T, TIO>>(xtile_bytes<T>());
  k_net_low_out<T, TIO><<<tiles_of<T>(m) * nvec, kFNT, xtile_bytes<T>(), st>>>(X, y, out, op);
  return check_launch("net solve: low bits");
}

template <typename T, typename TIO>
int net_mll(uint32_t m, uint32_t nvec, uint32_t nrhs, const double *lam, const TIO *y, T *X, double *part, double *ysum,
            TIO *u, cudaStream_t st) {
  if (one_tile<T>(m)) {
    const size_t sm = net_small_smem<T>(m);
    smem_optin<k_net_mll_small<T, TIO>>(sm);
    k_net_mll_small<T, TIO><<<nvec, net_small_threads(m), sm, st>>>(y, lam, (int)m, nrhs, part, ysum, u);
    return check_launch("net MLL");
  }
  int rc = launch_low_in<T, TIO>(y, X, m, nvec, ysum, st);
  if (rc) return rc;
  MidArgs a{};
  a.nrhs = nrhs, a.lam = lam, a.part = part, a.back = sizeof(T) == 8;
  if ((rc = launch_mid<T, TIO, MID_MLL>(X, nullptr, m, nvec, a, st)) || !u) return rc;
  if constexpr (sizeof(T) == 8) {
    smem_optin<k_net_low_out<T, TIO>>(xtile_bytes<T>());
    k_net_low_out<T, TIO><<<tiles_of<T>(m) * nvec, kFNT, xtile_bytes<T>(), st>>>(X, nullptr, u, NET_SET);
    return check_launch("net MLL: low bits");
  } else {
    // FP32: the adjoint transform upwards from bit 0, as the multi-pass transform rounds it
    if ((rc = launch_low_in<T, T>(X, X, m, nvec, nullptr, st))) return rc;
    return launch_mid<T, TIO, MID_STORE>(X, u, m, nvec, MidArgs{}, st);
  }
}

template int net_eigs<float>(uint32_t, uint32_t, const float *, float *, double, double, double, const double *, double *, uint32_t *, cudaStream_t);
template int net_eigs<double>(uint32_t, uint32_t, const double *, double *, double, double, double, const double *, double *, uint32_t *, cudaStream_t);
#define QK_NET_T(T, TIO)                                                                                              \
  template int net_apply<T, TIO>(uint32_t, uint32_t, uint32_t, const double *, const TIO *, const TIO *, TIO *, T *, int, \
                                 int, cudaStream_t);                                                                   \
  template int net_mll<T, TIO>(uint32_t, uint32_t, uint32_t, const double *, const TIO *, T *, double *, double *, TIO *, \
                               cudaStream_t);
QK_NET_T(float, float)
QK_NET_T(double, double)
QK_NET_T(double, float)

}  // namespace qk
