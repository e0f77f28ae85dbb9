// FP64 gradient sweep shared by the vectors of one first column (arXiv 2502.14256, Sec. 5.4,
// adjoint of the eigenvalue map).  All right-hand sides of a net's randomization, and all
// shifts and right-hand sides of a lattice (whose differences do not depend on the shift),
// run over the same factors:
//   su[v][j] = sum_i u_v[i] dk1_i/dc_j,   s1[j] = sum_i dk1_i/dc_j,
//   dk1_i/dc_j = k1_i q_ij,  q_ij = K_ij / (1 + c_j K_ij).
//
// Bound: FP64 issue (GB300: about 2 FP64 lanes per SM and cycle; 32 integer or 57 FP32
// instructions issue in the time of one FP64 instruction).  So the sweep spends FP64 instructions on the
// factors and the sums only: a thread owns one dimension j and walks over points, so its sums
// stay in registers and no FP64 shuffles are needed; q_ij is formed once for up to 16
// vectors (5 FP64 instructions at DSI order 2, then one fma per vector and one for s1: 14 at
// 8 vectors, where the sweep of one vector at a time spent 8 x 10 and its warp sums); words
// become doubles by integer operations.  Nets of 2^14 to 2^17 points, d = 16, 8 right-hand
// sides: 8470 us inside phase C, 1152 us shared, 995 us with the quotient in three FP64
// instructions instead of four (FP64 pipe 92 % busy).
#pragma once

#include "qk_column.cuh"

namespace qk {

constexpr int kGradNT = 256;
constexpr int kGradMaxNV = 16;    // vectors per pass over the factors
constexpr uint32_t kGradSP = 256;  // points staged in shared memory per step (fixed: the order of a
                                   // thread's additions does not depend on the number of vectors)

// log2 of the points of one CTA: 256 CTAs per randomization where n allows it (a CTA's FP64
// work takes tens of microseconds, so a nearly empty last wave shows), 128 to 1024 points.
// A function of m alone, so that every schedule forms the same partial sums.
__host__ __device__ inline uint32_t grad64_log_points(uint32_t m) {
  return m <= 15 ? 7u : (m >= 18 ? 10u : m - 8u);
}
__host__ __device__ inline uint32_t grad64_points(uint32_t m) {
  const uint32_t lg = grad64_log_points(m);
  return 1u << (m < lg ? m : lg);
}
__host__ __device__ inline uint32_t grad64_blocks(uint32_t m) { return (uint32_t)((1ull << m) / grad64_points(m)); }

// Smallest power of two >= min(nvec, kGradMaxNV): the instantiation that takes nvec vectors.
inline uint32_t grad64_nv(uint64_t nvec) {
  uint32_t v = 1;
  while (v < nvec && v < (uint32_t)kGradMaxNV) v *= 2;
  return v;
}

// Difference words: 32 digits (FAM 0: DSI nets; 1: SI lattices) or 64 (FAM 2: interlaced nets).
template <int FAM> struct GradWord { using type = uint32_t; };
template <> struct GradWord<2> { using type = uint64_t; };

__host__ __device__ inline size_t grad64_tab_bytes(uint32_t d, uint32_t m) {  // weights, factor rows, two word tables
  const uint32_t hi = (grad64_points(m) + 31) / 32;
  return weights_bytes(d) + dsi_tab_bytes<double>() + ((size_t)(32 + hi) * d * sizeof(uint64_t) + 15 & ~(size_t)15);
}
inline size_t grad64_smem(uint32_t d, uint32_t m, uint32_t nv) {
  static_assert(kGradSP == kGradNT, "the staged values and the group sums share one region");
  return grad64_tab_bytes(d, m) + sizeof(double) * (size_t)kGradNT * (nv + 1);
}

// Order-alpha DSI factor at x = Z 2^-64 from rows keyed by clz64(Z) (0..64; 64 is Z = 0), the
// Theorem's coefficients as polynomials in x: order 2 (A, B): A + B x; order 3 (A, B, C);
// order 4 (A, B, C, D) and E S'(Z), S' from the top 21 digits.  8 doubles per row.
constexpr int kHoRows = 65, kHoNC = 8;
struct DsiTable64 { double v[kHoRows * kHoNC]; };
static_assert(sizeof(DsiTable64) <= (kTabRows * kTabNC + kOctRows) * sizeof(double), "rows fit the shared table region");
template <int ALPHA>
__host__ __device__ constexpr DsiTable64 make_dsi_table64() {
  DsiTable64 tab{};
  for (int q = 0; q < kHoRows; ++q) {
    const double b = q < 64 ? q + 1.0 : 0.0, t1 = q < 64 ? pow2neg(q + 1) : 0.0, t2 = t1 * t1, t3 = t2 * t1;
    double *r = tab.v + q * kHoNC;
    if (ALPHA == 1) {
      r[0] = q < 64 ? 1.0 - 3.0 * t1 : 1.0;
    } else if (ALPHA == 2) {
      r[0] = 1.5 - 2.5 * t1, r[1] = -b;
    } else if (ALPHA == 3) {
      r[0] = -1.0 + (43.0 / 18.0) * (1.0 - t2), r[1] = -5.0 * (1.0 - t1), r[2] = b;
    } else {
      r[0] = -1.0 + (701.0 / 294.0) * (1.0 - t3), r[1] = -(43.0 / 9.0) * (1.0 - t2), r[2] = 5.0 * (1.0 - t1);
      r[3] = -(2.0 / 3.0) * b, r[4] = -b / 24.0;
    }
  }
  return tab;
}
static __device__ const DsiTable64 g_dsi_d64[4] = {make_dsi_table64<1>(), make_dsi_table64<2>(), make_dsi_table64<3>(),
                                                   make_dsi_table64<4>()};

template <int ALPHA>
__device__ __forceinline__ double dsi_tab_eval64(const double *tab, uint64_t Z) {
  const double *row = tab + __clzll((long long)Z) * kHoNC;
  const double2 r0 = *reinterpret_cast<const double2 *>(row);
  if constexpr (ALPHA == 1) return r0.x;
  const double x = u64_to_double(Z, 64);
  if constexpr (ALPHA == 2) return fma(r0.y, x, r0.x);
  const double2 r1 = *reinterpret_cast<const double2 *>(row + 2);
  if constexpr (ALPHA == 3) return fma(fma(r1.x, x, r0.y), x, r0.x);
  // S' 2^60 = octal digits a = 0 .. 20 of the word's leading bits as one 63-bit integer
  const uint32_t zh = (uint32_t)(Z >> 32);
  const uint32_t t11 = (zh >> 11) & 0x7FFu;
  const uint64_t oct = ((uint64_t)spread3_10(zh >> 22) << 33) | ((uint64_t)(t11 >> 10) << 30) | spread3_10(t11);
  return fma(row[4], u64_to_double(oct, 60), fma(fma(fma(r1.y, x, r1.x), x, r0.y), x, r0.x));
}

// Tables of one CTA: zlo[x][j] (the low 5 position bits) and zhi[x][j] (the others), so that
// neighbouring threads (dimensions) read neighbouring words.
template <int FAM, int ALPHA>
struct GradTables {
  using W = typename GradWord<FAM>::type;
  double *w;
  DiffTables tb;
  W *zlo, *zhi;
  const uint32_t *g;
  uint32_t d, base;
  __device__ __forceinline__ W word(uint32_t i, uint32_t j) const {
    if constexpr (FAM == 1) return __brev(base + i) * g[j];
    else return zhi[(i >> 5) * d + j] ^ zlo[(i & 31) * d + j];
  }
  __device__ __forceinline__ double factor(W z) const {
    if constexpr (FAM == 2) return dsi_tab_eval64<ALPHA>(reinterpret_cast<const double *>(tb.ktab), z);
    else return kfac<double, FAM, ALPHA>(tb, z);
  }
  // columns: this randomization's generator columns (nets)
  __device__ __forceinline__ void build(const ColJob &job, const W *columns, uint32_t base_, uint32_t cnt,
                                        unsigned char *smem) {
    d = job.d, base = base_, g = job.g;
    w = reinterpret_cast<double *>(smem);
    tb.ktab = smem + weights_bytes(d);
    zlo = reinterpret_cast<W *>(smem + weights_bytes(d) + dsi_tab_bytes<double>());
    zhi = zlo + 32 * d;
    const uint32_t t = threadIdx.x;
    for (uint32_t q = t; q < d; q += kGradNT) w[q] = job.w[q];
    if constexpr (FAM != 1) {
      const uint32_t nhi = (cnt + 31) >> 5;
      for (uint32_t q = t; q < (32 + nhi) * d; q += kGradNT) {
        const uint32_t x = q / d, j = q - x * d;
        const uint32_t v = order_map(job.order, x < 32 ? x : base + ((x - 32) << 5));
        W acc = 0;
#pragma unroll
        for (int k = 0; k < 32; ++k)  // independent loads
          if ((v >> k) & 1u) acc ^= columns[j * 32 + k];
        zlo[q] = acc;  // zhi follows zlo
      }
      double *tab = reinterpret_cast<double *>(tb.ktab);
      if constexpr (FAM == 0) {
        build_dsi_tab<double, ALPHA>(tab);
      } else {
        for (uint32_t q = t; q < kHoRows * kHoNC; q += kGradNT) tab[q] = g_dsi_d64[ALPHA - 1].v[q];
      }
    }
  }
};

// Points base .. base + cnt - 1 of one randomization, vectors 0 .. nva - 1 (nva <= NV): u(v, i)
// returns u_v at point base + i; pcol: the column in form P at base, or nullptr (formed here,
// once for all vectors); dst + v dstride receives the 2 d partial sums of vector v.  Every
// thread of the CTA (kGradNT) calls it.
template <int FAM, int ALPHA, int NV, typename UF>
__device__ __forceinline__ void grad64_item(const ColJob &job, const typename GradWord<FAM>::type *columns, uint32_t base,
                                            uint32_t cnt, uint32_t nva, UF u, const double *pcol, double *dst,
                                            size_t dstride, unsigned char *smem) {
  constexpr uint32_t SP = kGradSP;
  const uint32_t d = job.d, t = threadIdx.x;
  GradTables<FAM, ALPHA> T;
  T.build(job, columns, base, cnt, smem);
  double *stage = reinterpret_cast<double *>(smem + grad64_tab_bytes(d, job.m));  // [SP][NV] u k1
  double *k1s = stage + SP * NV;                                                  // [SP]
  const uint32_t G = kGradNT / d, grp = t / d, j = t - grp * d;
  double su[NV], s1 = 0.0;
#pragma unroll
  for (int v = 0; v < NV; ++v) su[v] = 0.0;
  for (uint32_t s0 = 0; s0 < cnt; s0 += SP) {
    const uint32_t sc = cnt - s0 < SP ? cnt - s0 : SP;
    __syncthreads();  // tables built / the previous step's staged values read
    for (uint32_t i = t; i < sc; i += kGradNT) {
      double p;
      if (pcol) {
        p = __ldcg(pcol + s0 + i);
      } else {
        p = 0.0;
        for (uint32_t jj = 0; jj < d; ++jj) p = pm1_step(p, T.w[jj] * T.factor(T.word(s0 + i, jj)));
      }
      const double k1 = fma(job.zeta, p, job.zeta);
      k1s[i] = k1;
#pragma unroll
      for (uint32_t v = 0; v < (uint32_t)NV; ++v) stage[i * NV + v] = v < nva ? u(v, s0 + i) * k1 : 0.0;
    }
    __syncthreads();
    if (grp < G) {
      const double wj = T.w[j];
#pragma unroll 2
      for (uint32_t i = grp; i < sc; i += G) {
        const double K = T.factor(T.word(s0 + i, j));
        const double f = fma(wj, K, 1.0);
        double q;
        if (!ratio_lean(K, f, q) && !ratio_fast(K, f, q)) {
          if (f == 0.0) {  // the explicit product over the other dimensions; k1 = 0 here
            double dk = job.zeta;
            for (uint32_t jj = 0; jj < d; ++jj) {
              const double Kj = T.factor(T.word(s0 + i, jj));
              dk *= jj == j ? Kj : fma(T.w[jj], Kj, 1.0);
            }
            s1 += dk;
#pragma unroll
            for (uint32_t v = 0; v < (uint32_t)NV; ++v)
              if (v < nva) su[v] = fma(u(v, s0 + i), dk, su[v]);
            continue;
          }
          q = K / f;
        }
        s1 = fma(k1s[i], q, s1);
#pragma unroll
        for (int v = 0; v < NV; ++v) su[v] = fma(stage[i * NV + v], q, su[v]);
      }
    }
  }
  __syncthreads();
  double *red = stage;  // [NV + 1][G][d]
  if (grp < G) {
#pragma unroll
    for (int v = 0; v < NV; ++v) red[(v * G + grp) * d + j] = su[v];
    red[(NV * G + grp) * d + j] = s1;
  }
  __syncthreads();
  // The G = 256 / d groups' sums in pairs, eight at a time into two chains: one chain over all of
  // them was up to twice as far from the exact sum (d = 4, G = 64) and a dependent addition per
  // group; pairs through shared memory, a barrier per level, cost 2 % at 8 vectors and d = 16.
  auto eight = [&](const double *r, uint32_t g0) {
    double x[8];
#pragma unroll
    for (uint32_t k = 0; k < 8; ++k) x[k] = g0 + k < G ? r[(g0 + k) * d] : 0.0;
    return ((x[0] + x[1]) + (x[2] + x[3])) + ((x[4] + x[5]) + (x[6] + x[7]));
  };
  for (uint32_t q = t; q < (NV + 1) * d; q += kGradNT) {
    const uint32_t v = q / d, jj = q - v * d;
    if (v < (uint32_t)NV && v >= nva) continue;
    const double *r = red + v * G * d + jj;
    double s0 = eight(r, 0), s1 = G > 8 ? eight(r, 8) : 0.0;
    for (uint32_t g = 16; g < G; g += 16) {
      s0 += eight(r, g);
      if (g + 8 < G) s1 += eight(r, g + 8);
    }
    const double s = s0 + s1;
    if (v < (uint32_t)NV) dst[v * dstride + jj] = s;
    else
      for (uint32_t x = 0; x < nva; ++x) dst[x * dstride + d + jj] = s;
  }
  __syncthreads();  // the caller may reuse the shared memory
}

// One CTA: block blockIdx.x of the points, vectors v0 .. of chunk blockIdx.y, randomization
// blockIdx.z (SI: all vectors belong to the one point set, grid.z = 1).  With `pairs`, u is the
// pair layout of the lattice transforms: vector v is the real (v even) or imaginary (v odd)
// part of complex vector v / 2.  nper: vectors per column; part: (vectors, blocks, 2 d).
template <int FAM, int ALPHA, int NV>
__global__ void __launch_bounds__(kGradNT) k_grad64(ColJob job, const typename GradWord<FAM>::type *__restrict__ columns,
                                                    uint32_t nper, const double *__restrict__ u, int pairs,
                                                    const double *__restrict__ pcol, double *__restrict__ part) {
  extern __shared__ __align__(16) unsigned char smem[];
  const uint64_t n = 1ull << job.m;
  const uint32_t cnt = grad64_points(job.m), base = blockIdx.x * cnt, r = blockIdx.z;
  const uint32_t q0 = blockIdx.y * NV, nva = nper - q0 < (uint32_t)NV ? nper - q0 : (uint32_t)NV;
  const uint64_t v0 = (uint64_t)r * nper + q0;
  auto uget = [&](uint32_t v, uint32_t i) -> double {
    const uint64_t vv = v0 + v, ii = base + i;
    return u[pairs ? ((((vv >> 1) * n) + ii) << 1) + (vv & 1) : vv * n + ii];
  };
  grad64_item<FAM, ALPHA, NV>(job, FAM == 1 ? nullptr : columns + (size_t)r * job.d * 32, base, cnt, nva, uget,
                              pcol ? pcol + (uint64_t)r * n + base : nullptr,
                              part + (v0 * gridDim.x + blockIdx.x) * 2 * job.d, (size_t)gridDim.x * 2 * job.d, smem);
}

template <int FAM, int ALPHA, int NV>
static int launch_grad64_nv(const ColJob &job, const typename GradWord<FAM>::type *columns, uint32_t nset, uint32_t nper,
                            const double *u, int pairs, const double *pcol, double *part, cudaStream_t st) {
  const size_t smem = grad64_smem(job.d, job.m, NV);
  const uint32_t chunks = (nper + NV - 1) / NV;
  const uint64_t n = 1ull << job.m;
  if (chunks > 65535) return fail(QK_EINVAL, "gradient: too many vectors per point set");
  smem_optin<k_grad64<FAM, ALPHA, NV>>(smem);
  for (uint32_t r0 = 0; r0 < nset; r0 += 65535) {  // grid.z limit
    const uint32_t nr = nset - r0 < 65535 ? nset - r0 : 65535;
    const uint64_t v0 = (uint64_t)r0 * nper;  // pairs: one set only, v0 = 0
    k_grad64<FAM, ALPHA, NV><<<dim3(grad64_blocks(job.m), chunks, nr), kGradNT, smem, st>>>(
        job, columns ? columns + (size_t)r0 * job.d * 32 : nullptr, nper, u + v0 * n, pairs,
        pcol ? pcol + (uint64_t)r0 * n : nullptr, part + v0 * grad64_blocks(job.m) * 2 * job.d);
    int rc = check_launch("gradient partials (FP64)");
    if (rc) return rc;
  }
  return QK_OK;
}

// nset point sets of nper vectors each.
template <int FAM, int ALPHA>
static int launch_grad64(const ColJob &job, const typename GradWord<FAM>::type *columns, uint32_t nset, uint32_t nper,
                         const double *u, int pairs, const double *pcol, double *part, cudaStream_t st) {
  switch (grad64_nv(nper)) {
    case 1: return launch_grad64_nv<FAM, ALPHA, 1>(job, columns, nset, nper, u, pairs, pcol, part, st);
    case 2: return launch_grad64_nv<FAM, ALPHA, 2>(job, columns, nset, nper, u, pairs, pcol, part, st);
    case 4: return launch_grad64_nv<FAM, ALPHA, 4>(job, columns, nset, nper, u, pairs, pcol, part, st);
    case 8: return launch_grad64_nv<FAM, ALPHA, 8>(job, columns, nset, nper, u, pairs, pcol, part, st);
    default: return launch_grad64_nv<FAM, ALPHA, 16>(job, columns, nset, nper, u, pairs, pcol, part, st);
  }
}

}  // namespace qk
