// Point generation (arXiv 2502.14256, Sec. 4.2-4.3), first Gram columns
// (Sec. 5.4, k_1[i] = K(x_i, x_0)) and the gradient reductions that recompute
// the kernel factors instead of storing them.
//
// Digital nets: the point at sequence position i is
//   X_i = D (+) XOR_{bit k of h(i)} Ct[k],  h(i) = i (natural) or i ^ (i >> 1) (Gray),
// and h is linear over GF(2).  A CTA covers 2048 consecutive positions (columns of few tiles: 512
// or 1024)
// i = tile | (l << 8) | (warp << 5) | lane with disjoint bit fields, so
//   X_i (+) X_0 = Z(h(lane)) (+) Z(h(warp << 5)) (+) Z(h(tile | l << 8)),
// three small per-CTA tables in shared memory: each difference word costs one
// broadcast shared load and one XOR, and the outputs of a warp are contiguous.
// Lattices: X_i (-) X_0 = v(i) 2^32 g mod 2^32 = brev(i) * g (wrapping multiply).
#include <cstdio>

#include "qk_common.cuh"
#include "qk_factors.cuh"
#include "qk_internal.h"
#include "qk_column.cuh"
#include "qk_grad.cuh"

namespace qk {

constexpr int kNT = 256;  // threads per CTA
constexpr int kL = 8;     // points per thread
constexpr int kTile = kNT * kL;

// --------------------------------------------------------------- LMS setup
__global__ void k_lms(uint32_t d, const uint32_t *__restrict__ C, const uint32_t *__restrict__ S,
                      uint32_t *__restrict__ Ct) {
  const uint32_t rj = blockIdx.x;       // r * d + j
  const uint32_t j = rj % d;
  const int k = threadIdx.x;            // column
  __shared__ uint32_t rows[32];
  rows[k] = S[(size_t)rj * 32 + k];
  __syncthreads();
  const uint32_t col = C[(size_t)j * 32 + k];
  uint32_t out = 0;
#pragma unroll
  for (int t = 0; t < 32; ++t) out |= (uint32_t)(__popc(rows[t] & col) & 1) << (31 - t);
  Ct[(size_t)rj * 32 + k] = out;
}

int launch_lms(uint32_t d, uint32_t R, const uint32_t *C, const uint32_t *S, uint32_t *Ct,
               cudaStream_t st) {
  const uint64_t blocks = (uint64_t)d * R;
  if (blocks == 0) return QK_OK;
  k_lms<<<(unsigned)blocks, 32, 0, st>>>(d, C, S, Ct);
  return check_launch("qk_lms_setup");
}

// ---------------------------------------------------------- point generation
// Store-bound: 4 n d R bytes.  A tile is NP = 2^lognp consecutive points (aligned to NP) of every
// dimension of one randomization: NP d consecutive output words, written by NTA = NP d / 32
// threads as 8 groups of 4 words each, thread t's group `it` at word 4 t + 4 NTA it: whole warps
// store 512 consecutive bytes.  4 NTA words are 2^(lognp - 3) points, so a thread's four words
// keep their dimensions, and the points' index bits split into disjoint fields: position inside
// the group, it (3 bits), tile.  The index maps h(i) = i and i ^ (i >> 1) are linear over GF(2),
// so with one word per field
//   nets:     X = F(thread) ^ A(it) ^ T(tile), T stepping by the XOR of the columns of the tile
//             bits that flip (one table word per step);
//   lattices: brev(i) g is additive over the fields: X = F + A(it) + T, T = brev(tile) g + D,
// i.e. one XOR or add per word and a 16-byte store per four, no shared-memory staging and no
// barrier between tiles (32 x 1000003 x 13 words: see the launch below).
// Warps' stores start on 128-byte lines (a line written in two parts by two warps costs L2 a
// merge): where a randomization's tiles start phi words past such a boundary, the groups shift
// down by phi; the first phi words of the shifted groups then belong to the region before (for
// the first group: to the tile's end), their values lagging one group.  One thread at most
// stores its first and last words one by one; so do the tiles cut by the range's ends.
constexpr int kGenNT = 256;

// log2 of the tile's points: NTA = 2^(lognp - 5) d threads, the largest that fit a CTA.
static uint32_t gen_lognp(uint32_t d) {
  uint32_t k = 5;
  while ((2u << (k - 5)) * d <= (uint32_t)kGenNT) ++k;
  return k;
}

template <bool NET>
__device__ __forceinline__ uint32_t gen_add(uint32_t a, uint32_t b) {
  if constexpr (NET) return a ^ b;
  else return a + b;
}

template <bool NET>
__global__ void __launch_bounds__(kGenNT) k_points(uint32_t d, int order, const uint32_t *__restrict__ Ct,
                                                   const uint32_t *__restrict__ g, const uint32_t *__restrict__ D,
                                                   uint32_t r0, uint32_t nr, uint64_t i0, uint64_t n, uint32_t lognp,
                                                   uint32_t tiles, uint32_t *__restrict__ X) {
  // nets: sC[j][k] = word of position 1 << k (Gray order: columns k and k - 1), rows of 33 words;
  // sP[j][c] = XOR of the words of tile bits 0 .. c
  extern __shared__ uint32_t gsm[];
  uint32_t *sC = gsm, *sP = gsm + 33 * d;
  const uint32_t t = threadIdx.x, NP = 1u << lognp, NTA = d << (lognp - 5), words = NP * d;
  const bool active = t < NTA;
  const uint64_t total = (uint64_t)nr * tiles, chunk = (total + gridDim.x - 1) / gridDim.x;
  const uint64_t it0 = (uint64_t)blockIdx.x * chunk, it1 = it0 + chunk < total ? it0 + chunk : total;
  if (it0 >= it1) return;
  uint32_t rl = (uint32_t)(it0 / tiles), tt = (uint32_t)(it0 - (uint64_t)rl * tiles);
  bool fresh = true;                        // a new randomization: tables and the thread's words
  uint32_t phi = 0;                         // its alignment shift
  uint32_t F[4], A[3][4], T[4], J[4], E[4];  // E: word index in the group's region; J: nets j, lattices g_j
  uint32_t *out = X;                        // word 0 of the tile
  for (uint64_t left = it1 - it0; left; --left) {
    const uint32_t r = r0 + rl;
    const uint64_t tile = (i0 >> lognp) + tt, base = tile << lognp;  // < 2^32
    if (fresh) {
      if constexpr (NET) {
        __syncthreads();
        const uint32_t *C = Ct + (size_t)r * d * 32;
        for (uint32_t q = t; q < 32 * d; q += blockDim.x) {
          const uint32_t j = q >> 5, k = q & 31;
          const uint32_t c = C[q];
          sC[j * 33 + k] = order == QK_GRAY && k ? c ^ C[q - 1] : c;
        }
        __syncthreads();
        for (uint32_t j = t; j < d; j += blockDim.x) {
          uint32_t acc = 0;
          for (uint32_t c = lognp; c < 32; ++c) sP[j * 33 + c - lognp] = acc ^= sC[j * 33 + c];
        }
        __syncthreads();
      }
      // word index of position i, dimension j: (rl n + i - i0) d + j, modulo 2^64 (the tile may
      // start before i0)
      const uint64_t first = ((uint64_t)rl * n - i0 + base) * d;
      out = X + (int64_t)first;
      phi = ((uint32_t)first + (uint32_t)((uintptr_t)X >> 2)) & 31u;
      if (active) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint32_t e = 4 * t + k >= phi ? 4 * t + k - phi : words / 8 - phi + 4 * t + k;
          const uint32_t p = e / d, j = e - p * d;
          E[k] = e;
          uint32_t f = 0, z = 0;
          if constexpr (NET) {
            const uint32_t *c = sC + j * 33;
            for (uint32_t b = 0; b < lognp; ++b) f ^= (p >> b) & 1u ? c[b] : 0u;
            for (uint32_t b = lognp; b < 32; ++b) z ^= (uint32_t)(base >> b) & 1u ? c[b] : 0u;
            for (int b = 0; b < 3; ++b) A[b][k] = c[lognp - 3 + b];
            z ^= D ? D[(size_t)r * d + j] : 0u;
            J[k] = j;
          } else {
            const uint32_t gj = J[k] = g[j];
            f = __brev(p) * gj;
            for (int b = 0; b < 3; ++b) A[b][k] = __brev(1u << (lognp - 3 + b)) * gj;
            z = __brev((uint32_t)base) * gj + (D ? D[(size_t)r * d + j] : 0u);
          }
          F[k] = f, T[k] = z;
        }
      }
    } else if (active) {  // the next tile: bits 0 .. ctz(tile) of the tile index flip
      const uint32_t c = __ffs((int)(uint32_t)tile) - 1;
      const uint32_t db = __brev((uint32_t)base) - __brev((uint32_t)(base - NP));
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if constexpr (NET) T[k] ^= sP[J[k] * 33 + c];
        else T[k] += db * J[k];
      }
    }
    if (active) {
      const uint64_t lo = base > i0 ? base : i0, hi = base + NP < i0 + n ? base + NP : i0 + n;
      const uint32_t elo = (uint32_t)(lo - base) * d, ehi = (uint32_t)(hi - base) * d;
      const uint32_t lag = phi > 4 * t ? (phi - 4 * t < 4 ? phi - 4 * t : 4) : 0;  // this thread's lagging words
      uint32_t V[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) V[k] = gen_add<NET>(F[k], T[k]);
      if (elo == 0 && ehi == words) {
        uint32_t *dst = out + (int32_t)(4 * t - phi);
        uint32_t prev[4] = {0, 0, 0, 0};
#pragma unroll
        for (int it = 0; it < 8; ++it) {
          uint32_t v[4], o[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            v[k] = V[k];
#pragma unroll
            for (int b = 0; b < 3; ++b)
              if (it & (1 << b)) v[k] = gen_add<NET>(v[k], A[b][k]);
            o[k] = (uint32_t)k < lag ? prev[k] : v[k];
            prev[k] = v[k];
          }
          if (it > 0 || lag == 0) {
            *reinterpret_cast<uint4 *>(dst + 4 * NTA * it) = make_uint4(o[0], o[1], o[2], o[3]);
          } else {
#pragma unroll
            for (int k = 1; k < 4; ++k)
              if ((uint32_t)k >= lag) dst[k] = o[k];
          }
        }
        if (lag) {
          uint32_t *tail = dst + words;
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if ((uint32_t)k < lag) tail[k] = prev[k];
        }
      } else {
        for (uint32_t it = 0; it < 8; ++it) {
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const uint32_t q = (uint32_t)k < lag ? (it + 7) & 7 : it, e = E[k] + 4 * NTA * q;
            uint32_t v = V[k];
#pragma unroll
            for (int b = 0; b < 3; ++b)
              if (q & (1u << b)) v = gen_add<NET>(v, A[b][k]);
            if (e >= elo && e < ehi) out[e] = v;
          }
        }
      }
    }
    out += words;
    fresh = ++tt == tiles;
    if (fresh) tt = 0, ++rl;
  }
}

int launch_gen_points(const qk_pointset *ps, uint32_t r0, uint32_t nr, uint64_t i0, uint64_t n,
                      uint32_t *X, cudaStream_t st) {
  if (n == 0 || nr == 0) return QK_OK;
  const uint32_t d = ps->d, lognp = gen_lognp(d), threads = ((d << (lognp - 5)) + 31) & ~31u;
  const uint64_t tiles = ((i0 + n - 1) >> lognp) - (i0 >> lognp) + 1;  // <= 2^27
  const bool net = ps->kind == QK_NET_B2;
  const size_t smem = net ? sizeof(uint32_t) * 66 * d : 0;
  int occ = 0;
  if (net) {
    smem_optin<k_points<true>>(smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_points<true>, (int)threads, smem);
  } else {
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_points<false>, (int)threads, smem);
  }
  if (occ < 1) occ = 1;
  // one wave of resident CTAs, each taking an equal contiguous chunk of the (r, tile) items
  const uint64_t total = (uint64_t)nr * tiles;
  uint64_t grid = (uint64_t)sm_count() * occ;
  if (grid > total) grid = total;
  if (net)
    k_points<true><<<(unsigned)grid, threads, smem, st>>>(d, ps->order, ps->Ct, nullptr, ps->D, r0, nr, i0, n, lognp,
                                                          (uint32_t)tiles, X);
  else
    k_points<false><<<(unsigned)grid, threads, smem, st>>>(d, ps->order, nullptr, ps->g, ps->D, r0, nr, i0, n, lognp,
                                                           (uint32_t)tiles, X);
  return check_launch("qk_gen_points");
}

// First columns.  A CTA covers kNT L points of one randomization (positions job.i0 + [0, n);
// job.i0 is a multiple of kTile, so position bits split into disjoint tile, l, warp and lane
// fields for the XOR tables) and writes `copies` equal rows: a lattice's differences do not
// depend on the shift, so its column is formed once for all randomizations (n = 2^18, d = 32,
// 16 shifts, FP64: 1278 us one by one, 95 us once).
template <typename T, int FAM, int ALPHA, int L>
__global__ void __launch_bounds__(kNT) k_kernel_col(ColJob job, int form, uint32_t copies, T *__restrict__ out) {
  extern __shared__ __align__(16) unsigned char smem[];
  double *wd;
  DiffTables tb;
  carve_tables<L>(smem, job.d, &wd, tb);
  T *wT = reinterpret_cast<T *>(wd);
  const uint32_t rl = blockIdx.y;
  const uint64_t n = 1ull << job.m;
  const uint64_t tile_base = job.i0 + (uint64_t)blockIdx.x * (kNT * L);
  for (uint32_t q = threadIdx.x; q < job.d; q += kNT) wT[q] = (T)job.w[q];
  build_all<T, FAM, ALPHA, L>(job, job.Ct ? job.Ct + (size_t)rl * job.d * 32 : nullptr, job.g, tile_base, tb);
  __syncthreads();
  uint32_t bi[L];
#pragma unroll
  for (int l = 0; l < L; ++l) bi[l] = __brev((uint32_t)(tile_base + threadIdx.x + (l << 8)));
  T p[L];
  column_sweep<T, FAM, ALPHA, L>(job, tb, wT, bi, p);
  const T zeta = (T)job.zeta;
#pragma unroll
  for (int l = 0; l < L; ++l)
    if (form != QK_COL_P) p[l] = zeta * (T(1) + p[l]);
  for (uint32_t c = 0; c < copies; ++c)
#pragma unroll
    for (int l = 0; l < L; ++l) {
      const uint64_t i = tile_base - job.i0 + threadIdx.x + ((uint64_t)l << 8);
      if (i < n) out[((size_t)rl + c) * n + i] = p[l];
    }
}

// The first column in float-float arithmetic on the FP32 pipes (about 2^-46 relative per
// factor), written as FP64: for spectra that reach far below eps32 ||k_1||, where an FP32
// column would perturb the small eigenvalues beyond the 1/lambda-weighted outputs' tolerance.
template <int FAM, int ALPHA, int L>
__global__ void __launch_bounds__(kNT) k_kernel_col_ff(ColJob job, int form, uint32_t copies, double *__restrict__ out) {
  extern __shared__ __align__(16) unsigned char smem[];
  double *wd;
  DiffTables tb;
  carve_tables<L>(smem, job.d, &wd, tb);
  float2 *wff = reinterpret_cast<float2 *>(wd);
  const uint32_t rl = blockIdx.y;
  const uint64_t n = 1ull << job.m;
  const uint64_t tile_base = job.i0 + (uint64_t)blockIdx.x * (kNT * L);
  for (uint32_t q = threadIdx.x; q < job.d; q += kNT) wff[q] = ff_split(job.w[q]);
  build_all_ff<FAM, ALPHA, L>(job, job.Ct ? job.Ct + (size_t)rl * job.d * 32 : nullptr, job.g, tile_base, tb);
  __syncthreads();
  uint32_t bi[L];
#pragma unroll
  for (int l = 0; l < L; ++l) bi[l] = __brev((uint32_t)(tile_base + threadIdx.x + (l << 8)));
  float ph[L], pl[L];
  column_sweep_ff<FAM, ALPHA, L>(job, tb, wff, bi, ph, pl);
#pragma unroll
  for (int l = 0; l < L; ++l) {
    const uint64_t i = tile_base - job.i0 + threadIdx.x + ((uint64_t)l << 8);
    double p = f2d_exact(ph[l]) + f2d_exact(pl[l]);
    if (form != QK_COL_P) p = job.zeta + job.zeta * p;
    if (i < n)
      for (uint32_t c = 0; c < copies; ++c) out[((size_t)rl + c) * n + i] = p;
  }
}

// Rows to compute and copies of each: lattices one row for all randomizations.
static void col_rows(const ColJob &job, uint32_t &rows, uint32_t &copies) {
  const bool shared = job.kind == QK_LATTICE;
  rows = shared ? 1 : job.nr;
  copies = shared ? job.nr : 1;
}
// Points per thread: 8, or LS where tiles of 8 would leave fewer than four CTAs per SM (a
// column of 2^18 points is 128 tiles of 2048 on 152 SMs).
static bool col_small(const ColJob &job, uint32_t rows) {
  return (uint64_t)ceil_div_u(1ull << job.m, kTile) * rows < 4ull * sm_count();
}

template <typename T, int FAM, int ALPHA, int L>
static void launch_col_l(const ColJob &job, int form, uint32_t rows, uint32_t copies, T *out, cudaStream_t st) {
  const size_t smem = col_smem_bytes<L>(job.d);
  smem_optin<k_kernel_col<T, FAM, ALPHA, L>>(smem);
  k_kernel_col<T, FAM, ALPHA, L><<<dim3(ceil_div_u(1ull << job.m, kNT * L), rows), kNT, smem, st>>>(job, form, copies, out);
}
template <typename T, int FAM, int ALPHA>
static void launch_col_t(const ColJob &job, int form, T *out, cudaStream_t st) {
  constexpr int LS = sizeof(T) == 8 ? 2 : 4;
  uint32_t rows, copies;
  col_rows(job, rows, copies);
  if (col_small(job, rows)) launch_col_l<T, FAM, ALPHA, LS>(job, form, rows, copies, out, st);
  else launch_col_l<T, FAM, ALPHA, kL>(job, form, rows, copies, out, st);
}

template <int FAM, int ALPHA, int L>
static void launch_col_ff_l(const ColJob &job, int form, uint32_t rows, uint32_t copies, double *out, cudaStream_t st) {
  const size_t smem = col_smem_bytes<L>(job.d);
  smem_optin<k_kernel_col_ff<FAM, ALPHA, L>>(smem);
  k_kernel_col_ff<FAM, ALPHA, L><<<dim3(ceil_div_u(1ull << job.m, kNT * L), rows), kNT, smem, st>>>(job, form, copies, out);
}
template <int FAM, int ALPHA>
static void launch_col_ff(const ColJob &job, int form, double *out, cudaStream_t st) {
  uint32_t rows, copies;
  col_rows(job, rows, copies);
  if (col_small(job, rows)) launch_col_ff_l<FAM, ALPHA, 4>(job, form, rows, copies, out, st);
  else launch_col_ff_l<FAM, ALPHA, kL>(job, form, rows, copies, out, st);
}

static int dispatch_col_ff(const ColJob &job, int form, double *out, cudaStream_t st) {
  if (job.family == QK_DSI) {
    switch (job.alpha) {
      case 1: launch_col_ff<0, 1>(job, form, out, st); break;
      case 2: launch_col_ff<0, 2>(job, form, out, st); break;
      case 3: launch_col_ff<0, 3>(job, form, out, st); break;
      case 4: launch_col_ff<0, 4>(job, form, out, st); break;
      default: return fail(QK_EINVAL, "DSI order must be 1..4");
    }
  } else {
    switch (job.alpha) {
      case 1: launch_col_ff<1, 1>(job, form, out, st); break;
      case 2: launch_col_ff<1, 2>(job, form, out, st); break;
      default: return fail(QK_EINVAL, "SI smoothness must be 1 or 2");
    }
  }
  return check_launch("qk_kernel_col (float-float)");
}

template <typename T>
static int dispatch_col(const ColJob &job, int form, T *out, cudaStream_t st) {
  if (job.family == QK_DSI) {
    switch (job.alpha) {
      case 1: launch_col_t<T, 0, 1>(job, form, out, st); break;
      case 2: launch_col_t<T, 0, 2>(job, form, out, st); break;
      case 3: launch_col_t<T, 0, 3>(job, form, out, st); break;
      case 4: launch_col_t<T, 0, 4>(job, form, out, st); break;
      default: return fail(QK_EINVAL, "DSI order must be 1..4");
    }
  } else {
    switch (job.alpha) {
      case 1: launch_col_t<T, 1, 1>(job, form, out, st); break;
      case 2: launch_col_t<T, 1, 2>(job, form, out, st); break;
      default: return fail(QK_EINVAL, "SI smoothness must be 1 or 2");
    }
  }
  return check_launch("qk_kernel_col");
}

int launch_kernel_col(const ColJob &job, int32_t dtype, int32_t form, void *out, cudaStream_t st) {
  if (job.nr == 0) return QK_OK;
  if (dtype == QK_F32W) return dispatch_col_ff(job, form, (double *)out, st);
  return dtype == QK_F64 ? dispatch_col<double>(job, form, (double *)out, st)
                         : dispatch_col<float>(job, form, (float *)out, st);
}

// ------------------------------------------------------- gradient partials
// dk_1[i]/dc_j = zeta K_ij prod_{j' != j} f_ij' with f_ij = 1 + c_j K_ij, computed as
// zeta (1 + p_i) K_ij / f_ij (explicit product where f_ij == 0).  FP32 sweeps; FP64 ones are in
// qk_grad.cuh.
template <int FAM, int ALPHA>
__global__ void __launch_bounds__(kNT) k_grad_partials(ColJob job, uint32_t nrhs, const float *__restrict__ u,
                                                       double *__restrict__ partial, int pairs,
                                                       const double *__restrict__ pcol) {
  extern __shared__ __align__(16) unsigned char smem[];
  double *wd;
  DiffTables tb;
  carve_tables<kL>(smem, job.d, &wd, tb);
  float *wT = reinterpret_cast<float *>(wd);
  const uint32_t d = job.d;
  double *red = reinterpret_cast<double *>(smem + col_smem_bytes<kL>(d));  // [warp][2d]
  const uint32_t v = blockIdx.y;  // vector = r * nrhs + rhs
  const uint32_t rl = v / nrhs;
  const uint64_t n = 1ull << job.m;
  const uint64_t tile_base = (uint64_t)blockIdx.x * kTile;
  for (uint32_t q = threadIdx.x; q < d; q += kNT) wT[q] = (float)job.w[q];
  build_all<float, FAM, ALPHA, kL>(job, job.Ct ? job.Ct + (size_t)rl * d * 32 : nullptr, job.g, tile_base, tb);
  __syncthreads();
  uint32_t bi[kL];
  float uu[kL], k1[kL];
  bool ok[kL];
#pragma unroll
  for (int l = 0; l < kL; ++l) {
    const uint64_t i = tile_base + threadIdx.x + ((uint64_t)l << 8);
    bi[l] = __brev((uint32_t)i);
    ok[l] = i < n;
    const size_t ui = pairs ? ((((size_t)(v >> 1) * n) + i) << 1) + (v & 1) : (size_t)v * n + i;
    uu[l] = ok[l] ? u[ui] : 0.f;
  }
  float p[kL];
  if (pcol) {  // the first column as computed before (p form, FP64; lattices: one row for all shifts)
    const uint32_t pr = FAM == 1 ? 0u : rl;
#pragma unroll
    for (int l = 0; l < kL; ++l) {
      const uint64_t i = tile_base + threadIdx.x + ((uint64_t)l << 8);
      p[l] = ok[l] ? (float)pcol[(size_t)pr * n + i] : 0.f;
    }
  } else {
    column_sweep<float, FAM, ALPHA, kL>(job, tb, wT, bi, p);
  }
  const float zeta = (float)job.zeta;
  float wk[kL];
#pragma unroll
  for (int l = 0; l < kL; ++l) {
    k1[l] = ok[l] ? zeta * (1.f + p[l]) : 0.f;
    wk[l] = uu[l] * k1[l];
  }
  gradient_sweep<FAM, ALPHA, kL>(job, tb, wT, bi, k1, wk, ok, [&](int l) { return uu[l]; }, red);
  __syncthreads();
  double *dst = partial + ((size_t)v * gridDim.x + blockIdx.x) * 2 * d;
  for (uint32_t q = threadIdx.x; q < 2 * d; q += kNT) dst[q] = red_total(red, kNT / 32, 2 * d, q);
}

uint32_t grad_blocks(uint32_t m, bool fp64) { return fp64 ? grad64_blocks(m) : ceil_div_u(1ull << m, kTile); }

__global__ void k_ratio_selftest(const double *__restrict__ a, const double *__restrict__ b, double *__restrict__ q,
                                 uint64_t n) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    double v;  // as in the FP64 gradient sweep
    if (!ratio_lean(a[i], b[i], v)) v = ratio(a[i], b[i]);
    q[i] = v;
  }
}

template <int FAM, int ALPHA>
static void launch_grad_t(const ColJob &job, uint32_t nrhs, const float *u, double *partial, int pairs,
                          const double *pcol, cudaStream_t st) {
  dim3 grid(grad_blocks(job.m, false), job.nr * nrhs);
  const size_t smem = col_smem_bytes<kL>(job.d) + (size_t)(kNT / 32) * 2 * job.d * sizeof(double);
  smem_optin<k_grad_partials<FAM, ALPHA>>(smem);
  k_grad_partials<FAM, ALPHA><<<grid, kNT, smem, st>>>(job, nrhs, u, partial, pairs, pcol);
}

static int dispatch_grad(const ColJob &job, uint32_t nrhs, const float *u, double *partial, int pairs,
                         const double *pcol, cudaStream_t st) {
  if (job.family == QK_DSI) {
    switch (job.alpha) {
      case 1: launch_grad_t<0, 1>(job, nrhs, u, partial, pairs, pcol, st); break;
      case 2: launch_grad_t<0, 2>(job, nrhs, u, partial, pairs, pcol, st); break;
      case 3: launch_grad_t<0, 3>(job, nrhs, u, partial, pairs, pcol, st); break;
      case 4: launch_grad_t<0, 4>(job, nrhs, u, partial, pairs, pcol, st); break;
      default: return fail(QK_EINVAL, "DSI order must be 1..4");
    }
  } else {
    switch (job.alpha) {
      case 1: launch_grad_t<1, 1>(job, nrhs, u, partial, pairs, pcol, st); break;
      case 2: launch_grad_t<1, 2>(job, nrhs, u, partial, pairs, pcol, st); break;
      default: return fail(QK_EINVAL, "SI smoothness must be 1 or 2");
    }
  }
  return check_launch("gradient partials");
}

int launch_grad_partials(const ColJob &job, uint32_t nrhs, int32_t dtype, const void *u, double *partial,
                         cudaStream_t st, bool pairs, const double *pcol) {
  if (job.nr == 0 || nrhs == 0) return QK_OK;
  if (job.kind == kHONet) {
    if (pairs || pcol) return fail(QK_EINVAL, "gradient partials: pair layout and stored column are for lattices");
    return launch_grad_partials_ho(job, nrhs, dtype, u, partial, st);
  }
  return dtype == QK_F64 ? launch_grad_partials_f64(job, nrhs, (const double *)u, partial, st, pairs, pcol)
                         : dispatch_grad(job, nrhs, (const float *)u, partial, pairs ? 1 : 0, pcol, st);
}

}  // namespace qk

using namespace qk;

extern "C" int qk_ratio_selftest(const double *a, const double *b, double *q, uint64_t n, qk_stream stream) {
  set_error("%s", "");
  if (n == 0) return QK_OK;
  if (!a || !b || !q) return fail(QK_EINVAL, "qk_ratio_selftest: NULL array");
  uint64_t blocks = (n + 255) / 256;
  const uint64_t cap = (uint64_t)sm_count() * 8;
  if (blocks > cap) blocks = cap;
  k_ratio_selftest<<<(unsigned)blocks, 256, 0, (cudaStream_t)stream>>>(a, b, q, n);
  return check_launch("qk_ratio_selftest");
}
