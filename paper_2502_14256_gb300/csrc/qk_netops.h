// Host entry points of the fused standalone net operations (qk_netops.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace qk {

// What a net operation does with its result v: out = v, out += v, out = y - v.
enum { NET_SET = 0, NET_ADD = 1, NET_RESIDUAL = 2 };

// Whether the fused forms take n = 2^m (transform precision FP64 or FP32) for nvec vectors.
bool net_ops_supported(uint32_t m, uint64_t nvec, bool fp64);
// Partial sums per vector that net_mll writes (quadratic form and sum g in pairs; sum y).
uint32_t net_mll_blocks(uint32_t m, bool fp64);

// T: transform precision; X: scratch of nvec * n elements of T.  With old (the eigenvalues of the
// first half, batch * n), col is the new half's and lam (batch * 2n) the doubled set's.
template <typename T>
int net_eigs(uint32_t m, uint32_t batch, const T *col, T *X, double zmul, double dc, double eta, const double *old,
             double *lam, uint32_t *status, cudaStream_t st);
// out = op(K^-1 in) (inverse) or op(K in); in may alias out.
template <typename T, typename TIO>
int net_apply(uint32_t m, uint32_t nvec, uint32_t nrhs, const double *lam, const TIO *in, const TIO *y, TIO *out, T *X,
              int inverse, int op, cudaStream_t st);
// u = H g (nullable) and the partial sums; u may be X.
template <typename T, typename TIO>
int net_mll(uint32_t m, uint32_t nvec, uint32_t nrhs, const double *lam, const TIO *y, T *X, double *part, double *ysum,
            TIO *u, cudaStream_t st);

}  // namespace qk
