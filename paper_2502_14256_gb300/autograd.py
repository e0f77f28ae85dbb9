"""torch.autograd.Function over the library's marginal log-likelihood and Bayesian-cubature
posterior mean (Sec. 3.2 with the spectral forms of Sec. 5.4).

The hyper-parameters are per-dimension weights gamma_j, log-lengthscales theta_j (effective
weight c_j = gamma_j exp(theta_j)) and the log-nugget log(eta).  The forward pass runs the
library's kernels: first column in the p = k_1/zeta - 1 form (qk_kernel_col), eigenvalues
(qk_eigs) and the MLL with its gradient block (qk_mll), whose hand-written gradient carries
g_w = (|y~_w|^2/lambda_w^2 - 1/lambda_w)/2 back through the transform and recomputes the
kernel factors.  The backward pass only contracts that block with the incoming gradients and
applies the chain rule from c_j and eta to the parameters.
"""
from __future__ import annotations

import math

import torch

from . import qk


class BayesCubatureMLL(torch.autograd.Function):
    """Returns (mll, post_mean), each of shape (nr, nrhs), for randomizations r0 .. r0+nr-1.

    forward(gamma (d,), log_ls (d,), log_eta () or one element, y (nr, nrhs, n), spec) with spec a
    tuple (ps, family, alpha, zeta, m, r0); gamma, log_ls, log_eta FP64 device tensors;
    y in the computation dtype (FP64 or FP32).  y is data: no gradient flows to it.
    """

    @staticmethod
    def forward(ctx, gamma, log_ls, log_eta, y, spec):
        ps, family, alpha, zeta, m, r0 = spec
        nr, nrhs, n = y.shape
        if n != 1 << m:
            raise ValueError(f"y has {n} points per right-hand side, 2^{m} expected")
        ls = torch.exp(log_ls)
        c = (gamma * ls).to(torch.float64).contiguous()
        le = float(log_eta)  # the one host read before the launches
        eta = math.inf if le > 709.782712893384 else math.exp(le)
        kern = qk.kernel(family, alpha, c, zeta)
        col = torch.empty((nr, n), dtype=y.dtype, device=y.device)
        qk.kernel_col(ps, kern, r0, nr, m, col, form=qk.QK_COL_P)
        lam = torch.empty((nr, n), dtype=torch.float64, device=y.device)
        status = torch.zeros(1, dtype=torch.int32, device=y.device)
        qk.eigs(family, m, col, lam, zeta=zeta, eta=eta, form=qk.QK_COL_P, status=status)
        out = torch.empty((nr, nrhs, qk.QK_MLL_NOUT), dtype=torch.float64, device=y.device)
        want_grad = any(ctx.needs_input_grad[:3])
        d = c.numel()
        grad = torch.empty((nr, nrhs, 2 * d + 2), dtype=torch.float64, device=y.device) if want_grad else None
        qk.mll(ps, kern, r0, nr, m, nrhs, eta, lam, y.contiguous(), out, grad, status=status)
        qk.read_status(status)
        if want_grad:
            ctx.save_for_backward(grad, c, ls)
        ctx.d, ctx.eta, ctx.eta_shape = d, eta, log_eta.shape
        return out[..., qk.QK_MLL_MLL].clone(), out[..., qk.QK_MLL_MEAN].clone()

    @staticmethod
    def backward(ctx, g_mll, g_mean):
        # the block is [dMLL/dc, dMLL/deta | dMEAN/dc, dMEAN/deta]: both halves contracted at once
        grad, c, ls = ctx.saved_tensors
        d, total = ctx.d, None
        for g, half in ((g_mll, grad[..., :d + 1]), (g_mean, grad[..., d + 1:])):
            if g is None:
                continue
            g = g.to(torch.float64)[..., None]
            total = g * half if total is None else torch.addcmul(total, g, half)
        if total is None:
            total = torch.zeros_like(grad[..., :d + 1])
        total = total.sum(dim=(0, 1))
        dc = total[:d]
        return dc * ls, dc * c, (total[d] * ctx.eta).reshape(ctx.eta_shape), None, None


def mll_and_mean(gamma, log_ls, log_eta, y, ps, family: int, alpha: int, m: int, zeta: float = 1.0, r0: int = 0):
    """Differentiable (mll, post_mean) of shape (nr, nrhs); see BayesCubatureMLL."""
    return BayesCubatureMLL.apply(gamma, log_ls, log_eta, y, (ps, family, alpha, zeta, m, r0))
