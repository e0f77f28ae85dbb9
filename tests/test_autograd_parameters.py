"""The autograd function's treatment of its parameters, with the native calls replaced by
stand-ins (no GPU): the gradient of the log-nugget takes the shape of the parameter."""
import types

import pytest
import torch

from paper_2502_14256_gb300 import build

build.build()
from paper_2502_14256_gb300 import autograd, qk  # noqa: E402

F64 = torch.float64


@pytest.fixture
def native(monkeypatch):
    """mll fills its outputs with fixed numbers, the other calls do nothing."""
    def mll(ps, kern, r0, nr, m, nrhs, eta, lam, y, out, grad=None, status=None):
        out.copy_(torch.arange(out.numel(), dtype=F64).view(out.shape))
        if grad is not None:
            grad.copy_(torch.arange(1, grad.numel() + 1, dtype=F64).view(grad.shape))

    none = lambda *a, **k: None  # noqa: E731
    fake = types.SimpleNamespace(kernel=none, kernel_col=none, eigs=none, mll=mll, read_status=none, QK_COL_P=qk.QK_COL_P,
                                 QK_MLL_NOUT=qk.QK_MLL_NOUT, QK_MLL_MLL=qk.QK_MLL_MLL, QK_MLL_MEAN=qk.QK_MLL_MEAN)
    monkeypatch.setattr(autograd, "qk", fake)


def _call(log_eta, d=3):
    gamma = torch.linspace(0.5, 1.0, d, dtype=F64, requires_grad=True)
    ls = torch.linspace(-0.1, 0.1, d, dtype=F64, requires_grad=True)
    mll, mean = autograd.mll_and_mean(gamma, ls, log_eta, torch.zeros((2, 1, 8), dtype=F64), None, 0, 1, 3)
    return torch.autograd.grad(mll.sum() + 2 * mean.sum(), (gamma, ls, log_eta))


@pytest.mark.parametrize("shape", [(), (1,), (1, 1)])
def test_log_nugget_gradient_has_the_parameters_shape(native, shape):
    d, le = 3, torch.full(shape, -2.0, dtype=F64, requires_grad=True)
    g = _call(le, d)[2]
    # two blocks of 2 d + 2 entries, counted from 1: entry d of the MLL half, entry d of the mean half
    want = sum((b * (2 * d + 2) + d + 1) + 2 * (b * (2 * d + 2) + 2 * d + 2) for b in range(2)) * float(torch.exp(le.detach()))
    assert g.shape == le.shape and torch.allclose(g.double(), torch.full(shape, want, dtype=F64), rtol=1e-14, atol=0)
