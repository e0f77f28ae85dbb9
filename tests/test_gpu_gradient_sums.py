"""How the FP64 gradient sweep adds up its terms: with zero weights and zero generator columns
every term of sum_i dk1_i/dc_j is zeta itself, whose low bits are just under half a unit of the
partial sums, so that every addition to a long chain is rounded the same way and the result's
distance from n zeta counts the additions behind one another.

Bound: one rounding (2^-53) per addition on the longest path: a thread's own points, 3 levels of
pairs, a chain of every second group of eight (256 / d groups of threads), the CTAs' sums of 128
to 1024 points in two chains and 4 levels, and 4 more for the last products."""
import math

import pytest
import torch

from tests import qkcases as qc

pytestmark = pytest.mark.gpu
F64 = torch.float64


@pytest.fixture(scope="module")
def qk():
    from paper_2502_14256_gb300 import build
    build.build()
    from paper_2502_14256_gb300 import qk as q
    return q


@pytest.mark.parametrize("d", [1, 2, 3, 4, 7, 13, 15, 16, 17, 28, 32, 33, 128, 129, 256])
@pytest.mark.parametrize("m,nrhs", [(0, 1), (5, 3), (10, 1), (15, 2), (18, 1)])
def test_long_sums_of_equal_terms(qk, d, m, nrhs):
    n, zeta = 1 << m, 1.0 + 63 * 2.0 ** -52
    Ct = torch.zeros((1, d, 32), dtype=torch.int32, device=qc.dev())
    ps = qk.pointset(qk.QK_NET_B2, d, 1, Ct=Ct)
    w = torch.zeros(d, dtype=F64, device=qc.dev())
    lam, y = torch.ones((1, n), dtype=F64, device=qc.dev()), torch.ones((1, nrhs, n), dtype=F64, device=qc.dev())
    out = torch.empty((1, nrhs, qk.QK_MLL_NOUT), dtype=F64, device=qc.dev())
    grad = torch.empty((1, nrhs, 2 * d + 2), dtype=F64, device=qc.dev())
    qk.mll(ps, qk.kernel(qk.QK_DSI, 1, w, zeta), 0, 1, m, nrhs, 0.0, lam, y, out, grad)
    points = min(n, 128 if m <= 15 else 1 << (m - 8) if m < 18 else 1024)  # of one CTA
    groups, blocks = 256 // d, n // points
    depth = math.ceil(points / groups) + 3 + math.ceil(groups / 16) + 1 + math.ceil(blocks / 32) + 1 + 4 + 4
    want = -zeta * n * n * zeta  # mfac = -zeta sum y / lambda_0^2 times n zeta
    assert float((grad[0, :, d + 1:2 * d + 1] - want).abs().max()) <= depth * 2.0 ** -53 * abs(want)
