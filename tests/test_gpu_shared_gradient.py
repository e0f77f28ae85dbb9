"""The FP64 gradient sweep that runs over a point set's factors once for all its right-hand
sides: each vector's block against the same vector alone (nets: the same sums in the same
order, so bit for bit; lattices pair other vectors in a complex transform, so to rounding),
at one vector, ragged and full passes of 16 vectors, and tiles below one block of points."""
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


@pytest.mark.parametrize("kind,alpha", [("net", 1), ("net", 2), ("net", 3), ("net", 4), ("lattice", 1), ("lattice", 2)])
@pytest.mark.parametrize("m,d,nrhs", [(3, 1, 2), (7, 5, 3), (11, 17, 17), (10, 200, 4), (13, 16, 8)])
def test_blocks_of_many_vectors_equal_those_of_one(qk, kind, alpha, m, d, nrhs):
    R, n = 2, 1 << m
    case = qc.make_case(kind, "dsi" if kind == "net" else "si", alpha, d, R, seed=900 + m + d)
    kern, fam = qc.kernel_of(case), qk.QK_DSI if kind == "net" else qk.QK_SI
    col = torch.empty((R, n), dtype=F64, device=qc.dev())
    lam = torch.empty((R, n), dtype=F64, device=qc.dev())
    qk.kernel_col(case.ps, kern, 0, R, m, col, form=qk.QK_COL_P)
    qk.eigs(fam, m, col, lam, eta=1e-2, form=qk.QK_COL_P)
    g = torch.Generator(device=qc.dev()).manual_seed(m)
    y = torch.randn((R, nrhs, n), dtype=F64, device=qc.dev(), generator=g)

    def grad(yy):
        q = yy.shape[1]
        out = torch.empty((R, q, qk.QK_MLL_NOUT), dtype=F64, device=qc.dev())
        gr = torch.empty((R, q, 2 * d + 2), dtype=F64, device=qc.dev())
        qk.mll(case.ps, kern, 0, R, m, q, 1e-2, lam, yy.contiguous(), out, gr)
        return gr

    many = grad(y)
    for q in range(nrhs):
        one = grad(y[:, q:q + 1])[:, 0]
        if kind == "net":
            assert torch.equal(many[:, q], one), q
        else:
            scale = one.abs().amax(dim=1, keepdim=True)
            assert bool(((many[:, q] - one).abs() <= 1e-11 * scale).all()), q
