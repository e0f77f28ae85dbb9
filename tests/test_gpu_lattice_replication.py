"""Lattice batch tasks form the first column and its transform once and repeat the eigenvalue rows
for the other randomizations (from four on; below, every row is transformed): at even and odd
counts the rows equal those of the standalone eigenvalues on all columns bit for bit, and solve,
MLL and gradient equal the standalone operations on the task's own eigenvalues.

Bounds at a condition below 2^10: 20 cond u, i.e. 2e-12 in FP64 and 1.2e-3 with FP32 data, with
room for the gradients' cancellation in FP64 (1e-10); a wrong row is off by its own size."""
import numpy as np
import pytest
import torch

from tests import qkcases as qc

pytestmark = pytest.mark.gpu
F64, F32 = torch.float64, torch.float32


@pytest.fixture(scope="module")
def qk():
    from paper_2502_14256_gb300 import build
    build.build()
    from paper_2502_14256_gb300 import qk as q
    return q


@pytest.mark.parametrize("R", [3, 4, 5, 7, 16])
@pytest.mark.parametrize("precision,refine", [("f64", 0), ("f32w", 1), ("f32", 0), ("f32", 1)])
def test_rows_of_many_randomizations(qk, R, precision, refine):
    m, d, q, eta = 10, 3, 2, 4.0
    n, dt = 1 << m, {"f64": F64, "f32": F32, "f32w": qk.F32W}[precision]
    case = qc.make_case("lattice", "si", 2, d, R, seed=6100 + R, c=0.3 ** np.arange(1, d + 1), m_gen=m)
    kern = qc.kernel_of(case)
    g = torch.Generator(device=qc.dev()).manual_seed(R)
    y = torch.randn((R, q, n), dtype=F64, device=qc.dev(), generator=g).to(qk.data_dtype(dt)).contiguous()
    sol, lam = torch.empty_like(y), torch.full((R, n), 7.0, dtype=F64, device=qc.dev())
    out = torch.empty((R, q, qk.QK_MLL_NOUT), dtype=F64, device=qc.dev())
    grad = torch.empty((R, q, 2 * d + 2), dtype=F64, device=qc.dev())
    task = qk.Task(case.ps, kern, m, q, eta, y.data_ptr(), sol.data_ptr(), lam.data_ptr(), out.data_ptr(), grad.data_ptr())
    ws = qk.workspace(qk.batch_workspace_bytes([task], dt))
    qk.batch_plan([task], dt, refine, ws)
    qk.batch_run(ws, torch.zeros(1, dtype=torch.int32, device=qc.dev()))
    if precision != "f32w":  # whose transforms run in float-float
        col, want = torch.empty((R, n), dtype=dt, device=qc.dev()), torch.empty_like(lam)
        qk.kernel_col(case.ps, kern, 0, R, m, col, form=qk.QK_COL_P)
        qk.eigs(qk.QK_SI, m, col, want, eta=eta, form=qk.QK_COL_P)
        assert torch.equal(lam, want)
    assert all(torch.equal(lam[r], lam[r % 2]) for r in range(R - R % 2))  # an odd last row has its own rounding
    # the same operations one by one, in FP64, on the task's eigenvalues
    y64, sol64, out64, grad64 = y.to(F64), torch.empty_like(y, dtype=F64), torch.empty_like(out), torch.empty_like(grad)
    qk.solve(qk.QK_SI, m, lam, y64, sol64)
    qk.mll(case.ps, kern, 0, R, m, q, eta, lam, y64, out64, grad64)
    tol = 1e-10 if precision == "f64" else 1.2e-3
    assert float(lam.max() / lam.min()) < 2 ** 10
    for got, ref in ((sol, sol64), (out, out64), (grad[..., :d], grad64[..., :d]), (grad[..., d], grad64[..., d]),
                     (grad[..., d + 1:], grad64[..., d + 1:])):
        for r in range(R):
            assert qc.rel_err(got[r].cpu().numpy(), ref[r].cpu().numpy()) < tol, r
