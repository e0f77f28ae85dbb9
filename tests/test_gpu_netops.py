"""Standalone net operations (eigenvalues, doubling, solve with refinement, product, MLL sums)
against extended precision, from one element over one tile to the largest two-pass size and the
first generic one, at nuggets that floor nothing, something or everything, in place and not.

Bounds in the 2-norm: a butterfly stage rounds each value once (u relative, and a stage is
sqrt(2) times an isometry), so a transform of m stages is off by (m + 1) u, and the scaling by
an eigenvalue and the conversions add 4 u; two transforms: 2 (m + 3) u, u = 2^-24 or 2^-53, times
the norm that the exact operator can reach.  Above 2^17 the reference transforms FP64 data in
FP64 too (extended precision is software on some machines) and adds as much."""
import numpy as np
import pytest
import torch

from tests import qkcases as qc

pytestmark = pytest.mark.gpu
F64 = torch.float64
SIZES = [0, 1, 5, 12, 13, 14, 17]


@pytest.fixture(scope="module")
def qk():
    from paper_2502_14256_gb300 import build
    build.build()
    from paper_2502_14256_gb300 import qk as q
    return q


def _wht(x):
    h, n = 1, x.shape[-1]
    x = x.astype(np.longdouble if n <= 1 << 17 else np.float64)
    while h < n:
        v = x.reshape(-1, n // (2 * h), 2, h)
        a, b = v[:, :, 0].copy(), v[:, :, 1].copy()
        v[:, :, 0], v[:, :, 1] = a + b, a - b
        h *= 2
    return x


def _norm(x):
    x = x.astype(np.float64) if x.dtype == np.float32 else x
    return np.sqrt(np.sum(x ** 2, axis=-1))


def _gpu(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to(qc.dev())


def _slack(m, dtype):
    return 2 if m > 17 and dtype == np.float64 else 1


def _cpu(t):
    t = t.cpu().numpy()
    return t.astype(np.longdouble) if t.shape[-1] <= 1 << 17 else t.astype(np.float64)


@pytest.mark.parametrize("dtype,u", [(np.float32, 2.0 ** -24), (np.float64, 2.0 ** -53)])
@pytest.mark.parametrize("m", SIZES + [20, 21])
@pytest.mark.parametrize("eta", [0.0, 1e-8, 0.75, 1e30])
def test_eigenvalues_and_doubling(qk, m, dtype, u, eta):
    if m > 17 and eta not in (1e-8, 0.75):
        pytest.skip("largest sizes at two nuggets")
    n, R, zeta, rng = 1 << m, 3, 1.75, np.random.default_rng(m)
    col = (rng.standard_normal((R, n)) / np.sqrt(n)).astype(dtype)
    want = zeta * _wht(col)
    want[:, 0] += zeta * n
    tol = _slack(m, dtype) * ((m + 5) * u * (zeta * (_norm(col) * np.sqrt(n) + n)) + 2 * u * (eta * np.sqrt(n)))[:, None]
    want = np.maximum(want + eta, eta) if eta > 0 else want
    lam = torch.empty((R, n), dtype=F64, device=qc.dev())
    status = torch.zeros(1, dtype=torch.int32, device=qc.dev())
    qk.eigs(qk.QK_DSI, m, _gpu(col), lam, zeta=zeta, eta=eta, form=qk.QK_COL_P, status=status)
    got = _cpu(lam)
    assert np.all(_norm(got - want)[:, None] <= tol)
    assert not eta > 0 or bool((lam >= eta).all())
    if m == 0:
        return
    # the doubled set from its two halves, against the whole column
    half = torch.empty((R, n // 2), dtype=F64, device=qc.dev())
    qk.eigs(qk.QK_DSI, m - 1, _gpu(col[:, :n // 2]), half, zeta=zeta, eta=eta, form=qk.QK_COL_P)
    lo = _cpu(half) - eta  # the old eigenvalues as stored (floored ones included)
    new = zeta * _wht(col[:, n // 2:].copy())
    new[:, 0] += zeta * (n // 2)
    both = np.concatenate([lo + new, lo - new], axis=1) + eta
    both = np.maximum(both, eta) if eta > 0 else both
    ext = torch.full((R, n), 7.0, dtype=F64, device=qc.dev())
    qk.eigs_extend(qk.QK_DSI, m - 1, _gpu(col[:, n // 2:]), half, ext, zeta=zeta, eta=eta, form=qk.QK_COL_P)
    assert np.all(_norm(_cpu(ext) - both)[:, None] <= 2 * tol)


@pytest.mark.parametrize("dtype,u", [(np.float32, 2.0 ** -24), (np.float64, 2.0 ** -53)])
@pytest.mark.parametrize("m,nrhs", [(m, 3) for m in SIZES] + [(20, 1), (21, 2)])
@pytest.mark.parametrize("inplace", [False, True])
def test_solve_refine_and_product(qk, m, nrhs, dtype, u, inplace):
    n, R, rng = 1 << m, 2, np.random.default_rng(100 + m)
    lam = 2.0 ** rng.uniform(-6, 6, (R, n))
    y = rng.standard_normal((R, nrhs, n)).astype(dtype)
    f = _wht(y) / n
    l3 = lam[:, None, :].astype(np.longdouble if m <= 17 else np.float64)
    lt, ny = _gpu(lam), _norm(y)
    for name, want, gain, steps in (("solve", f / l3, 1 / l3.min(), 0), ("solve", f / l3, 1 / l3.min(), 1),
                                    ("solve", f / l3, 1 / l3.min(), 2), ("matvec", f * l3, l3.max(), 0)):
        want = _wht(want)
        yt = _gpu(y)
        # refinement reads y again, so it writes elsewhere
        out = yt if inplace and steps == 0 else torch.empty_like(yt)
        if name == "solve":
            qk.solve(qk.QK_DSI, m, lt, yt, out, refine_steps=steps)
        else:
            qk.matvec(qk.QK_DSI, m, lt, yt, out)
        assert np.all(_norm(_cpu(out) - want) <= _slack(m, dtype) * 2 * (m + 3) * u * float(gain) * ny), (name, steps)


@pytest.mark.parametrize("dtype,u", [(np.float32, 2.0 ** -24), (np.float64, 2.0 ** -53)])
@pytest.mark.parametrize("m,nrhs", [(m, 3) for m in SIZES] + [(20, 1), (21, 2)])
def test_mll_sums(qk, m, nrhs, dtype, u):
    n, R, rng = 1 << m, 2, np.random.default_rng(200 + m)
    lam = 2.0 ** rng.uniform(-6, 6, (R, n))
    y = rng.standard_normal((R, nrhs, n)).astype(dtype)
    out = torch.empty((R, nrhs, qk.QK_MLL_NOUT), dtype=F64, device=qc.dev())
    qk.mll_spectrum(qk.QK_DSI, m, _gpu(lam), _gpu(y), out)
    got = _cpu(out)
    quad = np.sum(_wht(y) ** 2 / n / lam[:, None, :], axis=-1)
    logdet = np.sum(np.log(lam.astype(np.longdouble)), axis=-1)[:, None]
    # quad = |Y|^2 / lambda: relative error twice that of the transform, through the gain
    tq = _slack(m, dtype) * 2 * 2 * (m + 4) * u * np.sum(y.astype(np.float64) ** 2, axis=-1) / lam.min()
    tl = (2 * u if dtype == np.float32 else 64 * u) * np.sum(np.abs(np.log(lam)), axis=-1)[:, None] + 2 * n * u
    assert np.all(np.abs(got[..., qk.QK_MLL_QUAD] - quad) <= tq)
    assert np.all(np.abs(got[..., qk.QK_MLL_LOGDET] - logdet) <= tl)
