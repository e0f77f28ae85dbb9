"""The scaling by 1 / lambda (solve) and lambda (product) in every net route: one element, one
tile, two passes, and the multi-pass transform.  With y = a delta_0 and one eigenvalue lambda
for all frequencies every butterfly adds equal values or subtracts them to zero, so entry 0 of
the result is the scaled value itself: a * (1 / lambda) or a * lambda formed in FP64 and rounded
to the data's precision, bit for bit.  FP32 quotients and products are placed next to the
midpoints of two FP32 numbers, where any error before the last rounding would show; FP64
eigenvalues reach from subnormal reciprocals to the largest numbers."""
import numpy as np
import pytest
import torch

from tests import qkcases as qc

pytestmark = pytest.mark.gpu
SIZES = [(0, 20000), (5, 4096), (12, 64), (13, 64), (14, 64), (18, 8), (22, 2)]


@pytest.fixture(scope="module")
def qk():
    from paper_2502_14256_gb300 import build
    build.build()
    from paper_2502_14256_gb300 import qk as q
    return q


def _run(qk, name, m, a, lam):
    R = len(a)
    y = torch.zeros((R, 1, 1 << m), dtype=torch.float32 if a.dtype == np.float32 else torch.float64, device=qc.dev())
    y[:, 0, 0] = torch.from_numpy(a).to(qc.dev())
    lt = torch.from_numpy(lam).to(qc.dev())[:, None].expand(R, 1 << m).contiguous()
    out = torch.empty_like(y)
    (qk.solve if name == "solve" else qk.matvec)(qk.QK_DSI, m, lt, y, out)
    assert m == 0 or bool((out[:, 0, 1:] == 0).all())
    return out[:, 0, 0].cpu().numpy()


@pytest.mark.parametrize("m,R", SIZES)
@pytest.mark.parametrize("name", ["solve", "matvec"])
def test_fp32_scaling_rounds_the_fp64_value(qk, name, m, R):
    rng = np.random.default_rng(m)
    a = (rng.uniform(1, 2, R) * 2.0 ** rng.integers(-8, 8, R) * rng.choice([-1, 1], R)).astype(np.float32)
    mid = rng.integers(1 << 23, 1 << 24, R) + 0.5  # between two FP32 numbers
    q = mid * 2.0 ** rng.integers(-30, -16, R)
    # half of them next to the midpoints, half anywhere
    lam = np.where(rng.random(R) < 0.5, np.abs(a) / q if name == "solve" else q / np.abs(a), 2.0 ** rng.uniform(-20, 20, R))
    want = (a.astype(np.float64) * (1.0 / lam if name == "solve" else lam)).astype(np.float32)
    assert np.array_equal(_run(qk, name, m, a, lam), want)


@pytest.mark.parametrize("m,R", SIZES)
@pytest.mark.parametrize("name", ["solve", "matvec"])
def test_fp64_scaling_is_one_division_and_one_product(qk, name, m, R):
    rng = np.random.default_rng(50 + m)
    a = rng.uniform(1, 2, R) * rng.choice([-1, 1], R)
    lam = 2.0 ** rng.uniform(-30, 30, R)
    k = min(R // 4, 1000)
    lam[:k] = 2.0 ** rng.uniform(-990, 990, k)
    lam[k:2 * k] = np.nextafter(2.0 ** rng.integers(-60, 60, k), rng.choice([0.0, np.inf], k))
    want = a * (1.0 / lam if name == "solve" else lam)
    assert np.array_equal(_run(qk, name, m, a, lam), want)
    # 1 / lambda overflows (or underflows), 1 / (n lambda) does not
    if name == "solve" and m >= 12:
        lam = np.full(R, 2.0 ** -1025)
        assert np.array_equal(_run(qk, name, m, a * 2.0 ** -40, lam), a * 2.0 ** 985)


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_mll_step_divides_as_fp64_does(qk, dtype):
    """One point per set: the quadratic form a is y^2 / lambda, each operation rounded once, and
    the derivative by the nugget (a - 1) / (2 lambda) of that a to two roundings."""
    R, rng = 4000, np.random.default_rng(9)
    lam, y = 2.0 ** rng.uniform(-30, 30, R), rng.uniform(1, 2, R).astype(dtype)
    lam[:400], lam[400:800] = 2.0 ** rng.uniform(-300, 300, 400), np.nextafter(2.0 ** rng.integers(-60, 60, 400), 0.0)
    y[800:1600] = np.sqrt(lam[800:1600] * (1 + 1e-9 * rng.standard_normal(800))).astype(dtype)  # a next to one
    y[1600:1610] = 0.0
    Ct = torch.randint(-(1 << 31), 1 << 31, (R, 1, 32), device=qc.dev()).to(torch.int32)
    w = torch.ones(1, dtype=torch.float64, device=qc.dev())
    out = torch.empty((R, 1, qk.QK_MLL_NOUT), dtype=torch.float64, device=qc.dev())
    grad = torch.empty((R, 1, 4), dtype=torch.float64, device=qc.dev())
    qk.mll(qk.pointset(qk.QK_NET_B2, 1, R, Ct=Ct), qk.kernel(qk.QK_DSI, 2, w), 0, R, 0, 1, 0.0,
           torch.from_numpy(lam[:, None]).to(qc.dev()), torch.from_numpy(y[:, None, None]).to(qc.dev()), out, grad)
    y64 = y.astype(np.float64)
    a = y64 * y64 / lam
    assert np.array_equal(out[:, 0, qk.QK_MLL_QUAD].cpu().numpy(), a)
    g = (a.astype(np.longdouble) - 1) / (2 * lam.astype(np.longdouble))
    assert np.all(np.abs(grad[:, 0, 1].cpu().numpy() - g) <= 2.0 ** -52 * np.abs(g))
