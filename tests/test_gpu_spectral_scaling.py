"""The scaling by 1 / lambda (solve) and lambda (product) in every net route: one element, one
tile, two passes, and the multi-pass transform.  With y = a delta_0 and one eigenvalue lambda
for all frequencies every butterfly adds equal values or subtracts them to zero, so entry 0 of
the result is the scaled value itself: a * (1 / lambda) or a * lambda formed in FP64 and rounded
to the data's precision, bit for bit.  FP32 quotients and products are placed next to the
midpoints of two FP32 numbers, where any error before the last rounding would show."""
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
