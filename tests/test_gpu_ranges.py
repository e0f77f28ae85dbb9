"""Point generation into runs that start and end off a 128-byte line, at many dimensions and
positions, with guard words on both sides (bit-exact); FP64 integrands at large dimensions.

Bound of the integrands: sums and products of d terms round d times in the oracle and no more
here, and the corner peak raises its sum to the power d + 1: 4 (d + 2)^2 2^-53 of the largest
value."""
import numpy as np
import pytest
import torch

from oracle import qk_oracle as o
from tests import qkcases as qc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qk():
    from paper_2502_14256_gb300 import build
    build.build()
    from paper_2502_14256_gb300 import qk as q
    return q


@pytest.mark.parametrize("kind,order", [("net", "gray"), ("net", "natural"), ("lattice", "natural")])
@pytest.mark.parametrize("d", [2, 3, 8, 13, 32, 120, 256])
def test_points_of_ragged_runs(qk, kind, order, d):
    case = qc.make_case(kind, "dsi" if kind == "net" else "si", 2, d, 2, seed=d, order=order)
    guard = -0x5A5A5A5B
    for i0, n, off in ((0, 1, 1), (31, 33, 3), (12345, 1003, 0), (4095, 257, 31), (1 << 19, 2049, 2)):
        buf = torch.full((off + 2 * n * d + 33,), guard, dtype=torch.int32, device=qc.dev())
        X = buf[off:off + 2 * n * d].view(2, n, d)
        qk.gen_points(case.ps, 0, 2, i0, n, X)
        got = qc.u32_host(X.clone())
        for r in range(2):
            assert np.array_equal(got[r], case.points_ref(r, np.arange(i0, i0 + n), 20)), (i0, n, off, r)
        assert bool((buf[:off] == guard).all()) and bool((buf[off + 2 * n * d:] == guard).all())


@pytest.mark.parametrize("name", ["gfun", "genz_osc", "genz_cp"])
@pytest.mark.parametrize("kind", ["net", "lattice"])
@pytest.mark.parametrize("d", [64, 129, 256])
def test_integrands_of_many_dimensions(qk, name, kind, d):
    case = qc.make_case(kind, "dsi" if kind == "net" else "si", 2, d, 1, seed=d)
    n, i0 = 777, 1 << 11
    y = torch.empty((1, n), dtype=torch.float64, device=qc.dev())
    qk.integrand(case.ps, 0, 1, i0, n, name, y)
    want = o.integrand(name, case.points_ref(0, np.arange(i0, i0 + n), 20).astype(np.float64) / 2.0 ** 32)
    tol = 4 * (d + 2) ** 2 * 2.0 ** -53 * np.max(np.abs(want))
    assert np.max(np.abs(y.cpu().numpy()[0] - want)) <= tol
