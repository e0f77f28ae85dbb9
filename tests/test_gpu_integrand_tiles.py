"""Integrands from the large tiles (2048 points per CTA, taken from eight CTAs per SM on) at the
smallest dimensions and at the largest, where a CTA's tables reach 48 KB of shared memory: a
ragged range of positions against the oracle.

Bound: sums and products of d terms round about d times in either evaluation, and the corner
peak raises its sum to the power d + 1: 4 (d + 2)^2 u of the largest value, u = 2^-53 or 2^-24."""
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


@pytest.mark.parametrize("dtype,u", [(torch.float64, 2.0 ** -53), (torch.float32, 2.0 ** -24)])
@pytest.mark.parametrize("kind", ["net", "lattice"])
@pytest.mark.parametrize("d", [3, 254, 255, 256])
def test_large_tiles(qk, d, kind, dtype, u):
    n, i0 = 2 * 2048 + 3, 2048 + 5
    R = 4 * torch.cuda.get_device_properties(0).multi_processor_count + 1  # (n / 2048) R >= 8 SMs
    g = torch.Generator(device=qc.dev()).manual_seed(d)
    word = lambda *s: torch.randint(-(1 << 31), 1 << 31, s, generator=g, device=qc.dev()).to(torch.int32)  # noqa: E731
    D = word(R, d)
    if kind == "net":
        Ct = word(R, d, 32)
        ps = qk.pointset(qk.QK_NET_B2, d, R, Ct=Ct, D=D)
    else:
        gv = word(d) | 1
        ps = qk.pointset(qk.QK_LATTICE, d, R, g=gv, D=D)
    X = torch.empty((1, n, d), dtype=torch.int32, device=qc.dev())
    for name in ("gfun", "genz_osc", "genz_cp"):
        y = torch.full((R, n), float("nan"), dtype=dtype, device=qc.dev())
        qk.integrand(ps, 0, R, i0, n, name, y, baker=name == "genz_osc")
        assert bool(torch.isfinite(y).all())
        for r in (0, R - 1):
            x = qc.u32_host(qk.gen_points(ps, r, 1, i0, n, X))[0].astype(np.float64) / 2.0 ** 32
            want = o.integrand(name, o.baker(x) if name == "genz_osc" else x)
            err = np.max(np.abs(y[r].cpu().numpy().astype(np.float64) - want))
            assert err <= 4 * (d + 2) ** 2 * u * np.max(np.abs(want)), (name, r, err)
