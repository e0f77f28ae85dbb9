"""The FP64 Walsh-Hadamard transform, whose butterflies run in 96-bit integers over each tile's
largest exponent: against sums in extended precision, over value ranges inside that path and
outside it (zero, tiny, huge, infinite and NaN tiles take FP64 butterflies).

Bound: the low pass rounds each value once (2^-53 relative), the column pass sums 2^(m-12) of
them, rounds once and scales: |error| <= 4 2^-53 ||x||_2 for the orthonormal transform; values
cut at 2^-82 of a tile's largest add less than 2^-60 of it."""
import numpy as np
import pytest
import torch

from tests import qkcases as qc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qk():
    from paper_2502_14256_gb300 import build
    build.build()
    from paper_2502_14256_gb300 import qk as q
    return q


def _wht(x):
    x, h, n = x.copy(), 1, x.shape[-1]
    while h < n:
        v = x.reshape(-1, n // (2 * h), 2, h)
        a, b = v[:, :, 0].copy(), v[:, :, 1].copy()
        v[:, :, 0], v[:, :, 1] = a + b, a - b
        h *= 2
    return x


def _values(kind, rng, n):
    x = rng.standard_normal(n)
    if kind == "spread":
        x *= 2.0 ** rng.integers(-60, 60, n)
    elif kind == "spike":
        x[rng.integers(n)] = 1e16
    elif kind == "zero":
        x[:] = 0.0
    elif kind == "zero_tiles":
        x[4096:8192] = 0.0
        x[:17] = 0.0
    elif kind == "tiny":
        x *= 1e-290
    elif kind == "huge":
        x *= 1e290
    return x


@pytest.mark.parametrize("kind", ["normal", "spread", "spike", "zero", "zero_tiles", "tiny", "huge"])
@pytest.mark.parametrize("m", [4, 12, 13, 17, 20])
def test_transform_against_extended_precision(qk, m, kind):
    n, rng = 1 << m, np.random.default_rng(m)
    x = np.stack([_values(kind, rng, n) if n > 8192 or kind != "zero_tiles" else _values("spread", rng, n) for _ in range(3)])
    want = _wht(x.astype(np.longdouble)) / np.sqrt(np.longdouble(n))
    for run in (qk.fwht, qk.fwht_ws):
        t = torch.from_numpy(x).to(qc.dev())
        run(m, t)
        err = np.max(np.abs(t.cpu().numpy().astype(np.longdouble) - want), axis=1)
        norm = np.sqrt(np.sum(x.astype(np.longdouble) ** 2, axis=1))
        # the generic path (m <= 12) rounds at each stage: sqrt(m + 1) roundings in a random walk
        assert np.all(err <= (4 if m > 12 else 4 * np.sqrt(m + 1)) * 2.0 ** -53 * norm), (run, err / norm)


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_non_finite_values_spread_as_in_floating_point(qk, bad):
    m = 13
    x = np.random.default_rng(1).standard_normal((2, 1 << m))
    x[0, 4100] = bad
    t = torch.from_numpy(x).to(qc.dev())
    qk.fwht(m, t)
    got = t.cpu().numpy()
    with np.errstate(invalid="ignore"):
        want = _wht(x)
    assert np.array_equal(np.isfinite(got), np.isfinite(want)) and np.array_equal(np.isnan(got), np.isnan(want))
