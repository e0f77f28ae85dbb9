"""Row sums by clusters of CTAs: rows shorter than the CTAs of a cluster reach (most of its CTAs
then have no element and meet in the first one's shared memory at once), rows around a CTA's and
a cluster's stride, and many rows in one launch.  The values are whole numbers, so every sum is
exact and the results equal NumPy's bit for bit."""
import numpy as np
import pytest
import torch

from tests import qkcases as qc

pytestmark = pytest.mark.gpu
DTYPES = [torch.float64, torch.float32]


@pytest.fixture(scope="module")
def qk():
    from paper_2502_14256_gb300 import build
    build.build()
    from paper_2502_14256_gb300 import qk as q
    return q


def _whole(shape, dtype, seed):
    g = torch.Generator().manual_seed(seed)
    return torch.randint(-1000, 1001, shape, generator=g).to(dtype).to(qc.dev())


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("n", [1, 31, 511, 512, 513, 3585, 4096, 4097, 8192, 12289])
def test_means_of_short_rows(qk, dtype, n):
    for R in (2, 3, 1500):
        y = _whole((R, n), dtype, n + R)
        out = qk.rqmc(y, 0.05).cpu().numpy()
        assert np.array_equal(out[4:], y.cpu().numpy().astype(np.float64).sum(axis=1) / n)


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("m", [0, 3, 9, 10, 13])
def test_column_and_weight_sums(qk, dtype, m):
    n, batch = 1 << m, 700
    col = _whole((batch, n), dtype, m).abs()
    S = col.cpu().numpy().astype(np.float64).sum(axis=1)
    out = qk.discrepancy(qk.QK_DSI, m, col).cpu().numpy()
    assert np.array_equal(out[:, 0], S / n) and np.array_equal(out[:, 1], S / (n + S)) and np.array_equal(out[:, 2], 1 / (n + S))
    # with zero eigenvalues the quadratic form vanishes: zeta - 2 zeta sum w is left
    w, lam = _whole((batch, 2, n), dtype, 50 + m), torch.zeros((batch, n), dtype=torch.float64, device=qc.dev())
    got = qk.discrepancy_weights(qk.QK_DSI, m, lam, w).cpu().numpy()
    assert np.array_equal(got, 1 - 2 * w.cpu().numpy().astype(np.float64).sum(axis=2))
