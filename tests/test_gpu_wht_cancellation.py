"""FP64 Walsh-Hadamard transforms of vectors whose large entries cancel exactly and whose small
ones lie far below them (beyond the integer butterflies' 82 bits): every small result keeps its
digits, as in FP64 butterflies."""
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


@pytest.mark.parametrize("m", [12, 13, 14, 16, 20, 22])
@pytest.mark.parametrize("far", [40, 60, 90, 200])
def test_small_entries_under_cancelling_large_ones(qk, m, far):
    n, rng = 1 << m, np.random.default_rng(m + far)
    # two equal neighbours: the transform's values at odd places are sums without them, and with
    # one small entry besides they are plus or minus that entry
    x = np.zeros((3, n))
    x[:, 0] = x[:, 1] = rng.uniform(1, 2, 3)
    x[:, 1 << (m // 2)] = rng.uniform(1, 2, 3) * 2.0 ** -far
    want = _wht(x)
    small = np.arange(n) % 2 == 1
    assert np.all(np.abs(want[:, small]) == x[:, 1 << (m // 2)][:, None])
    for run in (qk.fwht, qk.fwht_ws):
        t = torch.from_numpy(x).to(qc.dev())
        run(m, t)
        got = t.cpu().numpy()
        scale = 2.0 ** (-m / 2)
        assert np.all(np.abs(got[:, small] - want[:, small] * scale) <= 2.0 ** -51 * np.abs(want[:, small] * scale))


@pytest.mark.parametrize("m", [2, 5, 9, 11, 12, 13, 15])
@pytest.mark.parametrize("far", [40, 60, 90])
def test_quadratic_form_of_the_small_values(qk, m, far):
    """The same vectors with eigenvalues that leave only the odd places in |Y|^2 / lambda."""
    n, rng = 1 << m, np.random.default_rng(m + far)
    x, lam = np.zeros((2, 1, n)), np.ones((2, n))
    x[..., 0] = x[..., 1] = rng.uniform(1, 2, (2, 1))
    x[..., 2] = rng.uniform(1, 2, (2, 1)) * 2.0 ** -far
    lam[:, ::2] = 2.0 ** 300
    out = torch.empty((2, 1, qk.QK_MLL_NOUT), dtype=torch.float64, device=qc.dev())
    qk.mll_spectrum(qk.QK_DSI, m, torch.from_numpy(lam).to(qc.dev()), torch.from_numpy(x).to(qc.dev()), out)
    # n / 2 values t^2 / n, summed in a tree of n: a rounding per level and three per value
    want = x[..., 2] ** 2 / 2
    assert np.all(np.abs(out[..., qk.QK_MLL_QUAD].cpu().numpy() - want) <= (m + 4) * 2.0 ** -53 * want)
