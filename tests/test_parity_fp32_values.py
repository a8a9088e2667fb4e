"""FP32 entries of the tensor-core sums on their own, and densities that are not finite."""
import numpy as np
import pytest

from oracle import geometry, operators
from paper_1408_1578_gb300 import inputs
from paper_1408_1578_gb300 import inputs
from tests.gpu_util import empty, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1408_1578_gb300 import cfie
    c = cfie.Context(0)
    yield c
    c.close()


def _entries_next_to_the_band(ctx, ratio):
    """Products of unit columns over the exact entries, and omega r, of the pairs with
    16.4 < omega r < 17.4 (the largest arguments of the short series) at eta = ratio omega."""
    n, omega, m = 4096, 64.0, 64
    eta = omega * ratio
    c = geometry.ellipse(n, 1.0, 0.8)
    op = ctx.ellipse(1.0, 0.8).discretise(n, omega, eta=eta, bc="soft", precision="fp32")
    op.set_variant(2)
    cols = (3 * np.arange(m) - 96) % n          # about the slowest node, where the band is widest
    rows = np.arange(-450, 450) % n
    X = np.zeros((m, n), complex)
    X[np.arange(m), cols] = 1.0
    y = empty(m, n)
    op.apply(to_dev(X), y)
    got = to_host(y)[:, rows]
    op.close()
    D, S = (operators.layer_rows(c, omega, rows, k)[:, cols].T for k in "DS")
    A = D - 1j * eta * S
    x = omega * np.hypot(*(c.z[rows][None, :, :] - c.z[cols][:, None, :]).transpose(2, 0, 1))
    pick = (x > 16.4) & (x < 17.4)
    assert pick.sum() > 1000
    return got[pick] / A[pick], x[pick]


def test_amplitude_next_to_the_band(ctx):
    """Unit columns give single entries; with eta small against omega they are H1 times plain
    factors.  Their mean amplitude is no further off than with two terms of P and Q (the leading
    dropped one is 0.144 / x^4), and 3e-7 for the arithmetic: two special-function values of
    1.2e-7, one and a half of them in the amplitude, FP32 per-node factors (6e-8), and the bf16
    hi + lo splits (up to 3e-6, but of either sign) averaged over a thousand distances."""
    q, x = _entries_next_to_the_band(ctx, 1e-6)
    bias = np.mean(np.abs(q)) - 1.0
    assert abs(bias) < np.mean(0.144195556640625 / x ** 4) + 3e-7, bias


@pytest.mark.parametrize("ratio", [1e6, 1e-6])
def test_phase_next_to_the_band(ctx, ratio):
    """The mean phase of H0 (eta large) and H1 (small): the argument 4e-7, sine and cosine 3.6e-7,
    the third term of the phase 3e-7, and 4e-7 for the splits.  (Its second term is 1.5e-5 and
    3.7e-5 there.)"""
    q, _ = _entries_next_to_the_band(ctx, ratio)
    assert abs(np.mean(np.angle(q))) < 1.5e-6, np.mean(np.angle(q))


def test_infinite_density_gives_infinities(ctx):
    """A density with one infinite real part: every product of its column is infinite, as FP64
    sums of the splits' partial sums have it; the other columns stay as they are."""
    n, omega, nrhs = 512, 30.0, 9
    op = ctx.kite().discretise(n, omega, bc="soft", precision="fp32")
    op.set_variant(1)
    X = inputs.random_density(n, nrhs, seed=2)
    y0, y1 = empty(nrhs, n), empty(nrhs, n)
    op.apply(to_dev(X), y0)
    X[3, 100] = complex(np.inf, 0.0)
    op.apply(to_dev(X), y1)
    a, b = to_host(y0), to_host(y1)
    assert np.isinf(b[3].real).all() and np.isinf(b[3].imag).all()
    keep = np.arange(nrhs) != 3
    assert np.array_equal(a[keep], b[keep])
    op.close()
