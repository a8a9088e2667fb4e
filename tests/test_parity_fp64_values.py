"""FP64 Hankel values on their own, through the field of one node: with the density 1 at node 0
of the unit circle, (1, 0), zero elsewhere, and points (1 + x, 0), the sound-soft field is
(h / 4) i (omega H1(x) - i eta H0(x)) at omega = 1.  The distance x is exact in FP64 and eta = 2^60
or 2^-60 leaves (almost) one of the two orders.  Against mpmath at 40 digits.

Bound relative to |H|: 24 units of 2^-53 for the value, its amplitude and the factors (a dozen
roundings each), and the phase's 2 x units (one rounding of the distance each in r and in x)."""
import numpy as np
import pytest

from tests.gpu_util import empty, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1408_1578_gb300 import cfie
    c = cfie.Context(0)
    yield c
    c.close()


def _arguments():
    x = [np.geomspace(1e-6, 19.9, 60), np.geomspace(20.0, 5e4, 160)]
    for c in (20.0, 32.0, 64.0):        # changes of series
        x.append(c + 2.0 ** -np.arange(1, 40, 4))
        x.append(c - 2.0 ** -np.arange(1, 40, 4))
    k = np.arange(1, 40)                # Taylor centres and the middles between them
    x += [k / 2.0, k / 2.0 + 0.25, k / 2.0 - 0.25 + 2.0 ** -45, [20.0, 32.0, 64.0]]
    p = 1.0 + np.concatenate(x)
    return p, p - 1.0                   # the exact distance of each rounded point


@pytest.mark.parametrize("order", [0, 1])
def test_hankel_values(ctx, order):
    mpmath = pytest.importorskip("mpmath")
    n, eta = 64, 2.0 ** (60 if order == 0 else -60)
    p, x = _arguments()
    op = ctx.circle(1.0).discretise(n, 1.0, eta=eta, bc="soft", precision="fp64")
    q = np.zeros((1, n), complex)
    q[0, 0] = 1.0
    u = empty(1, len(p))
    op.field_eval(to_dev(q), to_dev(p.astype(complex)), u)
    got = to_host(u)[0]
    with mpmath.workdps(40):
        err = []
        for g, v in zip(got, x):
            h0, h1 = (mpmath.hankel1(k, mpmath.mpf(float(v))) for k in (0, 1))
            want = mpmath.pi / (2 * n) * (mpmath.mpc(0, 1) * h1 + mpmath.mpf(eta) * h0)
            err.append(float(abs(mpmath.mpc(g.real, g.imag) - want) / abs(want)))
    bound = 2.0 ** -53 * (24 + 2 * x)
    worst = np.argmax(np.array(err) / bound)
    assert err[worst] < bound[worst], (x[worst], err[worst], bound[worst])
    op.close()
