"""The FFT derivative of the sound-hard operator at the longest transforms the library accepts
(Bluestein's N = 2^19 in FP64, 2^21 in FP32), inside the product: on the unit circle exp(i m t) is
an eigenvector, whose eigenvalue is a closed form.

Bounds: FP64, the derivative's modes reach n / 2, so the product carries 2^-53 n / omega, eight
times that here; FP32, 1e-4 as for the other raw FP32 products."""
import numpy as np
import pytest

from tests.closed_forms import disk_hard_eigenvalue
from tests.gpu_util import empty, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1408_1578_gb300 import cfie
    c = cfie.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("precision,n,omega,m", [
    ("fp64", 131074, 50.0, 37), ("fp32", 524290, 40000.0, 20011)])
def test_long_derivative(ctx, precision, n, omega, m):
    op = ctx.circle(1.0).discretise(n, omega, bc="hard", precision=precision)
    if precision == "fp32":
        op.set_variant(2)
    v = np.exp(2j * np.pi * ((m * np.arange(n, dtype=np.int64)) % n) / n)
    y = empty(1, n)
    op.apply(to_dev(v), y)
    lam = disk_hard_eigenvalue(m, omega, omega)
    tol = 8 * 2.0 ** -53 * n / omega if precision == "fp64" else 1e-4
    err = np.linalg.norm(to_host(y)[0] - lam * v) / (abs(lam) * np.sqrt(n))
    assert err < tol, err
    op.close()
