"""Field points that are not numbers."""
import numpy as np
import pytest

from oracle import field as ofield
from oracle import geometry
from paper_1408_1578_gb300 import inputs
from tests.gpu_util import empty, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1408_1578_gb300 import cfie
    c = cfie.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("bc", ["soft", "hard"])
@pytest.mark.parametrize("nrhs", [1, 5])
def test_points_that_are_not_numbers(ctx, bc, nrhs):
    """NaN of either sign and infinities among the points: their own values are not numbers, the
    other points' are as without them."""
    n, omega = 64, 9.0
    pts = np.array([2.0 + 1j, 3.0 - 2j, -4.0 + 0.5j, 5.0 + 0j])
    bad = np.array([complex(np.nan, 1), complex(1, np.nan), complex(-np.nan, -np.nan),
                    complex(np.copysign(np.nan, -1.0), 2), complex(np.inf, 0),
                    complex(0, -np.inf)])
    every = np.concatenate([pts[:2], bad, pts[2:]])
    q = inputs.random_density(n, nrhs, seed=3)
    op = ctx.kite().discretise(n, omega, bc=bc, precision="fp64")
    u = empty(nrhs, len(every))
    op.field_eval(to_dev(q), to_dev(every), u)
    got = to_host(u)
    xy = np.stack([pts.real, pts.imag], 1)
    want = np.stack([ofield.scattered_field(geometry.kite(n), omega, omega, bc, q[k], xy)
                     for k in range(nrhs)])
    good = np.r_[0:2, 2 + len(bad):len(every)]
    assert np.max(np.abs(got[:, good] - want)) < 1e-12 * np.max(np.abs(want))
    assert not np.isfinite(np.delete(got, good, axis=1)).any()
    op.close()
