"""Residual matvecs at the edges of their tilings, both summation variants: 128-row tiles with
ragged ends, tiles inside, across and outside the double-float band, pairs on both sides of
omega r = 20 (band) and 64 (short series), right-hand-side passes of 4, 16, 32, 48 and 64.

Bound 1e-11 per right-hand side, as for the other residual tests."""
import numpy as np
import pytest

from oracle import geometry, operators
from paper_1408_1578_gb300 import inputs
from tests.gpu_util import col_rel, empty, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1408_1578_gb300 import cfie
    c = cfie.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("bc", ["soft", "hard"])
@pytest.mark.parametrize("n,omega", [(64, 6.0), (130, 11.0), (642, 55.0), (1026, 90.0)])
def test_residual_at_tile_edges(ctx, bc, n, omega):
    A = operators.cfie_matrix(geometry.kite(n), omega, omega, bc)
    op = ctx.kite().discretise(n, omega, bc=bc, precision="fp32")
    for nrhs in (1, 5, 9, 17, 33, 65):
        X = inputs.random_density(n, nrhs, seed=nrhs)
        want = (A @ X.T).T
        for variant in (1, 2):
            op.set_residual_variant(variant)
            y = empty(nrhs, n)
            op.apply_residual(to_dev(X), y)
            assert np.max(col_rel(to_host(y), want)) < 1e-11, (nrhs, variant)
    op.close()


@pytest.mark.parametrize("bc", ["soft", "hard"])
@pytest.mark.parametrize("nrhs", [32, 40, 48, 49, 64, 72, 96, 97])
def test_residual_pass_widths(ctx, bc, nrhs):
    """Passes of 16, 32, 48 and 64 right-hand sides, both sides of every change."""
    n, omega = 386, 32.0
    A = operators.cfie_matrix(geometry.kite(n), omega, omega, bc)
    op = ctx.kite().discretise(n, omega, bc=bc, precision="fp32")
    op.set_residual_variant(2)
    X = inputs.random_density(n, nrhs, seed=nrhs)
    y = empty(nrhs, n)
    op.apply_residual(to_dev(X), y)
    assert np.max(col_rel(to_host(y), (A @ X.T).T)) < 1e-11
    op.close()
