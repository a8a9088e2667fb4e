"""FP32 matvecs at the edges of their tilings, both summation variants: 128-row and 32-source
tiles with ragged ends, tiles the near band touches, right-hand-side blocks of 8, 16, 32, 64 and
the sound-hard passes (S and C together up to 32 right-hand sides, one pass each above).

Bounds as for the other raw FP32 matvecs, 1e-4 per right-hand side, and between the variants on
the same operator 5e-5 (bf16 hi + lo operands keep 2^-17 per factor, tripled by the products and
magnified at most threefold by the sound-hard derivative)."""
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
@pytest.mark.parametrize("n", [64, 126, 130, 642, 1026])
def test_variants_at_tile_edges(ctx, bc, n):
    omega = n / 12.0
    A = operators.cfie_matrix(geometry.kite(n), omega, omega, bc)
    op = ctx.kite().discretise(n, omega, bc=bc, precision="fp32")
    for nrhs in (1, 9, 17, 32, 33, 65):
        X = inputs.random_density(n, nrhs, seed=nrhs)
        want = (A @ X.T).T
        got = []
        for variant in (1, 2):
            op.set_variant(variant)
            y = empty(nrhs, n)
            op.apply(to_dev(X), y)
            got.append(to_host(y))
            assert np.max(col_rel(got[-1], want)) < 1e-4, (nrhs, variant)
        assert np.max(col_rel(got[1], got[0])) < 5e-5, nrhs
    op.close()


@pytest.mark.parametrize("nrhs", [33, 40, 41, 66, 80, 81])
def test_sound_hard_pass_widths(ctx, nrhs):
    """S and C together in passes of 32 or 40, or one after the other in passes of 64: both sides
    of every change."""
    n, omega = 386, 32.0
    A = operators.cfie_matrix(geometry.kite(n), omega, omega, "hard")
    op = ctx.kite().discretise(n, omega, bc="hard", precision="fp32")
    op.set_variant(2)
    X = inputs.random_density(n, nrhs, seed=nrhs)
    y = empty(nrhs, n)
    op.apply(to_dev(X), y)
    assert np.max(col_rel(to_host(y), (A @ X.T).T)) < 1e-4
    op.close()
