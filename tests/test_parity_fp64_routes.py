"""FP64 products of a few columns on both sides of the limits of their partial sums."""
import numpy as np
import pytest

from paper_1408_1578_gb300 import inputs
from tests.gpu_util import col_rel, empty, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1408_1578_gb300 import cfie
    c = cfie.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("n,bc,nrhs", [
    (2048, "soft", 4), (2050, "soft", 3), (2048, "hard", 2), (2050, "hard", 2),   # the size rule
    (8194, "soft", 2), (12290, "soft", 1), (8194, "hard", 1)])     # beyond the static scratch
def test_few_columns_regular_and_static(ctx, n, bc, nrhs):
    """One to four columns take the kernel that evaluates a pair of nodes once up to some size
    and while its partial sums fit, for the allocation-free product its 32 MB, else the block
    kernel: 1e-12 as for the other FP64 products."""
    op = ctx.kite().discretise(n, n / 12.0, bc=bc, precision="fp64")
    x = to_dev(inputs.random_density(n, nrhs, seed=n))
    y, z = empty(nrhs, n), empty(nrhs, n)
    op.apply_fp64(x, y)
    op.ctx.check(ctx.lib.cfie_apply_fp64_static(op.h, x.data_ptr(), z.data_ptr(), nrhs),
                 "cfie_apply_fp64_static")
    assert np.max(col_rel(to_host(y), to_host(z))) < 1e-12
    op.close()


def test_partial_sums_beyond_their_limit(ctx):
    """Two columns whose partial sums would pass the library's limit against one whose do not."""
    n = 33400
    op = ctx.kite().discretise(n, n / 12.0, bc="soft", precision="fp64")
    x = to_dev(inputs.random_density(n, 2, seed=1))
    y, z = empty(2, n), empty(1, n)
    op.apply_fp64(x, y)
    op.apply_fp64(x[:1].contiguous(), z)
    assert np.max(col_rel(to_host(y)[:1], to_host(z))) < 1e-12
    op.close()
