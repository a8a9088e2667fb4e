"""A solve alone and in a batch of matrix-free operators of other sizes: the same sums in the same
order, so the same result bit for bit, whatever else the batch holds."""
import numpy as np
import pytest

from paper_1408_1578_gb300 import inputs
from tests.gpu_util import to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1408_1578_gb300 import cfie
    c = cfie.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("sizes", [[(512, 2), (1026, 5)], [(300, 1), (2050, 33), (640, 4)],
                                   [(130, 3), (4098, 64), (6002, 33), (1200, 1)]])
def test_same_bits_alone_and_in_a_batch(ctx, precision, sizes):
    import torch
    from paper_1408_1578_gb300 import cfie
    if precision == "fp64" and sizes[-1][0] == 1200:
        pytest.skip("large sizes in FP32")
    ops = [ctx.kite().discretise(n, n / 16.0, precision=precision) for n, _ in sizes]
    fs = []
    for op, (n, k) in zip(ops, sizes):
        if precision == "fp32":
            op.set_variant(2)        # no timing decides which sums are taken
        f = to_dev(np.zeros((k, n), complex))
        op.rhs_plane_waves(inputs.directions(k), f)
        fs.append(f)
    b = cfie.Batch(ctx, ops, [k for _, k in sizes])
    f = torch.cat([v.reshape(-1) for v in fs]).contiguous()
    x = f.clone().zero_()
    b.gmres_solve(f, x, rtol=1e-8, restart=200, maxit=200)
    for k, op in enumerate(ops):
        alone = fs[k].clone().zero_()
        op.gmres_solve(fs[k], alone, rtol=1e-8, restart=200, maxit=200)
        assert np.array_equal(to_host(alone), to_host(b.block(x, k))), sizes[k]
    b.close()
    for op in ops:
        op.close()
