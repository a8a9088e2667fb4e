"""When the FP32 product of the two variants is timed: a choice made at one number of right-hand
sides is not taken at another whose passes are others (sound hard: S and C together or one after
the other, in passes of 32, 40 or 64).  A timed call issues more launches than the next one."""
import pytest

from paper_1408_1578_gb300 import inputs
from tests.gpu_util import empty, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1408_1578_gb300 import cfie
    c = cfie.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("bc,counts", [("hard", (34, 60, 72, 97, 200)), ("soft", (34, 65, 129))])
def test_every_pass_structure_is_timed(ctx, bc, counts):
    n = 3074
    op = ctx.kite().discretise(n, n / 12.0, bc=bc, precision="fp32")
    for nrhs in counts:
        x, y = to_dev(inputs.random_density(n, nrhs, seed=1)), empty(nrhs, n)
        spent = []
        for _ in range(2):
            before = ctx.lib.cfie_launch_count()
            op.apply(x, y)
            spent.append(ctx.lib.cfie_launch_count() - before)
        assert spent[0] > spent[1], (nrhs, spent)
    op.close()
