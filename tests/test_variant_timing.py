"""When the FP32 product of the two variants is timed: a choice made at one number of right-hand
sides is not taken at another whose passes are others (sound hard: S and C together or one after
the other, in passes of 32, 40 or 64).  A timed call issues more launches than the next one.  In a
process of its own: choices are kept for the process."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = """
import sys
from paper_1408_1578_gb300 import cfie, inputs
from tests.gpu_util import empty, to_dev
bc, n = sys.argv[1], 3074
ctx = cfie.Context(0)
op = ctx.kite().discretise(n, n / 12.0, bc=bc, precision="fp32")
for nrhs in map(int, sys.argv[2:]):
    x, y = to_dev(inputs.random_density(n, nrhs, seed=1)), empty(nrhs, n)
    spent = []
    for _ in range(2):
        before = ctx.lib.cfie_launch_count()
        op.apply(x, y)
        spent.append(ctx.lib.cfie_launch_count() - before)
    assert spent[0] > spent[1], (nrhs, spent)
op.close()
ctx.close()
"""


@pytest.mark.parametrize("bc,counts", [("hard", (34, 60, 72, 97, 200)), ("soft", (34, 65, 129))])
def test_every_pass_structure_is_timed(bc, counts):
    r = subprocess.run([sys.executable, "-c", CODE, bc, *map(str, counts)], cwd=ROOT,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
