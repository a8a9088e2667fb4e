"""Scratch of FP64 products and fields: what a call takes beyond 64 MB from the device's pool it
gives back."""
import ctypes

import numpy as np
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


def _pool_in_use():
    """Bytes allocated from the device's default memory pool (CU_MEMPOOL_ATTR_USED_MEM_CURRENT)."""
    import torch
    torch.cuda.synchronize()
    cu = ctypes.CDLL("libcuda.so.1")
    pool, used = ctypes.c_void_p(), ctypes.c_uint64()
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
    assert cu.cuMemPoolGetAttribute(pool, 7, ctypes.byref(used)) == 0
    return used.value


def test_products_and_fields_give_large_scratch_back(ctx):
    n = 12290
    op = ctx.kite().discretise(n, n / 12.0, precision="fp64")
    before = _pool_in_use()
    for nrhs in (1, 2, 5, 40):
        x, y = to_dev(inputs.random_density(n, nrhs, seed=1)), empty(nrhs, n)
        op.apply_fp64(x, y)
        assert _pool_in_use() - before <= 64 << 20, nrhs
    q = to_dev(inputs.random_density(n, 64, seed=2))
    pts = to_dev(2.0 + np.arange(40000) * 1e-3)
    op.field_eval(q, pts, empty(64, 40000))
    assert _pool_in_use() - before <= 64 << 20
    op.close()
