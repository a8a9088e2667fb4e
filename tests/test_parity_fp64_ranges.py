"""FP64 block sums where the entries of one tile of 32 sources range over many powers of two and
the densities meet the small ones: what is lost has to stay that of FP64 sums.

Bounds: n products and additions, each rounded to 2^-53 of its size, and 8 roundings of each
entry."""
import numpy as np
import pytest
from scipy.special import iv

from oracle import geometry, operators
from oracle.operators import hankel01
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
@pytest.mark.parametrize("gap", [1e-4, 1e-7])
def test_field_next_to_a_node_without_density(ctx, bc, gap):
    n, omega, nrhs = 64, 5.0, 5
    c = geometry.circle(n)
    pts = np.array([[1.0 + gap, 0.0], [0.0, 1.0 + gap], [-1.0 - gap, 1e-3]])
    q = inputs.random_density(n, nrhs, seed=11)
    for i in (0, n // 4, n // 2):
        q[:, i] = 0.0
    op = ctx.circle(1.0).discretise(n, omega, bc=bc, precision="fp64")
    u = empty(nrhs, len(pts))
    op.field_eval(to_dev(q), to_dev(pts[:, 0] + 1j * pts[:, 1]), u)
    d = pts[:, None, :] - c.z[None, :, :]
    r = np.hypot(d[..., 0], d[..., 1])
    h0, h1 = hankel01(omega * r)
    S = 0.25j * h0 * c.speed
    D = 0.25j * omega * h1 * np.einsum("pjk,jk->pj", d, c.normal_unscaled) / r
    K = 2 * np.pi / n * (D - 1j * omega * S if bc == "soft" else -S + D / (1j * omega))
    size = 2 * np.pi / n * (np.abs(D) + np.abs(omega * S)) * (1 if bc == "soft" else 1 / omega)
    bound = 2.0 ** -53 * (n + 16) * (np.abs(q) @ size.T)
    assert np.all(np.abs(to_host(u) - q @ K.T) < bound)
    op.close()


def _uneven_circle(n, a, k):
    """The unit circle with speed exp(a cos k t) / I0(a)."""
    t = 2 * np.pi * np.arange(n) / n
    th = t + sum(2 * iv(m, a) / iv(0, a) * np.sin(m * k * t) / (m * k) for m in range(1, 60))
    d1 = np.exp(a * np.cos(k * t)) / iv(0, a)
    d2 = -a * k * np.sin(k * t) * d1
    e, g = np.stack([np.cos(th), np.sin(th)], 1), np.stack([-np.sin(th), np.cos(th)], 1)
    return geometry.Curve(t, e, g * d1[:, None], g * d2[:, None] - e * (d1 ** 2)[:, None])


@pytest.mark.parametrize("nrhs", [8, 24, 48])
def test_entries_of_slow_nodes(ctx, nrhs):
    """Speeds 1 : 2^20 within 32 nodes: unit densities at the slow ones give their entries, next
    to which the row has entries a million times as large.  Pairs further apart than 1e-3 (the
    normal component of a short distance is itself uncertain), relative to |D| + eta |S|, with
    64 units of 2^-53 for the entry (log-split terms of both signs) on either side."""
    n, omega = 512, 20.0
    c = _uneven_circle(n, 7.0, 8)
    op = ctx.samples(c.z, c.dz, c.ddz).discretise(n, omega, bc="soft", precision="fp64")
    cols = 24 + 64 * (np.arange(nrhs) % 8) + np.arange(nrhs) // 8
    X = np.zeros((nrhs, n), complex)
    X[np.arange(nrhs), cols] = 1.0
    y = empty(nrhs, n)
    op.apply_fp64(to_dev(X), y)
    rows = np.arange(n)
    S, D = operators.layer_rows(c, omega, rows, "S"), operators.layer_rows(c, omega, rows, "D")
    A, size = (D - 1j * omega * S)[:, cols].T, (np.abs(D) + omega * np.abs(S))[:, cols].T
    r = np.hypot(*(c.z[None, :, :] - c.z[cols][:, None, :]).transpose(2, 0, 1))
    far = r > 1e-3
    assert far.sum() > nrhs * n // 2
    assert np.max((np.abs(to_host(y) - A) / size)[far]) < 2 * 64 * 2.0 ** -53
    op.close()
