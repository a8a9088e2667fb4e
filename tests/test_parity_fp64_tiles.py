"""FP64 matvec and field at the edges of their tilings: right-hand-side blocks of 1, 2, 4, 16,
32 / 64 and their remainders, 32- and 64-target tiles with ragged ends, source splits, pairs on
both sides of every change of the Hankel evaluation (omega r = 20, 32, 64).

Bounds: 1e-12 per right-hand side (the FP64 resolution of the Hankel argument, 4e-16 omega
diam, is below it at every size here), as for the other FP64 parity tests."""
import numpy as np
import pytest

from oracle import field as ofield
from oracle import geometry, operators
from paper_1408_1578_gb300 import inputs
from tests.gpu_util import col_rel, empty, to_dev, to_host

pytestmark = pytest.mark.gpu

TOL = 1e-12


@pytest.fixture(scope="module")
def ctx():
    from paper_1408_1578_gb300 import cfie
    c = cfie.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("bc", ["soft", "hard"])
@pytest.mark.parametrize("n,omega", [(8, 1.0), (62, 3.0), (66, 15.0), (510, 260.0), (1026, 30.0)])
def test_right_hand_side_blocks(ctx, bc, n, omega):
    A = operators.cfie_matrix(geometry.kite(n), omega, omega, bc)
    op = ctx.kite().discretise(n, omega, bc=bc, precision="fp64")
    for nrhs in (1, 2, 3, 4, 5, 16, 17, 33, 65):
        X = inputs.random_density(n, nrhs, seed=nrhs)
        x, y = to_dev(X), empty(nrhs, n)
        op.apply_fp64(x, y)
        want = (A @ X.T).T
        assert np.max(col_rel(to_host(y), want)) < TOL, (nrhs, "regular")
        y.zero_()
        op.ctx.check(ctx.lib.cfie_apply_fp64_static(op.h, x.data_ptr(), y.data_ptr(), nrhs),
                     "cfie_apply_fp64_static")
        assert np.max(col_rel(to_host(y), want)) < TOL, (nrhs, "static")
    op.close()


@pytest.mark.parametrize("n,nrhs", [(16, 3), (128, 2), (256, 5), (2048, 4), (4098, 2), (32768, 1)])
def test_spectral_derivative_lengths(ctx, n, nrhs):
    """The FFT derivative (direct for powers of two, Bluestein otherwise, both splits of each
    length) against the circulant one of the allocation-free matvec, inside the sound-hard
    product.  The derivative's modes reach n / 2, so the product carries ~2^-53 n / omega."""
    omega = n / 16.0
    op = ctx.kite().discretise(n, omega, bc="hard", precision="fp64")
    x = to_dev(inputs.random_density(n, nrhs, seed=n))
    y, z = empty(nrhs, n), empty(nrhs, n)
    op.apply_fp64(x, y)
    op.ctx.check(ctx.lib.cfie_apply_fp64_static(op.h, x.data_ptr(), z.data_ptr(), nrhs),
                 "cfie_apply_fp64_static")
    assert np.max(col_rel(to_host(y), to_host(z))) < TOL
    op.close()


@pytest.mark.parametrize("bc", ["soft", "hard"])
@pytest.mark.parametrize("npts,nrhs", [(1, 1), (63, 3), (65, 5), (130, 17)])
def test_field_splits(ctx, bc, npts, nrhs):
    n, omega = 258, 20.0
    c = geometry.kite(n)
    q = inputs.random_density(n, nrhs, seed=5)
    rng = np.random.default_rng(npts)
    pts = rng.uniform(2.0, 30.0, npts) * np.exp(2j * np.pi * rng.uniform(size=npts))
    op = ctx.kite().discretise(n, omega, bc=bc, precision="fp64")
    u = empty(nrhs, npts)
    op.field_eval(to_dev(q), to_dev(pts), u)
    xy = np.stack([pts.real, pts.imag], 1)
    want = np.stack([ofield.scattered_field(c, omega, omega, bc, q[k], xy) for k in range(nrhs)])
    assert np.max(np.abs(to_host(u) - want)) < TOL * np.max(np.abs(want))
    op.close()


@pytest.mark.parametrize("bc", ["soft", "hard"])
@pytest.mark.parametrize("n", [98, 1026])
def test_fixed_point_sums_scales(ctx, bc, n):
    """Sums in fixed point per tile of 32 sources: columns of any scale (those beyond 2^+-420
    take FP64 sums), a tile of zeros, a range of 1e12 over the nodes, every block width.
    Scaling by a power of two commutes with the product except for subnormal rounding."""
    omega = n / 16.0
    A = operators.cfie_matrix(geometry.kite(n), omega, omega, bc)
    op = ctx.kite().discretise(n, omega, bc=bc, precision="fp64")
    for nrhs in (8, 12, 13, 24, 32, 48, 64):
        X = inputs.random_density(n, nrhs, seed=nrhs)
        X[1] *= 2.0 ** 900
        X[2] *= 2.0 ** -900
        X[3, 32:64] = 0.0
        X[4] *= np.exp(-27.0 * np.linspace(0, 1, n))
        x, y = to_dev(X), empty(nrhs, n)
        op.apply_fp64(x, y)
        got, want = to_host(y), (A @ X.T).T
        s = np.ones(nrhs)
        s[1], s[2] = 2.0 ** -900, 2.0 ** 900
        assert np.max(col_rel(got * s[:, None], want * s[:, None])) < TOL, nrhs
        # infinities and NaN stay in their columns
        X[5, n // 3], X[6, 0] = np.inf, np.nan
        op.apply_fp64(to_dev(X), y)
        bad = to_host(y)
        assert not np.isfinite(bad[5:7]).any()
        keep = np.r_[0:5, 7:nrhs]
        assert np.max(col_rel(bad[keep] * s[keep, None], want[keep] * s[keep, None])) < TOL, nrhs
    op.close()


@pytest.mark.parametrize("bc", ["soft", "hard"])
@pytest.mark.parametrize("nrhs", [8, 12, 24, 40, 64])
def test_field_block_widths(ctx, bc, nrhs):
    n, omega, npts = 130, 9.0, 97
    q = inputs.random_density(n, nrhs, seed=7)
    q[2] *= 2.0 ** -900
    rng = np.random.default_rng(nrhs)
    pts = rng.uniform(2.0, 30.0, npts) * np.exp(2j * np.pi * rng.uniform(size=npts))
    op = ctx.kite().discretise(n, omega, bc=bc, precision="fp64")
    u = empty(nrhs, npts)
    op.field_eval(to_dev(q), to_dev(pts), u)
    q[2] *= 2.0 ** 900
    xy = np.stack([pts.real, pts.imag], 1)
    want = np.stack([ofield.scattered_field(geometry.kite(n), omega, omega, bc, q[k], xy)
                     for k in range(nrhs)])
    got = to_host(u)
    got[2] *= 2.0 ** 900
    assert np.max(np.abs(got - want)) < TOL * np.max(np.abs(want))
    op.close()


@pytest.mark.parametrize("bc", ["soft", "hard"])
def test_unit_columns(ctx, bc):
    """Unit densities give the matrix entry by entry, next to the diagonal too: the entries of a
    column to 1e-12 of the column's largest off-diagonal one (sound soft the diagonal, 1/2, is a
    thousand times that)."""
    n, omega, j = 1026, 60.0, 517
    A = operators.cfie_matrix(geometry.kite(n), omega, omega, bc)
    op = ctx.kite().discretise(n, omega, bc=bc, precision="fp64")
    X = np.zeros((8, n), complex)
    X[np.arange(8), j + 40 * np.arange(8)] = 1.0
    y = empty(8, n)
    op.apply_fp64(to_dev(X), y)
    got = to_host(y)
    for k in range(8):
        c = A[:, j + 40 * k].copy()
        off = np.arange(n) != j + 40 * k
        scale = np.max(np.abs(c[off])) if bc == "soft" else np.max(np.abs(c))
        assert np.max(np.abs(got[k] - c)[off]) < TOL * scale, k
        assert abs(got[k] - c)[~off].max() < TOL * np.max(np.abs(c)), k
    op.close()
