"""IB4 transfers where markers crowd into a few cells (a cell's markers are shared out
to several warps) or are far apart, by one or two to a cell or outside the box (one
thread each): around the sizes where the route changes.  Interpolation treats each
marker by itself, so a marker's velocity does not depend on who else is there, to the
bit; spreading adds integers, so neither does its order.  Against the oracle within
1e-11 for the interpolation; for spreading every contribution, a product of
double-float weights and a force, is good to 1e-12, so a face's sum is within 1e-12 of
the sum of the contributions' magnitudes (with a thousand random forces to a cell that
is some 30 times the sum itself)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import ib as oib
from oracle.grid import Grid
from paper_1901_07892_gb300 import inputs, wsi

SHAPE, L = (20, 12, 15), (1.0, 0.9, 0.8)


def _in_cells(rng, counts):
    """Markers in as many cells (along a diagonal), counts[k] of them in the k-th."""
    h = [L[d] / SHAPE[d] for d in range(3)]
    X = []
    for k, n in enumerate(counts):
        c = [(k * s) % SHAPE[d] for d, s in enumerate((1, 5, 4))]
        X.append(np.stack([(c[d] + rng.uniform(0.01, 0.99, n)) * h[d] for d in range(3)], 1))
    return np.concatenate(X)


@pytest.mark.parametrize("counts,outside", [
    ((1,), 0), ((1, 2, 3, 4, 5), 0), ((2, 4, 1, 3) * 5, 40), ((31, 33, 63, 64), 0), ((65, 127, 128, 129, 7), 0),
    ((1, 300, 2, 1000, 8), 300), ((1,) * 20, 1), ((), 200)])
def test_crowds(counts, outside):
    c = inputs.Case(nx=SHAPE[0], ny=SHAPE[1], nz=SHAPE[2], lx=L[0], ly=L[1], lz=L[2])
    g = Grid(c.nx, c.ny, c.nz, c.lx, c.ly, c.lz, c.bc)
    rng = np.random.default_rng(11)
    X = _in_cells(rng, counts) if counts else np.empty((0, 3))
    if outside:
        Y = np.stack([rng.uniform(0, L[d], outside) for d in range(3)], 1)
        Y[:, 0] = np.where(np.arange(outside) % 2, -0.4, SHAPE[0] + 0.4) * L[0] / SHAPE[0]
        X = np.concatenate([X, Y])
    X = X[rng.permutation(len(X))]
    ctx = wsi.Context(c.nx, c.ny, c.nz, c.lx, c.ly, c.lz, c.bc, c.gravity)
    vel = [rng.standard_normal(g.face_shape(d)) * g.interior_face_mask(d) for d in range(3)]
    flat = np.concatenate([a.ravel() for a in vel])
    for _ in range(2):  # the work arrays are left as the next call needs them
        U = ctx.interp(flat, X).reshape(-1, 3)
        ref = oib.interpolate(g, vel, X)
        assert np.abs(U - ref).max() < 1e-11 * np.abs(ref).max()
        F = rng.standard_normal(X.shape)
        S = ctx.spread(F, X, 2e-4)
        ref = np.concatenate([a.ravel() for a in oib.spread(g, F, X, 2e-4)])
        mag = np.concatenate([a.ravel() for a in oib.spread(g, np.abs(F), X, 2e-4)])
        assert np.abs(S - ref).max() < 1e-12 * np.abs(mag).max()
        p = rng.permutation(len(X))
        assert np.array_equal(ctx.spread(F[p], X[p], 2e-4), S)
        for q in (p[: len(p) // 2], p[:1]):
            assert np.array_equal(ctx.interp(flat, X[q]).reshape(-1, 3), U[q])
    ctx.close()


@pytest.mark.parametrize("n,out", [(24000, 0), (30000, 100), (140000, 3000)])
def test_many_sparse(n, out):
    """Markers at random, mostly by ones and twos to a cell: few enough for a warp per
    cell, enough for a thread each to interpolate, and to spread as well."""
    c = inputs.Case(nx=66, ny=60, nz=64, lx=1.1, ly=1.0, lz=1.0)
    g = Grid(c.nx, c.ny, c.nz, c.lx, c.ly, c.lz, c.bc)
    rng = np.random.default_rng(n)
    X = rng.uniform(0, 1, (n, 3)) * np.array([c.lx, c.ly, c.lz])
    X[rng.permutation(n)[:out], 1] = -0.3 * c.ly / c.ny
    ctx = wsi.Context(c.nx, c.ny, c.nz, c.lx, c.ly, c.lz, c.bc, c.gravity)
    vel = [rng.standard_normal(g.face_shape(d)) * g.interior_face_mask(d) for d in range(3)]
    flat = np.concatenate([a.ravel() for a in vel])
    U = ctx.interp(flat, X).reshape(-1, 3)
    ref = oib.interpolate(g, vel, X)
    assert np.abs(U - ref).max() < 1e-11 * np.abs(ref).max()
    p = rng.permutation(n)
    assert np.array_equal(ctx.interp(flat, X[p]).reshape(-1, 3), U[p])
    assert np.array_equal(ctx.interp(flat, X[p[:2000]]).reshape(-1, 3), U[p[:2000]])
    F = rng.standard_normal(X.shape)
    S = ctx.spread(F, X, 2e-4)
    ref = np.concatenate([a.ravel() for a in oib.spread(g, F, X, 2e-4)])
    mag = np.concatenate([a.ravel() for a in oib.spread(g, np.abs(F), X, 2e-4)])
    assert np.abs(S - ref).max() < 1e-12 * np.abs(mag).max()
    assert np.array_equal(ctx.spread(F[p], X[p], 2e-4), S)
    ctx.close()
