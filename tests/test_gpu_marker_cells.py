"""IB4 transfers cell by cell, at the edges of their batches: cells holding one
marker, a batch (four and eight), more than a batch, and dozens; markers
exactly on cell faces, on walls and outside the box by up to half a cell (the
list of irregular markers); 2-D; a marker count that grows on one context.
Against the oracle, with the bounds of the existing transfer tests (the
double-float sums land near 1e-13), and bit-identical when the markers come in
another order (spreading: integer sums; interpolation: marker by marker)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import ib as oib
from oracle.grid import Grid
from paper_1901_07892_gb300 import inputs, wsi


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()


def _markers(rng, n, L, outside):
    h = [L[d] / n[d] for d in range(3)]
    X = []
    for count in (1, 2, 3, 4, 5, 7, 8, 9, 16, 17, 37, 70):
        c = [rng.integers(0, n[d]) for d in range(3)]
        X.append(np.stack([(c[d] + rng.uniform(0, 1, count)) * h[d] for d in range(3)], 1))
    X.append(np.stack([rng.integers(0, n[d] + 1, 40) * h[d] for d in range(3)], 1))  # cell corners and walls
    if outside:
        Y = np.stack([rng.uniform(0, L[d], 30) for d in range(3)], 1)
        for t in range(30):
            d = t % 3 if n[2] > 1 else t % 2
            Y[t, d] = -rng.uniform(0.01, 0.5) * h[d] if t % 2 else L[d] + rng.uniform(0.01, 0.5) * h[d]
        X.append(Y)
    X = np.concatenate(X)
    return X[rng.permutation(len(X))]


@pytest.mark.parametrize("shape", [(21, 18, 15), (4, 2, 3), (16, 12, 1)])
@pytest.mark.parametrize("outside", [False, True])
def test_transfers(shape, outside):
    bc = (-1.0, -1.0, 1.0, -1.0, -1.0, 1.0) if shape[2] > 1 else (-1.0,) * 4 + (1.0, 1.0)
    c = inputs.Case(nx=shape[0], ny=shape[1], nz=shape[2], lx=1.0, ly=0.9, lz=0.8, bc=bc)
    g = Grid(c.nx, c.ny, c.nz, c.lx, c.ly, c.lz, c.bc)
    rng = np.random.default_rng(3)
    ctx = wsi.Context(c.nx, c.ny, c.nz, c.lx, c.ly, c.lz, c.bc, c.gravity)
    vel = [rng.standard_normal(g.face_shape(d)) * g.interior_face_mask(d) for d in range(3)]
    flat = np.concatenate([a.ravel() for a in vel])
    X = _markers(rng, shape, (c.lx, c.ly, c.lz), outside)
    few = ctx.interp(flat, X[:5])
    U = ctx.interp(flat, X).reshape(-1, 3)
    ref = oib.interpolate(g, vel, X)
    assert np.abs(U - ref).max() < 1e-11 * np.abs(ref).max()
    assert np.array_equal(few.reshape(-1, 3), U[:5])
    F = rng.standard_normal(X.shape)
    S = ctx.spread(F, X, 2e-4)
    ref = np.concatenate([a.ravel() for a in oib.spread(g, F, X, 2e-4)])
    assert np.abs(S - ref).max() < 1e-12 * max(np.abs(ref).max(), 1e-300)
    p = rng.permutation(len(X))
    assert np.array_equal(ctx.interp(flat, X[p]).reshape(-1, 3), U[p])
    assert np.array_equal(ctx.spread(F[p], X[p], 2e-4), S)
    ctx.close()
