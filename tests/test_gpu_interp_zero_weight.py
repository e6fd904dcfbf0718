"""Interpolation at markers on cell centres (and at the middle of cells along
one axis only): the kernel has support 2, so the outermost of the four centres
along that axis has weight exactly zero.  A velocity that is not finite there
(along y or z, whose taps are left out whole when their weight is zero) does not
reach the marker, whether the marker lies in the grid or, outside of it, in the
list of irregular markers; elsewhere it does.  Spacings are powers of two, so
the positions are exact."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.grid import Grid
from paper_1901_07892_gb300 import wsi


@pytest.mark.parametrize("bad", [np.inf, np.nan])
@pytest.mark.parametrize("axis", [1, 2])
@pytest.mark.parametrize("where", ["inside", "at the wall", "outside"])
def test_zero_weight(where, axis, bad):
    n, h = (32, 16, 16), 1.0 / 16
    L = [n[d] * h for d in range(3)]
    g = Grid(*n, *L, (-1.0,) * 6)
    rng = np.random.default_rng(6)
    vel = [rng.standard_normal(g.face_shape(d)) * g.interior_face_mask(d) for d in range(3)]
    # taps of the marker at centre 6 along the axis: 5, 6, 7 and, of weight zero, 8
    X = np.full((3, 3), 7.3) * h
    if where == "at the wall":
        X[:, 0] = 0.4 * h
    if where == "outside":
        X[:, 0] = -0.25 * h
    X[1, axis] = 6.5 * h
    X[2, axis] = 7.5 * h  # taps 6 .. 9: reaches plane 8
    ctx = wsi.Context(*n, *L)
    flat = lambda v: np.concatenate([a.ravel() for a in v])
    ref = np.asarray(ctx.interp(flat(vel), X)).reshape(-1, 3)
    for c in range(3):
        if c != axis:  # centres of this axis
            idx = [slice(None)] * 3
            idx[2 - axis] = 8
            vel[c][tuple(idx)] = bad
    got = np.asarray(ctx.interp(flat(vel), X)).reshape(-1, 3)
    ctx.close()
    assert np.array_equal(got[1], ref[1])
    for c in range(3):
        if c != axis:
            assert got[2, c] != ref[2, c]
        else:
            assert np.array_equal(got[:, c], ref[:, c])
