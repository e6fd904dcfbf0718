"""The multigrid set-up on a grid of many z-planes: the second level of 4 x 4 x 49152
cells has 24577 planes of faces, whose three arrays together are more than a launch
takes along z.  The same column along x is the measure: the pressure operator of one
phase, red-black colouring and transfers are symmetric under an exchange of axes, so
three V-cycles give the same iterate up to rounding.  In float64 a rounding of the
iterate changes the next residual by 1e-16 of M/h^2, M its largest value; here M/h^2
is some 1e6 times the right-hand side, so 1e-7 leaves a factor of 1000."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1901_07892_gb300 import wsi


def _solve(y, h):
    nz, ny, nx = y.shape
    ctx = wsi.Context(nx, ny, nz, nx * h, ny * h, nz * h, precision=wsi.PREC_FP64)
    one = np.ones(y.shape)
    ctx.set_phases(one, one, 1000.0, 1.2, 500.0, 1e-3, 1.8e-5, 1e-3)
    x, _ = wsi.pressure_solve(ctx, np.ascontiguousarray(y).ravel(), rtol=1e-30, max_cycles=3)
    ctx.close()
    return x.reshape(y.shape)


def test_many_planes():
    y = np.random.default_rng(7).uniform(-1, 1, (49152, 4, 4))
    y -= y.mean()
    a, b = _solve(y, 0.05), _solve(y.transpose(2, 1, 0), 0.05).transpose(2, 1, 0)
    assert np.isfinite(a).all() and np.abs(a).max() > 0
    err = np.abs(a - b).max() / np.abs(b).max()
    print(err)
    assert err < 1e-7
