"""Edges of the reinitialisation kernel's tiles (64 x 8 cells, two per thread
in x) and of its list of cells next to the interface, against the oracle: a
pair cut in half by the last column, a tile of one column, grids smaller than
the stencil, single-cell axes, and a field that changes sign between most
neighbours, where nearly every cell is listed.  Tolerances: float64 1e-11 of
the field's scale, float32 2e-6 (a few roundings of |phi| per stage)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import reinit as ori
from oracle.grid import Grid
from paper_1901_07892_gb300 import inputs, wsi

TOL = {wsi.PREC_FP64: 1e-11, wsi.PREC_MIXED: 2e-6}


@pytest.mark.parametrize("shape,noise,precision", [
    ((65, 8, 4), 0.0, wsi.PREC_MIXED), ((65, 8, 4), 0.0, wsi.PREC_FP64),
    ((63, 17, 33), 0.0, wsi.PREC_MIXED), ((4, 4, 1), 0.0, wsi.PREC_FP64), ((4, 4, 1), 0.0, wsi.PREC_MIXED),
    ((6, 3, 2), 0.0, wsi.PREC_MIXED), ((67, 9, 1), 0.0, wsi.PREC_FP64), ((130, 9, 6), 1.0, wsi.PREC_FP64)])
def test_reinit_tiles(shape, noise, precision):
    nx, ny, nz = shape
    bc = (-1.0,) * 4 + ((1.0, 1.0) if nz == 1 else (-1.0, -1.0))
    c = inputs.Case(nx=nx, ny=ny, nz=nz, lx=1.0, ly=0.9, lz=0.8, bc=bc)
    x, y, z = c.cell_xyz()
    phi = np.sqrt((x - 0.52) ** 2 + (y - 0.4) ** 2 + (z - 0.4) ** 2) - 0.3
    phi = np.broadcast_to(phi * (1.4 + 0.5 * np.sin(5 * x)), (nz, ny, nx)).copy()
    phi += noise * np.random.default_rng(3).standard_normal(phi.shape)
    ctx = wsi.Context(nx, ny, nz, c.lx, c.ly, c.lz, c.bc, c.gravity, c.n_cells, c.theta, precision=precision)
    got = np.asarray(ctx.reinit(phi.ravel(), 3))
    ctx.close()
    ref = ori.reinit(Grid(nx, ny, nz, c.lx, c.ly, c.lz), phi, 3).ravel()
    assert np.abs(got - ref).max() < TOL[precision] * np.abs(ref).max()
