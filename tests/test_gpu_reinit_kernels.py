"""The two kernels of the reinitialisation.  Small, narrow and flat grids take
the one with a cell per thread: one launch per stage (a second launch per stage
and tiles of 64 columns made these grids up to 1.8 times slower).  Large grids
with full tiles take the one with two cells per thread and a second launch for
the cells next to the interface.  Both against the oracle, at the edges of their
tiles (32 x 8 and 64 x 8 cells) and of their marches.  Tolerances: float64 1e-11
of the field's scale, float32 2e-6 (a few roundings of |phi| per stage)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import reinit as ori
from oracle.grid import Grid
from paper_1901_07892_gb300 import inputs, wsi

F64, MIX = wsi.PREC_FP64, wsi.PREC_MIXED
TOL = {F64: 1e-11, MIX: 2e-6}


def _case(shape, precision):
    nx, ny, nz = shape
    bc = (-1.0,) * 4 + ((1.0, 1.0) if nz == 1 else (-1.0, -1.0))
    c = inputs.Case(nx=nx, ny=ny, nz=nz, lx=1.0, ly=0.9, lz=0.8, bc=bc)
    x, y, z = c.cell_xyz()
    phi = np.sqrt((x - 0.52) ** 2 + (y - 0.4) ** 2 + (z - 0.4) ** 2) - 0.3
    phi = np.broadcast_to(phi * (1.4 + 0.5 * np.sin(5 * x)), (nz, ny, nx)).copy()
    return c, phi, wsi.Context(nx, ny, nz, c.lx, c.ly, c.lz, c.bc, c.gravity, c.n_cells, c.theta, precision=precision)


@pytest.mark.parametrize("shape,iters,precision,per_iteration", [
    ((12, 8, 8), 3, F64, 2), ((12, 8, 8), 3, MIX, 2), ((33, 17, 9), 3, F64, 2), ((33, 17, 9), 3, MIX, 2),
    ((17, 40, 33), 3, F64, 2), ((128, 9, 8), 3, MIX, 2), ((64, 64, 1), 3, F64, 2), ((64, 65, 1), 3, MIX, 2),
    ((31, 63, 40), 2, MIX, 2), ((96, 41, 32), 2, F64, 2),
    ((63, 63, 64), 2, F64, 4), ((126, 64, 33), 2, F64, 4), ((64, 63, 65), 2, F64, 4), ((250, 63, 256), 1, MIX, 4)])
def test_reinit_kernels(shape, iters, precision, per_iteration):
    c, phi, ctx = _case(shape, precision)
    n = []
    for it in (iters, iters + 1):
        a = wsi.launch_count()
        got = np.asarray(ctx.reinit(phi.ravel(), it))
        n.append(wsi.launch_count() - a)
        if it == iters:
            ref = ori.reinit(Grid(*shape, c.lx, c.ly, c.lz), phi, iters).ravel()
            assert np.abs(got - ref).max() < TOL[precision] * np.abs(ref).max()
    ctx.close()
    assert n[1] - n[0] == per_iteration
