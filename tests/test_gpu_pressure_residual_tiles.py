"""The pressure solve's fused residual (tiles of 32 x 8 cells, the fluxes through a
tile's upper x and y edges from a warp of their own) where the last tile ends on
the wall or has one column or row, in a closed box and with an open top, and on a
grid of many tiles, where a block marches over more than two planes and hands the
z-flux on: the relative residual that the solve reports equals that of the
returned pressure under the operator entry point, which has a kernel of its own.
The two differ by the float64 rounding of L x, about eps |L| |x| / |y| < 1e-12 for
these grids, and the residuals are 1e-4 and below, so 1e-5 of them with room for
the residual being a hundred times smaller."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1901_07892_gb300 import wsi


@pytest.mark.parametrize("prec", [wsi.PREC_MIXED, wsi.PREC_FP64])
@pytest.mark.parametrize("shape,open_top", [((64, 16, 8), 0), ((65, 16, 8), 0), ((64, 17, 8), 1), ((65, 16, 4), 1),
                                            ((33, 8, 9), 0), ((96, 24, 3), 0), ((128, 160, 36), 0),
                                            ((128, 160, 36), 1)])
def test_reported_residual(shape, open_top, prec):
    nx, ny, nz = shape
    h = 0.05
    ctx = wsi.Context(nx, ny, nz, nx * h, ny * h, nz * h, precision=prec, open_top=open_top)
    x = np.arange(nx) * h
    y = np.arange(ny)[:, None] * h
    z = np.arange(nz)[:, None, None] * h
    phi = np.ascontiguousarray(np.broadcast_to(y + 0.3 * z + 0.1 * np.sin(4 * x) - 0.5 * ny * h, (nz, ny, nx)))
    ctx.set_phases(phi, np.ones_like(phi), 1000.0, 1.2, 500.0, 1e-3, 1.8e-5, 1e-3)
    rhs = torch.from_numpy(np.random.default_rng(2).standard_normal(nx * ny * nz)).cuda()
    sol, st = wsi.pressure_solve(ctx, rhs.clone(), rtol=1e-4, max_cycles=300)
    if not open_top:
        rhs = rhs - rhs.mean()
    r = rhs - ctx.apply(wsi.OP_PRESSURE, sol)
    if not open_top:
        r = r - r.mean()
    ctx.close()
    rel = float(r.norm() / rhs.norm())
    assert st.rel_residual <= 1e-4
    assert abs(rel - st.rel_residual) <= 1e-5 * max(st.rel_residual, 1e-6)
