"""The dense inverse of the coarsest multigrid level, formed on the device up to 160
cells: grids that are a single level (no axis can be halved, or at most 64 cells),
with row counts around multiples of the warp, so that one V-cycle is one product with
the inverse.  What is left of the right-hand side is rounding: the operator of one
phase has a condition number below (2 n / pi)^2 = 1100 for the longest extent (53),
so float64 leaves less than 160 x 1100 x 1e-16 = 2e-11 (held to 1e-9) and a float32
iterate less than 1100 x 6e-8 = 7e-5 (held to 1e-3)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1901_07892_gb300 import wsi


@pytest.mark.parametrize("prec,tol", [(wsi.PREC_FP64, 1e-9), (wsi.PREC_MIXED, 1e-3)])
@pytest.mark.parametrize("n,open_top", [((2, 2, 2), 0), ((3, 11, 1), 0), ((4, 4, 4), 0), ((4, 4, 4), 1), ((5, 13, 1), 0),
                                        ((5, 5, 5), 0), ((5, 5, 5), 1), ((11, 7, 2), 0), ((3, 53, 1), 0)])
def test_single_level(n, open_top, prec, tol):
    nx, ny, nz = n
    h = 0.05
    bc = (-1.0,) * 4 + ((1.0,) * 2 if nz == 1 else (-1.0,) * 2)
    ctx = wsi.Context(nx, ny, nz, nx * h, ny * h, nz * h, precision=prec, bc=bc, open_top=open_top)
    one = np.ones((nz, ny, nx))
    ctx.set_phases(one, one, 1000.0, 1.2, 500.0, 1e-3, 1.8e-5, 1e-3)
    y = np.random.default_rng(5).uniform(-1, 1, nx * ny * nz)
    if not open_top:
        y -= y.mean()
    _, st = wsi.pressure_solve(ctx, y, rtol=1e-30, max_cycles=1)
    ctx.close()
    print(n, prec, st.rel_residual)
    assert st.iters == 1 and 0 <= st.rel_residual < tol
