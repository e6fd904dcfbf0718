"""The float32 multigrid kernels with four cells per thread (k_rbgs_p4,
k_restrict_res4, k_prolong_add4) on the levels that use them: grids above 65536
cells, below which a whole cycle is one launch of another kernel.  Each problem is
solved with its axes in several orders: rows of a multiple of four cells take the
four-cell kernels, rows of 34, 66 or 33 cells the one-cell kernels, on the finest
level or on the second, and red-black colouring, coarsening and transfers are
symmetric under an exchange of axes.  The measure is the float64 context, which
has no four-cell kernels.  After three V-cycles the iterates agree up to rounding:
float32 corrections of relative size 1 in the first cycle, some tens of roundings
of 6e-8 each, so 1e-5 of the solution; float64 against itself 1e-12.  The launch
count shows that the levels above the fused ones had launches of their own (four
half sweeps on either side, restriction and prolongation)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1901_07892_gb300 import wsi


def _solve(prec, phi, y, perm, L, cycles, open_top):
    a = np.ascontiguousarray(phi.transpose(perm))
    nz, ny, nx = a.shape
    lz, ly, lx = (L[p] for p in perm)
    ctx = wsi.Context(nx, ny, nz, lx, ly, lz, precision=prec, open_top=open_top)
    ctx.set_phases(a, np.ones_like(a), 1000.0, 1.2, 500.0, 1e-3, 1.8e-5, 1e-3)
    rhs = np.ascontiguousarray(y.transpose(perm)).ravel()
    wsi.pressure_solve(ctx, rhs, rtol=1e-30, max_cycles=1)  # set-up
    n = []
    for c in (cycles - 1, cycles):
        l0 = wsi.launch_count()
        x, st = wsi.pressure_solve(ctx, rhs, rtol=1e-30, max_cycles=c)
        n.append(wsi.launch_count() - l0)
    ctx.close()
    return x.reshape(a.shape).transpose(np.argsort(perm)), n[1] - n[0]


@pytest.mark.parametrize("shape,perms,open_top,levels", [
    ((64, 64, 34), ((0, 1, 2), (2, 1, 0), (0, 2, 1)), 0, 1),
    ((64, 80, 132), ((0, 1, 2), (2, 1, 0), (0, 2, 1)), 0, 2),
    ((96, 80, 128), ((0, 1, 2), (1, 0, 2)), 0, 2),
    ((40, 64, 66), ((0, 1, 2), (0, 2, 1)), 1, 1)])
def test_large_levels(shape, perms, open_top, levels):
    rng = np.random.default_rng(4)
    h = 0.05
    L = [n * h for n in shape]
    z, yy, xx = np.meshgrid(*[(np.arange(n) + 0.5) * h for n in shape], indexing="ij")
    phi = z - 0.5 * L[0] + 0.06 * np.sin(5 * xx) * np.cos(3 * yy)
    y = rng.uniform(-1, 1, shape)
    if not open_top:
        y -= y.mean()
    ref = None
    for perm in perms:
        for prec, tol in ((wsi.PREC_FP64, 1e-12), (wsi.PREC_MIXED, 1e-5)):
            got, launches = _solve(prec, phi, y, perm, L, 3, open_top)
            if ref is None:
                ref = got
            err = np.abs(got - ref).max() / np.abs(ref).max()
            print(shape, perm, prec, err, launches)
            assert err < tol
            assert launches >= 10 * levels + 4
