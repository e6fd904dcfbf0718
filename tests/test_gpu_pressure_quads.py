"""The float32 pressure multigrid with four cells per thread (rows of a
multiple of four cells) against the one-cell kernels: the same problem with its
axes exchanged takes the other path on the finest level or below.  Red-black
colouring, coarsening and transfers are symmetric under an exchange of axes,
so three V-cycles give the same iterate up to rounding: float32 corrections of
relative size 1 in the first cycle, some tens of roundings of 6e-8 each, so
1e-5 of the solution; float64 contexts 1e-12."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1901_07892_gb300 import wsi

TOL = {wsi.PREC_MIXED: 1e-5, wsi.PREC_FP64: 1e-12}


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()


def _solve(prec, phi, y, perm, L, cycles):
    a = np.ascontiguousarray(phi.transpose(perm))
    nz, ny, nx = a.shape
    lz, ly, lx = (L[p] for p in perm)
    ctx = wsi.Context(nx, ny, nz, lx, ly, lz, precision=prec)
    ctx.set_phases(a, np.ones_like(a), 1000.0, 1.2, 500.0, 1e-3, 1.8e-5, 1e-3)
    x, st = wsi.pressure_solve(ctx, np.ascontiguousarray(y.transpose(perm)).ravel(), rtol=1e-30, max_cycles=cycles)
    ctx.close()
    return x.reshape(a.shape).transpose(np.argsort(perm))


@pytest.mark.parametrize("prec", [wsi.PREC_MIXED, wsi.PREC_FP64])
@pytest.mark.parametrize("shape", [(10, 6, 4), (10, 8, 20), (6, 4, 36), (14, 10, 12), (6, 10, 256)])
def test_exchanged_axes(prec, shape):
    rng = np.random.default_rng(4)
    h = 0.05
    L = [n * h for n in shape]
    z, yy, xx = np.meshgrid(*[(np.arange(n) + 0.5) * h for n in shape], indexing="ij")
    phi = z - 0.5 * L[0] + 0.06 * np.sin(5 * xx) * np.cos(3 * yy)
    y = rng.uniform(-1, 1, shape)
    y -= y.mean()
    ref = _solve(prec, phi, y, (0, 1, 2), L, 3)
    for perm in ((2, 1, 0), (0, 2, 1)):
        got = _solve(prec, phi, y, perm, L, 3)
        err = np.abs(got - ref).max() / np.abs(ref).max()
        print(shape, perm, err)
        assert err < TOL[prec]
