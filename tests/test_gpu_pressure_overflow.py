"""A right-hand side whose residual cannot be measured in float64 (its square sum
overflows, or its sum does in one order of summation and not in another, or it
holds an infinity or a NaN) ends the pressure solve with the
error for non-finite values, in a closed box and with an open top; it is not
taken for a residual of zero."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1901_07892_gb300 import wsi


@pytest.mark.parametrize("prec", [wsi.PREC_MIXED, wsi.PREC_FP64])
@pytest.mark.parametrize("open_top", [0, 1])
@pytest.mark.parametrize("what", ["1e180", "alternating 1.1e307", "one 1e200", "inf", "inf and -inf", "nan"])
def test_not_measurable(what, open_top, prec):
    nx, ny, nz = 20, 16, 12
    ctx = wsi.Context(nx, ny, nz, 1.0, 0.8, 0.6, precision=prec, open_top=open_top)
    z = (np.arange(nz) + 0.5)[:, None, None] * 0.05
    phi = np.ascontiguousarray(np.broadcast_to(z - 0.3, (nz, ny, nx)))
    ctx.set_phases(phi, np.ones_like(phi), 1000.0, 1.2, 500.0, 1e-3, 1.8e-5, 1e-3)
    y = np.random.default_rng(5).uniform(-1, 1, nx * ny * nz)
    ok, _ = wsi.pressure_solve(ctx, y, rtol=1e-6)
    assert np.isfinite(np.asarray(ok)).all()
    if what == "1e180":
        y *= 1e180
    elif what == "alternating 1.1e307":
        # ten of a row's columns over two planes overflow to inf, the others to
        # -inf; neighbours cancel
        y = np.where(np.arange(y.size) % 2, -1.1e307, 1.1e307)
    else:
        y[77] = {"one 1e200": 1e200, "inf": np.inf, "inf and -inf": np.inf, "nan": np.nan}[what]
        if what == "inf and -inf":
            y[1234] = -np.inf
    with pytest.raises(wsi.WsiError) as e:
        wsi.pressure_solve(ctx, y, rtol=1e-6)
    assert e.value.code == wsi.ERR_NAN
    again, _ = wsi.pressure_solve(ctx, torch.from_numpy(np.random.default_rng(5).uniform(-1, 1, nx * ny * nz)).cuda(), rtol=1e-6)
    ctx.close()
    assert np.array_equal(again.cpu().numpy(), np.asarray(ok))
