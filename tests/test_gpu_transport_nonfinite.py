"""Infinite and NaN entries in the float64 transport kernel, whose limiter folds
its cases into two factors and compares bit patterns: they spread exactly as far
as with the cases written out (below, in numpy; the oracle's form in normalized
variables has a quotient by the infinite difference and is not the measure here).
The entries are far enough from the walls that no wall flux (velocity zero) meets
them.  Tolerance of the operator where both are finite: 1e-11 of the scale."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import transport as otr
from oracle.grid import Grid
from oracle.materials import Materials
from paper_1901_07892_gb300 import inputs, wsi


def _cui(qU, qC, qD):
    den, num = qD - qU, qC - qU
    a, D = np.where(den > 0, num, -num), np.where(den > 0, den, -den)
    f = np.where((a > 0) & (13 * a <= 2 * D), 3 * num,
                 np.where((13 * a > 2 * D) & (5 * a <= 4 * D), num * (5 / 6) + den * (1 / 3),
                          np.where((5 * a > 4 * D) & (a <= D), den, num)))
    return np.where(den == 0, qC, qU + f)


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("comp", [0, 1, 2])
def test_nonfinite_entries(comp, bad, monkeypatch):
    nx, ny, nz = 45, 40, 38
    c = inputs.Case(nx=nx, ny=ny, nz=nz, lx=1.0, ly=0.9, lz=0.8, bc=(-1.0,) * 6)
    x, y, z = c.cell_xyz()
    rng = np.random.default_rng(8)
    c.phi = np.broadcast_to(y + 0.4 * z - 0.6 + 0.05 * np.sin(7 * x), (nz, ny, nx)).copy()
    c.psi = np.ones_like(c.phi)
    g = Grid(nx, ny, nz, c.lx, c.ly, c.lz, c.bc)
    mk = lambda: [rng.uniform(-1, 1, g.face_shape(d)) * 0.3 * g.interior_face_mask(d) for d in range(3)]
    un, unm1 = mk(), mk()
    for k, j, i in ((16, 17, 20), (16, 22, 24), (21, 17, 24), (21, 22, 20), (18, 20, 22)):
        un[comp][k, j, i] = bad
    flat = lambda v: np.concatenate([a.ravel() for a in v])
    ctx = wsi.Context.from_case(c)
    ctx.set_case(c, with_body=False)
    got = ctx.transport(flat(un), flat(unm1), None, 0, 1e-3)
    ctx.close()
    monkeypatch.setattr(otr, "cui", _cui)
    m = Materials(g, c.phi, c.psi, c.rho_l, c.rho_g, c.rho_s, c.mu_l, c.mu_g, c.mu_s, c.n_cells)
    with np.errstate(all="ignore"):
        ref = otr.ssp_rk3(g, m.rho_face, un, *otr.rk_velocities(un, unm1, None, 0), 1e-3)
    for a, b in zip(got, ref):
        b = flat(b)
        fa, fb = np.isfinite(a), np.isfinite(b)
        assert 0 < (~fb).sum() < 0.5 * b.size
        assert np.array_equal(fa, fb), (int((~fa).sum()), int((~fb).sum()))
        assert np.abs(a[fa] - b[fa]).max() < 1e-11 * np.abs(b[fb]).max()
