"""Edges of the transport kernel's tiles (32 x 8 faces marched in z) against
the oracle, in both precisions: extents that are a multiple of the tile, where
the wall column or row has no tile of its own; one face more and one less; one
cell in z (a march of one or two planes); fewer planes than the ring has slots.
Tolerances of the operator: float64 1e-11; float32 arithmetic 1e-6 of rho and
1e-5 of the convective term's scale (differences of float32 fluxes)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.materials import Materials
from oracle import transport as otr
from oracle.grid import Grid
from paper_1901_07892_gb300 import inputs, wsi


@pytest.mark.parametrize("precision", [wsi.PREC_FP64, wsi.PREC_MIXED])
@pytest.mark.parametrize("shape,k", [((32, 8, 4), 0), ((64, 16, 5), 1), ((31, 7, 3), 1), ((33, 9, 1), 0),
                                     ((32, 8, 1), 1), ((2, 2, 2), 0), ((65, 24, 35), 1)])
def test_transport_tiles(shape, k, precision):
    nx, ny, nz = shape
    bc = (-1.0,) * 4 + ((1.0, 1.0) if nz == 1 else (-1.0, -1.0))
    c = inputs.Case(nx=nx, ny=ny, nz=nz, lx=1.0, ly=0.9, lz=0.8, bc=bc)
    x, y, z = c.cell_xyz()
    rng = np.random.default_rng(5)
    c.phi = np.broadcast_to(y + 0.4 * z - 0.6 + 0.05 * np.sin(7 * x), (nz, ny, nx)).copy()
    c.psi = np.ones_like(c.phi)
    g = Grid(nx, ny, nz, c.lx, c.ly, c.lz, c.bc)
    ctx = wsi.Context.from_case(c, precision=precision)
    ctx.set_case(c, with_body=False)
    m = Materials(g, c.phi, c.psi, c.rho_l, c.rho_g, c.rho_s, c.mu_l, c.mu_g, c.mu_s, c.n_cells)
    mk = lambda: [rng.uniform(-1, 1, g.face_shape(d)) * 0.3 * g.interior_face_mask(d) for d in range(3)]
    un, unm1, uk = mk(), mk(), mk()
    flat = lambda v: np.concatenate([a.ravel() for a in v])
    rho, C = ctx.transport(flat(un), flat(unm1), flat(uk), k, 1e-3)
    ctx.close()
    u1, u2 = otr.rk_velocities(un, unm1, uk, k)
    r3, Co = otr.ssp_rk3(g, m.rho_face, un, u1, u2, 1e-3)
    rel = lambda a, b: np.abs(a - b).max() / max(np.abs(b).max(), 1e-300)
    tr, tc = (1e-11, 1e-11) if precision == wsi.PREC_FP64 else (1e-6, 1e-5)
    assert rel(rho, flat(r3)) < tr
    assert rel(C, flat(Co)) < tc
