"""The float64 smoother's stored inverse diagonals follow the time step: one
context that solves with two time steps in turn gives, to the bit, what a fresh
context gives for each (the sums are deterministic).  Also on grids with one
cell in z, with odd extents and with an open top."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1901_07892_gb300 import inputs, wsi


@pytest.mark.parametrize("shape,open_top", [((16, 12, 8), 0), ((15, 9, 1), 0), ((12, 10, 6), 1)])
def test_diagonal_follows_dt(shape, open_top):
    nx, ny, nz = shape
    bc = (-1.0,) * 4 + ((1.0, 1.0) if nz == 1 else (-1.0, -1.0))
    c = inputs.Case(nx=nx, ny=ny, nz=nz, lx=1.0, ly=0.9, lz=0.8, bc=bc)
    x, y, z = c.cell_xyz()
    c.phi = np.broadcast_to(y + 0.4 * z - 0.6 + 0.05 * np.sin(7 * x), (nz, ny, nx)).copy()
    c.psi = np.ones_like(c.phi)

    def make():
        ctx = wsi.Context(nx, ny, nz, c.lx, c.ly, c.lz, bc, c.gravity, c.n_cells, c.theta, open_top=open_top)
        ctx.set_phases(c.phi, c.psi, c.rho_l, c.rho_g, c.rho_s, c.mu_l, c.mu_g, c.mu_s)
        return ctx

    one = make()
    b = torch.from_numpy(np.random.default_rng(1).standard_normal(one.nstk)).cuda()
    b = one.apply(wsi.OP_STOKES, b, 1e-3).clone()  # a consistent right-hand side
    for dt in (1e-3, 5e-2, 1e-3):
        got, sg = one.solve(b, dt, rtol=1e-8, max_iters=100)
        ctx = make()
        ref, sr = ctx.solve(b, dt, rtol=1e-8, max_iters=100)
        ctx.close()
        assert sg.iters == sr.iters
        assert torch.equal(got, ref)
    one.close()
