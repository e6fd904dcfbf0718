"""Operator, transport and level-set calls read and write device arrays in
place of staging copies where they can.  The results are the same, to the bit,
for host arrays, device arrays, device arrays off the 16-byte alignment, and
outputs that lie on an input."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1901_07892_gb300 import inputs, wsi


def _ctx(precision, shape=(18, 11, 9)):
    nx, ny, nz = shape
    c = inputs.Case(nx=nx, ny=ny, nz=nz, lx=1.0, ly=0.9, lz=0.8)
    x, y, z = c.cell_xyz()
    c.phi = np.broadcast_to(z - 0.4 + 0.05 * np.sin(7 * x), (nz, ny, nx)).copy()
    c.psi = np.ones_like(c.phi)
    ctx = wsi.Context.from_case(c, precision=precision)
    ctx.set_case(c, with_body=False)
    return ctx, c


def _shifted(a):
    """a on the device, eight bytes off the alignment"""
    buf = torch.empty(a.size + 3, dtype=torch.float64, device="cuda")
    out = buf[1:1 + a.size]
    out.copy_(torch.from_numpy(a))
    assert out.data_ptr() % 16 == 8
    return out


@pytest.mark.parametrize("precision", [wsi.PREC_FP64, wsi.PREC_MIXED])
def test_where_arrays_lie(precision):
    ctx, c = _ctx(precision)
    rng = np.random.default_rng(0)
    places = [lambda a: a.copy(), lambda a: torch.from_numpy(a).cuda(), _shifted]
    host = lambda t: t.cpu().numpy() if isinstance(t, torch.Tensor) else np.asarray(t)
    nin = {wsi.OP_STOKES: ctx.nstk, wsi.OP_VISCOUS: ctx.nvel, wsi.OP_STRAIN: ctx.nvel, wsi.OP_PRESSURE: ctx.ncell,
           wsi.OP_GRAD: ctx.ncell, wsi.OP_DIV: ctx.nvel}
    nout = {wsi.OP_STOKES: ctx.nstk, wsi.OP_VISCOUS: ctx.nvel, wsi.OP_STRAIN: ctx.nvel, wsi.OP_PRESSURE: ctx.ncell,
            wsi.OP_GRAD: ctx.nvel, wsi.OP_DIV: ctx.ncell}
    for op in nin:
        a = rng.standard_normal(nin[op])
        ref, *other = [host(ctx.apply(op, p(a), 1e-3)) for p in places]
        for o in other:
            assert np.array_equal(ref, o)
        # on the input, and a few entries into it
        for off in (0, 2):
            buf = torch.zeros(nin[op] + nout[op], dtype=torch.float64, device="cuda")
            buf[:nin[op]] = torch.from_numpy(a).cuda()
            torch.cuda.synchronize()
            out = buf[off:off + nout[op]]
            rc = ctx.L.wsi_apply(ctx._h, op, ctypes.c_void_p(buf.data_ptr()), ctypes.c_void_p(out.data_ptr()),
                                 ctypes.c_double(1e-3))
            assert rc == wsi.OK
            assert np.array_equal(ref, host(out))
    u = [rng.uniform(-0.2, 0.2, ctx.nvel) for _ in range(3)]
    for k in (0, 1):
        ref, *other = [[host(t) for t in ctx.transport(*[p(a) for a in u], k, 1e-3)] for p in places]
        for o in other:
            assert np.array_equal(ref[0], o[0]) and np.array_equal(ref[1], o[1])
    phi = [c.phi.ravel() + 0.01 * rng.standard_normal(c.phi.size) for _ in range(2)]
    ref, *other = [host(ctx.advect_levelset(p(u[0]), p(phi[0]), p(phi[1]), 1e-3)) for p in places]
    for o in other:
        assert np.array_equal(ref, o)
    buf = torch.from_numpy(phi[0]).cuda()
    args = [torch.from_numpy(u[0]).cuda(), buf, torch.from_numpy(phi[1]).cuda()]
    torch.cuda.synchronize()
    rc = ctx.L.wsi_advect_levelset(ctx._h, *[ctypes.c_void_p(t.data_ptr()) for t in args], ctypes.c_double(1e-3),
                                   ctypes.c_void_p(buf.data_ptr()))
    assert rc == wsi.OK and np.array_equal(ref, host(buf))
    ctx.close()
