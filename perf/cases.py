"""The calls whose speed matters, each through the public binding (paper_1901_07892_gb300.wsi).

A case is a dict of plain values: ``kind`` names the entry point, ``nx, ny,
nz`` the grid, ``precision`` the context's precision, the rest are options of
that entry point.  ``listed()`` holds the fixed ones, ``draw(rng)`` gives
others of the same ranges, ``prepare(case, seed)`` what a program has in hand
before the call, ``run(state)`` one pass, ``work(case)`` the bytes and
operations a pass cannot do without, ``exact(case, seed)`` the result in
float64 from plain torch where there is one.

Geometry, material values and sizes are those of the repository's own
workloads (inputs.py, bench.py, wave_validation.py): air over water with a
sloshing surface, a locked box, a free cylinder, a submerged bar.
"""
import math

import numpy as np
import torch

from paper_1901_07892_gb300 import inputs, wsi

F64 = torch.float64
RHO = (1000.0, 1.2)      # liquid, gas
MU = (1e-3, 1.8e-5, 1e-3)  # liquid, gas, solid
DT = 5e-4


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest call: one 2-D implicit solve of the plain path (launches and host work count)
        dict(name="solve_2d_64", kind="solve", nx=64, ny=64, nz=1, precision="fp64", rtol=1e-10),
        # a small three-phase step, as in parameter studies: launch-bound on every level
        dict(name="step_tank_40x32x48", kind="step", body="box", nx=40, ny=32, nz=48, precision="mixed"),
        # the benchmark's time step
        dict(name="step_tank_256", kind="step", body="box", nx=256, ny=256, nz=256, precision="mixed"),
        # the wave tank with its submerged bar on the plain float64 path
        dict(name="step_bar_128x64x64_fp64", kind="step", body="bar", nx=128, ny=64, nz=64, precision="fp64"),
        # the largest configuration: a free cylinder in a regular wave
        dict(name="step_cylinder_512x256x256", kind="step", body="cylinder", nx=512, ny=256, nz=256,
             precision="mixed"),
        # the operator alone on a ragged grid (no extent a power of two), mixed path
        dict(name="apply_250x182x126", kind="apply", nx=250, ny=182, nz=126, precision="mixed"),
        # consistent mass and momentum transport alone, ragged
        dict(name="transport_250x126x130", kind="transport", nx=250, ny=126, nz=130, precision="mixed"),
        # the wave validation's slab (four cells thick), xsPPM7 limiter
        dict(name="advect_1024x4x128", kind="advect", nx=1024, ny=4, nz=128, precision="mixed", limiter="xsppm7"),
        # bringing the benchmark's surface back to a signed distance
        dict(name="reinit_256", kind="reinit", nx=256, ny=256, nz=256, precision="mixed", iters=10),
        # the rigidity projection with the wave tank's 1.5 million markers
        dict(name="rigid_256x128x128", kind="rigid", nx=256, ny=128, nz=128, precision="mixed"),
        # the pressure sub-problem to 1e-8 (the learned part's yardstick)
        dict(name="pressure_256", kind="pressure", nx=256, ny=256, nz=256, precision="mixed", rtol=1e-8),
        # one gradient of the correction network, 16/32/64 channels
        dict(name="train_64", kind="train", nx=64, ny=64, nz=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mg_size(rng, lo, hi):
    """An extent the multigrid hierarchy takes: 2, 3 or 5 times a power of two."""
    n = [m << p for m in (2, 3, 5) for p in range(2, 8)]
    n = [v for v in n if lo <= v <= hi]
    return rng.choice(n)


def draw(rng):
    kind = rng.choice(["solve", "step", "step", "apply", "transport", "advect", "reinit", "rigid", "pressure", "train"])
    prec = "mixed" if rng.random() < 0.65 else "fp64"
    hi = 256 if prec == "mixed" else 128
    if kind == "train":
        return dict(kind=kind, nx=4 * rng.randint(2, 18), ny=4 * rng.randint(2, 18), nz=4 * rng.randint(2, 16))
    if kind in ("solve", "pressure", "step"):
        if kind == "solve" and rng.random() < 0.3:
            n = rng.choice([16, 32, 48, 80, 96, 128])
            return dict(kind=kind, nx=n, ny=n, nz=1, precision="fp64", rtol=rng.choice([1e-8, 1e-10]))
        if kind == "step" and rng.random() < 0.5:
            body = rng.choice(["bar", "cylinder"])  # the cylinder's radius is at least 3.6 cells
            n = _mg_size(rng, 24 if body == "bar" else 48, min(hi, 160))
            return dict(kind=kind, body=body, nx=2 * n, ny=n, nz=n, precision=prec)
        n = _mg_size(rng, 16, hi)  # the cells of a unit cube stay within 1:1.5
        near = [_mg_size(rng, n / 1.5, min(hi, 1.5 * n)) for _ in range(2)]
        c = dict(kind=kind, nx=n, ny=near[0], nz=near[1], precision=prec)
        if kind == "step":
            return dict(c, body="box")
        return dict(c, rtol=rng.choice([1e-8, 1e-10]) if kind == "solve" else 1e-8)
    c = dict(kind=kind, nx=_log_int(rng, 12, hi), ny=_log_int(rng, 8, hi), nz=_log_int(rng, 8, hi), precision=prec)
    if kind == "advect":
        c["limiter"] = rng.choice(["cui", "xsppm7"])
    if kind == "reinit":
        c["iters"] = rng.randint(2, 12)
    if kind == "rigid":
        n = _log_int(rng, 24, 128)
        c.update(nx=rng.randint(int(1.6 * n), 2 * n), ny=n, nz=rng.randint(int(0.8 * n), n))
    return c


# ------------------------------------------------------------------ inputs
def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gen(seed):
    g = torch.Generator(device=_dev())
    g.manual_seed(int(seed) + 1)
    return g


def _lengths(case):
    """Box extents: the unit cube, a slab of equal spacings, or the 4:1:1 wave tank."""
    if case["kind"] == "advect":
        return case["nx"] / case["nz"], case["ny"] / case["nz"], 1.0
    if case.get("body") in ("bar", "cylinder") or case["kind"] == "rigid":
        return (8.0, 2.0, 2.0) if case.get("body") == "cylinder" else (4.0, 1.0, 1.0)
    return (1.0, 1.0, 1.0 / case["nx"]) if case["nz"] == 1 else (1.0, 1.0, 1.0)


def _cells(case, dev):
    L, n = _lengths(case), (case["nx"], case["ny"], case["nz"])
    ax = [(torch.arange(n[d], dtype=F64, device=dev) + 0.5) * (L[d] / n[d]) for d in range(3)]
    return ax[0].view(1, 1, -1), ax[1].view(1, -1, 1), ax[2].view(-1, 1, 1)


def _surface(case, seed, depth, amp):
    """Signed distance estimate z - depth - eta to a seeded sloshing surface
    (eight cosine modes, amplitudes summing to at most amp)."""
    x, y, z = _cells(case, _dev())
    L = _lengths(case)
    eta = inputs.fourier_surface(np.random.default_rng(seed), amp=amp)
    e = torch.from_numpy(np.ascontiguousarray(eta(x.cpu().numpy() / L[0], y.cpu().numpy() / L[1]))).to(z.device)
    return (z - depth - e).expand(case["nz"], case["ny"], case["nx"]).contiguous()


def _box_psi(case, center, half):
    q = [(a - center[d]).abs() - half[d] for d, a in enumerate(_cells(case, _dev()))]
    out = (q[0].clamp(min=0) ** 2 + q[1].clamp(min=0) ** 2 + q[2].clamp(min=0) ** 2).sqrt()
    return out + torch.maximum(torch.maximum(q[0], q[1]), q[2]).clamp(max=0)


def _spacing(case):
    L = _lengths(case)
    return L[0] / case["nx"], L[1] / case["ny"], L[2] / case["nz"]


def _tank(case, seed):
    """phi, psi and the body of a case, device tensors (the geometry of inputs.py)."""
    kind, body = case["kind"], case.get("body", "box")
    if case["nz"] == 1:
        c = inputs.tank2d(case["nx"])
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(_dev())  # noqa: E731
        return t(c.phi), t(c.psi), dict(markers=t(c.markers), dV=c.dV, box_half=c.box_half)
    if kind == "rigid" or body == "bar":
        c = inputs.wave_tank(nx=case["nx"], ny=case["ny"], nz=case["nz"])
        X = torch.from_numpy(c.markers).to(_dev())
        psi = torch.from_numpy(np.ascontiguousarray(c.psi)).to(_dev())
        return _surface(case, seed, 0.5, 0.02), psi, dict(markers=X, dV=c.dV)
    h = _spacing(case)
    if body == "cylinder":
        x, y, z = _cells(case, _dev())
        r, hl, ctr = 0.15, 0.8, (4.0, 1.0, 1.0)
        qr, qy = ((x - ctr[0]) ** 2 + (z - ctr[2]) ** 2).sqrt() - r, (y - ctr[1]).abs() - hl
        psi = (qr.clamp(min=0) ** 2 + qy.clamp(min=0) ** 2).sqrt() + torch.maximum(qr, qy).clamp(max=0)
        X, dV = inputs.cylinder_lattice(ctr, r, hl, h)
        b = dict(markers=torch.from_numpy(X).to(_dev()), dV=dV, lock=(0, 1, 0, 1, 0, 1), cylinder=(r, hl))
        return _surface(case, seed, 1.0, 0.02), psi, b
    ctr, half = (0.5, 0.5, 0.6), (0.1, 0.1, 0.05)
    if kind == "advect":
        return _surface(case, seed, 0.6, 0.05), torch.ones(case["nz"], case["ny"], case["nx"], dtype=F64, device=_dev()), {}
    X, dV = inputs.marker_lattice(ctr, half, h)
    b = dict(markers=torch.from_numpy(X).to(_dev()), dV=dV, box_half=half)
    return _surface(case, seed, 0.6, 0.05), _box_psi(case, ctr, half), b


def _bc(case):
    if case["nz"] == 1:
        return (-1.0,) * 4 + (1.0, 1.0)
    if case["kind"] == "advect":
        return (-1.0, -1.0, 1.0, 1.0, -1.0, -1.0)
    return (-1.0,) * 6


def _rho_s(case):
    return 500.0 if case.get("body") == "cylinder" else RHO[0]


def _context(case, seed, body=True):
    L = _lengths(case)
    grav = (0.0, -9.81, 0.0) if case["nz"] == 1 else (0.0, 0.0, -9.81)
    ctx = wsi.Context(case["nx"], case["ny"], case["nz"], *L, bc=_bc(case), gravity=grav,
                      precision=wsi.PREC_MIXED if case["precision"] == "mixed" else wsi.PREC_FP64,
                      ls_limiter=wsi.LIMIT_XSPPM7 if case.get("limiter") == "xsppm7" else wsi.LIMIT_CUI)
    phi, psi, b = _tank(case, seed)
    full = case.get("body") == "cylinder"
    ctx.set_phases(phi, psi, RHO[0], RHO[1], _rho_s(case), *MU,
                   gravity_mode=wsi.GRAVITY_FULL if full else wsi.GRAVITY_FLOW, **(b if body else {}))
    return ctx, phi, psi, b


def _shape(case, c):
    s = [case["nz"], case["ny"], case["nx"]]
    if c < 3:
        s[2 - c] += 1
    return tuple(s)


def _split(case, a, parts=3):
    """Packed vector -> its face (and cell) arrays."""
    out, o = [], 0
    for c in range(parts):
        s = _shape(case, c)
        n = s[0] * s[1] * s[2]
        out.append(a[..., o:o + n].reshape(a.shape[:-1] + s))
        o += n
    return out


def _pack(parts):
    return torch.cat([p.reshape(-1) for p in parts])


def _velocity(case, seed, umax=0.5):
    """A discretely divergence-free velocity that vanishes normal to the
    walls: the discrete curl of seeded smooth potentials on the edges."""
    dev, n, h = _dev(), (case["nx"], case["ny"], case["nz"]), _spacing(case)
    rng = np.random.default_rng(seed)

    def axis(d, nodes):
        t = torch.arange(n[d] + 1, dtype=F64, device=dev) / n[d] if nodes else (torch.arange(n[d], dtype=F64, device=dev) + 0.5) / n[d]
        return t.view(*[-1 if a == 2 - d else 1 for a in range(3)])

    def potential(c):
        ax = [axis(d, d != c) for d in range(3)]
        win = 1.0
        for d in range(3):
            if d != c:
                win = win * torch.sin(math.pi * ax[d])
        s = 0.0
        for _ in range(4):
            k, p = rng.integers(1, 4, 3), rng.uniform(0, 2 * math.pi, 3)
            m = float(rng.standard_normal())
            for d in range(3):
                m = m * torch.cos(math.pi * int(k[d]) * ax[d] + float(p[d]))
            s = s + m
        return s * win

    A = [potential(c) for c in range(3)]
    d = lambda a, ax: a.diff(dim=2 - ax) / h[ax]  # noqa: E731
    u = [d(A[2], 1) - d(A[1], 2), d(A[0], 2) - d(A[2], 0), d(A[1], 0) - d(A[0], 1)]
    for c in range(3):  # rounding of sin(pi) at the far walls
        u[c].narrow(2 - c, 0, 1).zero_()
        u[c].narrow(2 - c, n[c], 1).zero_()
    top = max(float(q.abs().max()) for q in u)
    return _pack(u) * (umax / top)


def _waves(case):
    if case.get("body") == "bar":
        return dict(H=0.05, T=1.0, depth=0.5, x_gen=0.5, x_damp=3.5)
    return dict(H=0.1, T=1.2, depth=1.0, x_gen=1.0, x_damp=7.0)


def _step_dt(case):
    return {"box": DT, "bar": 2.56 / case["nx"], "cylinder": 1.28 / case["nx"]}[case["body"]]


def _train_sizes():
    return [(16, 16), (16, 16), (32, 16), (32, 32), (64, 32), (64, 64), (32, 96), (32, 32), (16, 48), (16, 16)]


def _train_inputs(case, seed):
    rng = np.random.default_rng(seed)
    s = (case["nz"], case["ny"], case["nx"])
    z = (np.arange(s[0]) + 0.5)[:, None, None] / s[0]
    eta = inputs.fourier_surface(rng)
    phi = z - 0.6 - eta((np.arange(s[2]) + 0.5)[None, None, :] / s[2], (np.arange(s[1]) + 0.5)[None, :, None] / s[1])
    x = np.empty(s + (3,), np.float32)
    x[..., 0] = np.where(phi < 0, math.log(RHO[0]), math.log(RHO[1])) / 7.0
    x[..., 1] = np.clip(10.0 * phi, -4.0, 4.0)
    x[..., 2] = rng.standard_normal(s)
    t = rng.standard_normal(s).astype(np.float32)
    p = []
    for l, (co, ci) in enumerate(_train_sizes()):  # He-normal weights [tap][out][in]; the first layer has 3 inputs
        real = 3 if l == 0 else ci
        w = np.zeros((27, co, ci), np.float32)
        w[:, :, :real] = rng.standard_normal((27, co, real)) * math.sqrt(2.0 / (27 * real))
        p += [w.ravel(), (0.01 * rng.standard_normal(co)).astype(np.float32)]
    p += [(rng.standard_normal(16) * math.sqrt(2.0 / 16)).astype(np.float32), np.zeros(1, np.float32)]
    return x, t, np.concatenate(p).astype(np.float32)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        x, t, p = _train_inputs(case, seed)
        return dict(case=case, net=wsi.UNet(case["nz"], case["ny"], case["nx"], 16, 32, 64), x=x, t=t, p=p)
    ctx, phi, psi, b = _context(case, seed, body=kind != "advect")
    s = dict(case=case, ctx=ctx)
    g = _gen(seed)
    if kind == "step":
        # a moving state: two steps on from rest
        dt = _step_dt(case)
        if case["body"] != "box":
            ctx.set_waves(t0=0.1, **_waves(case))
        for _ in range(2):
            ctx.step(dt)
        s.update(dt=dt)
        if case["body"] != "cylinder":
            for name, f in (("vel", wsi.F_VEL), ("old", wsi.F_VEL_OLD), ("p", wsi.F_P), ("phi", wsi.F_PHI)):
                s[name] = ctx.get_field(f, like=phi)
        s["like"] = phi[:1, :1, :1]
    elif kind == "solve":
        u = (torch.rand(ctx.nvel, dtype=F64, device=_dev(), generator=g) * 2 - 1) * 1e-2
        s["rhs"] = torch.cat([u, torch.zeros(ctx.ncell, dtype=F64, device=_dev())])
    elif kind == "apply":
        s["x"] = torch.randn(ctx.nstk, dtype=F64, device=_dev(), generator=g)
        _zero_walls(case, s["x"])
    elif kind == "transport":
        s["un"] = _velocity(case, seed)
        s["old"] = 0.95 * s["un"] + 0.05 * _velocity(case, seed + 1000003)
    elif kind == "advect":
        s.update(vel=_velocity(case, seed), phi=phi.reshape(-1))
        s["half"] = s["phi"] + 1e-3 * torch.sin(5.0 * s["phi"])
    elif kind == "reinit":
        # distorted away from a distance function, as after advection
        s["phi"] = (phi * (1.0 + 0.3 * torch.sin(7.0 * phi))).reshape(-1).contiguous()
    elif kind == "rigid":
        s["vel"] = _velocity(case, seed)
    elif kind == "pressure":
        y = torch.rand(ctx.ncell, dtype=F64, device=_dev(), generator=g) * 2 - 1
        s["y"] = y - y.mean()
    return s


def _zero_walls(case, x):
    for c, q in enumerate(_split(case, x)):
        q.narrow(q.dim() - 1 - c, 0, 1).zero_()
        q.narrow(q.dim() - 1 - c, q.shape[q.dim() - 1 - c] - 1, 1).zero_()


# ------------------------------------------------------------------ the calls
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "train":
        net = s["net"]
        net.set_params(s["p"])
        out = net.forward(s["x"])
        loss = net.backward(s["t"])
        return dict(out=out, loss=loss, grads=net.grads())
    ctx = s["ctx"]
    if kind == "step":
        if "vel" in s:  # from a given state; a free body's run goes on
            if case["body"] != "box":
                ctx.set_waves(t0=0.1 + 2 * s["dt"], **_waves(case))
            ctx.set_field(wsi.F_VEL, s["vel"])
            ctx.set_field(wsi.F_VEL_OLD, s["old"])
            ctx.set_field(wsi.F_P, s["p"])
            ctx.set_field(wsi.F_PHI, s["phi"])
        ctx.step(s["dt"])
        return dict(vel=ctx.get_field(wsi.F_VEL, like=s["like"]), p=ctx.get_field(wsi.F_P, like=s["like"]),
                    phi=ctx.get_field(wsi.F_PHI, like=s["like"]))
    if kind == "solve":
        x, _ = ctx.solve(s["rhs"], DT, rtol=case["rtol"])
        return x
    if kind == "apply":
        return ctx.apply(wsi.OP_STOKES, s["x"], DT)
    if kind == "transport":
        rho, C = ctx.transport(s["un"], s["old"], None, 0, DT)
        return dict(rho=rho, C=C)
    if kind == "advect":
        return ctx.advect_levelset(s["vel"], s["phi"], s["half"], DT)
    if kind == "reinit":
        return ctx.reinit(s["phi"], case["iters"])
    if kind == "rigid":
        v, b = ctx.dlm_constrain(s["vel"])
        return dict(vel=v, U=list(b.U_r), W=list(b.W_r))
    x, _ = wsi.pressure_solve(ctx, s["y"], rtol=case["rtol"])
    return x


# ------------------------------------------------------------------ the work
def _n_markers(case):
    h = _spacing(case)
    if case["kind"] == "rigid" or case.get("body") == "bar":
        return int(0.3 * (1.0 + 0.182) / 2 / (h[0] * h[2] / 4) * case["ny"] * 2)
    vol = math.pi * 0.15 ** 2 * 1.6 if case.get("body") == "cylinder" else 0.2 * 0.2 * 0.1
    return int(vol / (h[0] * h[1] * h[2] / 8))


def work(case):
    """Bytes: every input read once and every output written once, 8 bytes a
    value (4 for the network); operations: of the operator or stencil."""
    n = [case["nx"], case["ny"], case["nz"]]
    N = n[0] * n[1] * n[2]
    F = sum((n[0] + (c == 0)) * (n[1] + (c == 1)) * (n[2] + (c == 2)) for c in range(3))
    E = sum((n[0] + (e != 2)) * (n[1] + (e != 1)) * (n[2] + (e != 0)) for e in range(3))
    kind = case["kind"]
    matvec = 44 * F + 8 * N
    if kind == "train":
        V = (N, N, N // 8, N // 8, N // 64, N // 64, N // 8, N // 8, N, N)
        fl = sum(2 * 27 * v * co * ci for v, (co, ci) in zip(V, _train_sizes()))
        par = sum(27 * co * ci + co for co, ci in _train_sizes()) + 17
        return dict(bytes=4 * (5 * N + 2 * par), flops=3 * fl)
    if kind == "step":  # u^n, u^{n-1}, p, phi, psi in; u, p, phi out; two solves
        return dict(bytes=8 * (3 * F + 5 * N + 9 * _n_markers(case)), flops=2 * matvec)
    if kind == "solve":
        return dict(bytes=8 * (3 * F + 3 * N + E), flops=matvec)
    if kind == "apply":
        return dict(bytes=8 * (3 * F + 3 * N + E), flops=matvec)
    if kind == "transport":
        return dict(bytes=8 * (4 * F + 2 * N), flops=4 * 60 * F)
    if kind == "advect":
        return dict(bytes=8 * (F + 3 * N), flops=100 * N)
    if kind == "reinit":
        return dict(bytes=8 * 2 * N, flops=2 * case["iters"] * 90 * N)
    if kind == "rigid":
        m = _n_markers(case)
        return dict(bytes=8 * (2 * F + 3 * m), flops=2 * 3 * 64 * 2 * m)
    return dict(bytes=8 * (2 * N + F), flops=20 * N)


# ------------------------------------------------------------------ 64-bit references
def _heaviside(phi, eps):
    t = (phi / eps).clamp(-1, 1)
    return 0.5 * (1 + t + torch.sin(math.pi * t) / math.pi)


def _two_stage(phi, psi, eps, zl, zg, zs):
    zf = zl + (zg - zl) * _heaviside(phi, eps)
    return zs + (zf - zs) * _heaviside(psi, eps)


def _edge_pad(a, ax):
    """One repeated layer on either side along axis ax (x = 0)."""
    d = a.dim() - 1 - ax
    return torch.cat([a.narrow(d, 0, 1), a, a.narrow(d, a.shape[d] - 1, 1)], dim=d)


def _mean(a, ax):
    d = a.dim() - 1 - ax
    n = a.shape[d] - 1
    return 0.5 * (a.narrow(d, 0, n) + a.narrow(d, 1, n))


class _Materials:
    """Face density, cell and edge viscosity of a case (Sec. 4.1)."""

    def __init__(self, case, phi, psi):
        h = _spacing(case)
        eps = 2.0 * (math.sqrt(h[0] * h[1]) if case["nz"] == 1 else (h[0] * h[1] * h[2]) ** (1 / 3))
        rho = lambda a, b: _two_stage(a, b, eps, RHO[0], RHO[1], _rho_s(case))  # noqa: E731
        self.rho = [rho(_mean(_edge_pad(phi, c), c), _mean(_edge_pad(psi, c), c)) for c in range(3)]
        self.mu = _two_stage(phi, psi, eps, *MU)
        inv = 1 / self.mu
        self.mu_e = {}
        for a, b in ((0, 1), (0, 2), (1, 2)):
            self.mu_e[a, b] = 1 / _mean(_mean(_edge_pad(_edge_pad(inv, a), b), a), b)


def _ghost(case, q, ax):
    """q with one ghost layer along the tangential axis ax (the wall's sign)."""
    d, bc = q.dim() - 1 - ax, _bc(case)
    return torch.cat([bc[2 * ax] * q.narrow(d, 0, 1), q, bc[2 * ax + 1] * q.narrow(d, q.shape[d] - 1, 1)], dim=d)


def _matvec(case, m, x, dt):
    """K x of the implicit Stokes system on packed vectors (any leading dimensions)."""
    h = _spacing(case)
    u = _split(case, x, 4)
    p, u = u[3], u[:3]
    d = lambda a, ax: a.diff(dim=a.dim() - 1 - ax) / h[ax]  # noqa: E731
    tau = {}
    for a, b in ((0, 1), (0, 2), (1, 2)):
        tau[a, b] = m.mu_e[a, b] * (d(_ghost(case, u[a], b), b) + d(_ghost(case, u[b], a), a))
    out, lead = [], x.shape[:-1]
    for c in range(3):
        dim, n = u[c].dim() - 1 - c, u[c].shape[u[c].dim() - 1 - c] - 2
        L = d(2 * m.mu * d(u[c], c), c) if n > 0 else None
        if n <= 0:
            out.append(torch.zeros_like(u[c]).reshape(lead + (-1,)))
            continue
        for b in range(3):
            if b != c:
                L = L + d(tau[min(b, c), max(b, c)], b).narrow(dim, 1, n)
        row = (m.rho[c] / dt * u[c]).narrow(dim, 1, n) - 0.5 * L + d(p, c)
        z = torch.zeros_like(u[c].narrow(dim, 0, 1))
        out.append(torch.cat([z, row, z], dim=dim).reshape(lead + (-1,)))
    out.append(-(d(u[0], 0) + d(u[1], 1) + d(u[2], 2)).reshape(lead + (-1,)))
    return torch.cat(out, dim=-1)


def _exact_solve(case, m, rhs):
    """The dense solution of a small system, zero-mean pressure."""
    free = torch.ones_like(rhs)
    _zero_walls(case, free)
    if case["nz"] == 1:
        _split(case, free)[2].zero_()
    idx = free.nonzero().squeeze(1)
    if idx.numel() > 14000:
        return None
    K = torch.empty(idx.numel(), idx.numel(), dtype=F64, device=rhs.device)
    for a in range(0, idx.numel(), 512):
        cols = idx[a:a + 512]
        e = torch.zeros(cols.numel(), rhs.numel(), dtype=F64, device=rhs.device)
        e[torch.arange(cols.numel(), device=e.device), cols] = 1.0
        K[:, a:a + 512] = _matvec(case, m, e, DT)[:, idx].T
    ncell = case["nx"] * case["ny"] * case["nz"]
    b = rhs[idx].clone()
    K[-1].zero_()  # one continuity row gives way to the mean of the pressure
    K[-1, -ncell:] = 1.0
    b[-1] = 0.0
    r = K.abs().amax(dim=1)
    x = torch.zeros_like(rhs)
    lu, piv = torch.linalg.lu_factor(K / r[:, None])
    y = torch.linalg.lu_solve(lu, piv, (b / r)[:, None])
    y = y + torch.linalg.lu_solve(lu, piv, (b / r)[:, None] - (K / r[:, None]) @ y)
    x[idx] = y[:, 0]
    return x


def _cui(qu, qc, qd):
    den, num = qd - qu, qc - qu
    t = torch.where(den != 0, num / torch.where(den != 0, den, torch.ones_like(den)), torch.zeros_like(den))
    f = torch.where((t > 0) & (t <= 2 / 13), 3 * t, t)
    f = torch.where((t > 2 / 13) & (t <= 0.8), 5 / 6 * t + 1 / 3, f)
    f = torch.where((t > 0.8) & (t <= 1), torch.ones_like(t), f)
    return torch.where(den == 0, qc, qu + f * den)


def _limited(taps, adv):
    return torch.where(adv > 0, _cui(taps[0], taps[1], taps[2]), _cui(taps[3], taps[2], taps[1]))


def _taps(a, dim, n, count=4):
    return [a.narrow(dim, o, n) for o in range(count)]


def _flux_div(case, vel, rho, with_q):
    """Divergence of the limited density (times velocity) fluxes over the
    face-centred control volumes of each component (Sec. 4.2.2)."""
    h, n, bc = _spacing(case), (case["nx"], case["ny"], case["nz"]), _bc(case)
    res = []
    for c in range(3):
        dc = 2 - c
        inner = n[c] - 1
        total = None
        for a in range(3):
            da = 2 - a

            def extended(q, vel_ghost):
                k = q.shape[da]
                idx = [q.narrow(da, i, 1) for i in ((2, 1) if a == c else (1, 0))]
                end = [q.narrow(da, i, 1) for i in ((k - 2, k - 3) if a == c else (k - 1, k - 2))]
                s = (1.0, 1.0) if not vel_ghost else ((-1.0, -1.0) if a == c else (bc[2 * a], bc[2 * a + 1]))
                return torch.cat([s[0] * idx[0], s[0] * idx[1], q, s[1] * end[0], s[1] * end[1]], dim=da)

            r, q = extended(rho[c], False), extended(vel[c], True)
            if a == c:  # CV faces at the cell centres
                adv = _mean(vel[c], a)
                r, q = r.narrow(da, 1, r.shape[da] - 2), q.narrow(da, 1, q.shape[da] - 2)
                m = n[a]
            else:       # CV faces on the edges, interior C-faces only
                adv = _mean(vel[a], c)
                r, q = r.narrow(dc, 1, inner), q.narrow(dc, 1, inner)
                m = n[a] + 1
            f = adv * _limited(_taps(r, da, m), adv)
            if with_q:
                f = f * _limited(_taps(q, da, m), adv)
            div = f.diff(dim=da) / h[a]
            total = div if total is None else total + div
        z = torch.zeros_like(total.narrow(dc, 0, 1))
        res.append(torch.cat([z, total, z], dim=dc))
    return res


def _exact_transport(case, m, un, old):
    R = lambda u, r, w=False: _flux_div(case, _split(case, u), r, w)  # noqa: E731
    u1, u2, rn = 2 * un - old, 1.5 * un - 0.5 * old, m.rho
    r1 = [a - DT * b for a, b in zip(rn, R(un, rn))]
    r2 = [0.75 * a + 0.25 * b - 0.25 * DT * c for a, b, c in zip(rn, r1, R(u1, r1))]
    rho = [a / 3 + 2 / 3 * b - 2 / 3 * DT * c for a, b, c in zip(rn, r2, R(u2, r2))]
    return dict(rho=_pack(rho), C=_pack(R(u2, r2, True)))


def _minmod(*v):
    lo, hi = torch.stack(v).amin(0), torch.stack(v).amax(0)
    return torch.where(lo > 0, lo, torch.where(hi < 0, hi, torch.zeros_like(lo)))


def _xsppm7(m3, m2, m1, q0, p1, p2, p3):
    u7 = (-3 * m3 + 25 * m2 - 101 * m1 + 319 * q0 + 214 * p1 - 38 * p2 + 4 * p3) / 420
    ump = q0 + _minmod(p1 - q0, 4 * (q0 - m1))
    dm1, d0, dp1 = m2 - 2 * m1 + q0, m1 - 2 * q0 + p1, q0 - 2 * p1 + p2
    dp = _minmod(4 * d0 - dp1, 4 * dp1 - d0, d0, dp1)
    dm = _minmod(4 * dm1 - d0, 4 * d0 - dm1, dm1, d0)
    uul, umd = q0 + 4 * (q0 - m1), 0.5 * (q0 + p1) - 0.5 * dp
    ulc = q0 + 0.5 * (q0 - m1) + 4 / 3 * dm
    lo = lambda a, b, c: torch.minimum(torch.minimum(a, b), c)  # noqa: E731
    hi = lambda a, b, c: torch.maximum(torch.maximum(a, b), c)  # noqa: E731
    umin, umax = torch.maximum(lo(q0, p1, umd), lo(q0, uul, ulc)), torch.minimum(hi(q0, p1, umd), hi(q0, uul, ulc))
    return torch.where((u7 - q0) * (u7 - ump) <= 0, u7, u7 + _minmod(umin - u7, umax - u7))


def _mirrored(a, d, k):
    """a with k mirrored layers on either side along dimension d."""
    n = a.shape[d]
    i = torch.arange(-k, n + k)
    for _ in range(8):
        i = torch.where(i < 0, -i - 1, i)
        i = torch.where(i >= n, 2 * n - 1 - i, i)
    return a.index_select(d, i.clamp(0, n - 1).to(a.device))


def _exact_advect(case, vel, phi, half):
    h, wide = _spacing(case), case["limiter"] == "xsppm7"
    k = 4 if wide else 2
    s = _shape(case, 3)
    ph, total = half.reshape(s), 0.0
    for a, u in enumerate(_split(case, vel)):
        d = 2 - a
        t = _taps(_mirrored(ph, d, k), d, u.shape[d], 2 * k)
        if wide:
            f = torch.where(u > 0, _xsppm7(*t[:7]), _xsppm7(*t[:0:-1]))
        else:
            f = _limited(t, u)
        total = total + (u * f).diff(dim=d) / h[a]
    return (phi.reshape(s) - DT * total).reshape(-1)


def _exact_reinit(case, phi0, iters):
    h, n = _spacing(case), (case["nx"], case["ny"], case["nz"])
    q0 = phi0.reshape(_shape(case, 3))
    sg = torch.sign(q0)

    def mm(a, b):
        return torch.where(a * b > 0, torch.where(a.abs() < b.abs(), a, b), torch.zeros_like(a))

    def frac(a, b, c):  # zero of the quadratic through a, b with second difference c
        c2, c1, c0 = 0.5 * c, b - a, 0.5 * (a + b) - 0.125 * c
        root = (c1 * c1 - 4 * c2 * c0).clamp(min=0).sqrt()
        return 0.5 - 2 * c0 / (c1 + torch.copysign(root, c1))

    fixed = []
    for a in range(3):
        q = _taps(_mirrored(q0, 2 - a, 2), 2 - a, n[a], 5)
        dd = [q[i] - 2 * q[i + 1] + q[i + 2] for i in range(3)]
        hp = (h[a] * frac(q[2], q[3], mm(dd[1], dd[2]))).clamp(1e-10 * h[a], h[a])
        hm = (h[a] * frac(q[2], q[1], mm(dd[1], dd[0]))).clamp(1e-10 * h[a], h[a])
        fixed.append((q[2] * q[3] < 0, hp, q[2] * q[1] < 0, hm))

    def stage(p_):
        g2, dt = 0.0, None
        for a in range(3):
            if n[a] == 1:
                continue
            p = _taps(_mirrored(p_, 2 - a, 2), 2 - a, n[a], 5)
            dd = [p[i] - 2 * p[i + 1] + p[i + 2] for i in range(3)]
            mp, mn = mm(dd[1], dd[2]), mm(dd[1], dd[0])
            xp, hp, xm, hm = fixed[a]
            Dp = torch.where(xp, -p[2] / hp - 0.5 * hp * mp / h[a] ** 2, (p[3] - p[2] - 0.5 * mp) / h[a])
            Dm = torch.where(xm, p[2] / hm + 0.5 * hm * mn / h[a] ** 2, (p[2] - p[1] + 0.5 * mn) / h[a])
            g2 = g2 + torch.maximum(sg * Dm, -sg * Dp).clamp(min=0) ** 2
            near = torch.where(xp, hp, torch.full_like(hp, h[a]))
            near = torch.where(xm, torch.minimum(near, hm), near)
            dt = near if dt is None else torch.minimum(dt, near)
        return p_ - 0.3 * dt * sg * (g2.sqrt() - 1)

    p = q0
    for _ in range(iters):
        p = 0.5 * p + 0.5 * stage(stage(p))
    return p.reshape(-1)


def _phi4(r):
    r = r.abs()
    near = (3 - 2 * r + (1 + 4 * r - 4 * r * r).clamp(min=0).sqrt()) / 8
    far = (5 - 2 * r - (-7 + 12 * r - 4 * r * r).clamp(min=0).sqrt()) / 8
    return torch.where(r <= 1, near, torch.where(r <= 2, far, torch.zeros_like(r)))


def _marker_taps(case, X, c):
    """Per axis the four (indices, weights) of component c, taps beyond a wall
    folded back with the ghost's sign."""
    h, n, bc, out = _spacing(case), (case["nx"], case["ny"], case["nz"]), _bc(case), []
    for d in range(3):
        xs = X[:, d] / h[d] - (0.0 if d == c else 0.5)
        base = torch.floor(xs).long() - 1
        taps = []
        for q in range(4):
            i = base + q
            w = _phi4(i.double() - xs)
            for _ in range(3):
                if d == c:
                    lo, hi = i < 0, i > n[d]
                    w = torch.where(lo | hi, -w, w)
                    i = torch.where(lo, -i, torch.where(hi, 2 * n[d] - i, i))
                else:
                    lo, hi = i < 0, i >= n[d]
                    w = torch.where(lo, bc[2 * d] * w, torch.where(hi, bc[2 * d + 1] * w, w))
                    i = torch.where(lo, -1 - i, torch.where(hi, 2 * n[d] - 1 - i, i))
            if d == c:
                w = torch.where((i <= 0) | (i >= n[d]), torch.zeros_like(w), w)
            taps.append((i.clamp(0, n[d] - 1 + (d == c)), w))
        out.append(taps)
    return out


def _exact_rigid(case, vel, X, dV):
    """Locked body at rest: u - S(J u)."""
    h, parts, U = _spacing(case), [], None
    for c, q in enumerate(_split(case, vel)):
        t, flat = _marker_taps(case, X, c), q.reshape(-1).clone()
        sx, sy = q.shape[2], q.shape[1] * q.shape[2]
        every = [(a[0] + b[0] * sx + z[0] * sy, a[1] * b[1] * z[1]) for z in t[2] for b in t[1] for a in t[0]]
        U = sum(w * flat[i] for i, w in every)
        scale = dV / (h[0] * h[1] * h[2])
        for i, w in every:
            flat.index_add_(0, i, -U * w * scale)
        parts.append(flat)
    return dict(vel=torch.cat(parts), U=[0.0] * 3, W=[0.0] * 3)


def _exact_pressure(case, m, y):
    """Conjugate gradients with the diagonal as preconditioner, to 1e-13."""
    h, s = _spacing(case), _shape(case, 3)
    beta = []
    for c in range(3):
        b = 1 / m.rho[c] / h[c] ** 2
        b.narrow(2 - c, 0, 1).zero_()
        b.narrow(2 - c, b.shape[2 - c] - 1, 1).zero_()
        beta.append(b)
    diag = sum(b.narrow(2 - c, 0, s[2 - c]) + b.narrow(2 - c, 1, s[2 - c]) for c, b in enumerate(beta))

    def A(p):
        out = diag * p
        for c, b in enumerate(beta):
            d, k = 2 - c, s[2 - c] - 1
            mid = b.narrow(d, 1, k)
            out.narrow(d, 0, k).sub_(mid * p.narrow(d, 1, k))
            out.narrow(d, 1, k).sub_(mid * p.narrow(d, 0, k))
        return out

    r = -(y - y.mean()).reshape(s)
    x, z = torch.zeros_like(r), r / diag
    p, rz, stop = z.clone(), float((r * z).sum()), 1e-13 * float(r.norm())
    for it in range(12 * max(s)):
        q = A(p)
        al = rz / float((p * q).sum())
        x.add_(p, alpha=al)
        r.sub_(q, alpha=al)
        if it % 20 == 0 and float(r.norm()) < stop:
            break
        z = r / diag
        new = float((r * z).sum())
        p.mul_(new / rz).add_(z)
        rz = new
    else:
        return None
    return (x - x.mean()).reshape(-1)


def _exact_train(case, seed):
    """The network in float64 with bfloat16-rounded weights and inputs (its
    storage of activations in bfloat16 is not part of the exact result)."""
    x, t, p = _train_inputs(case, seed)
    dev = _dev()
    up = lambda a: torch.from_numpy(a).to(dev)  # noqa: E731
    w = up(p).bfloat16().double()
    f = torch.nn.functional
    params, off = [], 0
    for l, (co, ci) in enumerate(_train_sizes()):
        k = w[off:off + 27 * co * ci].reshape(3, 3, 3, co, ci).permute(3, 4, 0, 1, 2).contiguous().requires_grad_()
        off += 27 * co * ci
        b = up(p)[off:off + co].double().requires_grad_()
        off += co
        params.append((k, b))
    hw, hb = up(p)[off:off + 16].double().requires_grad_(), up(p)[off + 16:].double().requires_grad_()

    def cv(l, a):
        # one shifted product per tap
        k, b = params[l]
        ap, s = f.pad(a, (1,) * 6), a.shape[1:]
        o = b.view(-1, 1, 1, 1)
        for q in range(27):
            z, yy, xx = q // 9, q // 3 % 3, q % 3
            o = o + torch.einsum("oc,czyx->ozyx", k[:, :, z, yy, xx], ap[:, z:z + s[0], yy:yy + s[1], xx:xx + s[2]])
        return torch.relu(o)

    grow = lambda a: a.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)  # noqa: E731
    a0 = f.pad(up(x).bfloat16().double().permute(3, 0, 1, 2), (0,) * 6 + (0, 13))
    a2 = cv(1, cv(0, a0))
    b2 = cv(3, cv(2, f.avg_pool3d(a2, 2)))
    c2 = cv(5, cv(4, f.avg_pool3d(b2, 2)))
    u2 = cv(7, cv(6, torch.cat([grow(c2), b2])))
    v2 = cv(9, cv(8, torch.cat([grow(u2), a2])))
    out = (hw.view(-1, 1, 1, 1) * v2).sum(0) + hb
    loss = 0.5 * (out - up(t).double()).square().mean()
    loss.backward()
    g = []
    for l, (k, b) in enumerate(params):
        g += [k.grad.permute(2, 3, 4, 0, 1).reshape(-1), b.grad]
    return dict(out=out.detach(), loss=float(loss.detach()), grads=torch.cat(g + [hw.grad, hb.grad]))


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        return None  # a converged iteration inside a nonlinear step
    if kind == "train":
        return _exact_train(case, seed)
    phi, psi, b = _tank(case, seed)
    # the same inputs as prepare() makes, without a context
    g, m = _gen(seed), _Materials(case, phi, psi) if kind != "reinit" else None
    nvel = sum(math.prod(_shape(case, c)) for c in range(3))
    ncell = math.prod(_shape(case, 3))
    if kind == "solve":
        if nvel + ncell > 60000:
            return None
        u = (torch.rand(nvel, dtype=F64, device=_dev(), generator=g) * 2 - 1) * 1e-2
        return _exact_solve(case, m, torch.cat([u, torch.zeros(ncell, dtype=F64, device=_dev())]))
    if kind == "apply":
        x = torch.randn(nvel + ncell, dtype=F64, device=_dev(), generator=g)
        _zero_walls(case, x)
        return _matvec(case, m, x, DT)
    if kind == "transport":
        un = _velocity(case, seed)
        return _exact_transport(case, m, un, 0.95 * un + 0.05 * _velocity(case, seed + 1000003))
    if kind == "advect":
        phi = phi.reshape(-1)
        return _exact_advect(case, _velocity(case, seed), phi, phi + 1e-3 * torch.sin(5.0 * phi))
    if kind == "reinit":
        return _exact_reinit(case, (phi * (1.0 + 0.3 * torch.sin(7.0 * phi))).reshape(-1), case["iters"])
    if kind == "rigid":
        return _exact_rigid(case, _velocity(case, seed), b["markers"], b["dV"])
    y = torch.rand(ncell, dtype=F64, device=_dev(), generator=g) * 2 - 1
    return _exact_pressure(case, m, y - y.mean())
