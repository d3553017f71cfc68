"""The work whose speed counts: what a user of this library has it do, over the range of sizes,
precisions, preconditioners and box conditions it is used at, through the public Python binding
of the C ABI (paper_2211_10698_gb300.ccm).

  step    projection steps of one resident case (ccm_step), fields left on the device
  batch   one step of many uneven cases advanced together (ccm_batch_step)
  solve   one pressure solve from host arrays (ccm_solve_pressure)
  noalloc one pressure solve on the caller's device buffers (ccm_solve_pressure_noalloc)
  serve   a burst of requests through the request loop, from submission to the fields on the host

Sizes, boxes, bodies and solver settings are those of inputs.py, bench.py and the tests; a seed
sets the velocity perturbation, the right-hand sides, or the bodies and Reynolds numbers of a mix.
Poisson tolerances are the 1e-10 of inputs.py for a solve and 1e-11 for steps, where the pressure
itself, not only its residual, is settled to a few 1e-10 whatever correct solver found it.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2211_10698_gb300 import ccm, inputs as I

FIELDS = (("u", ccm.CCM_F_U), ("v", ccm.CCM_F_V), ("p", ccm.CCM_F_P))


def listed():
    return [
        # The smallest use: the 128x64 cylinder at Re 40 stepped for its wake (FP64, latency-bound).
        dict(name="cylinder_128x64_fp64", kind="step", flow="cylinder", nx=128, ny=64, re=40.0, steps=5,
             precision="fp64", precond="jacobi", degree=1, guess=0, cfl=0.5, tol=1e-11),
        # Vortex shedding in full FP64 on the grid it is resolved on (the headline workload).
        dict(name="cylinder_1024x512_fp64", kind="step", flow="cylinder", nx=1024, ny=512, re=100.0, steps=1,
             precision="fp64", precond="jacobi", degree=1, guess=0, cfl=0.5, tol=1e-11),
        # A long FP64 run with the projected initial guess, half the resolution.
        dict(name="cylinder_512x256_guess", kind="step", flow="cylinder", nx=512, ny=256, re=100.0, steps=2,
             precision="fp64", precond="jacobi", degree=1, guess=32, cfl=0.5, tol=1e-11),
        # The same shedding flow in mixed precision with the Chebyshev preconditioner.
        dict(name="cylinder_1024x512_mixed", kind="step", flow="cylinder", nx=1024, ny=512, re=100.0, steps=1,
             precision="mixed", precond="chebyshev", degree=3, guess=0, cfl=0.5, tol=1e-11),
        # The airfoil in mixed precision: the largest single case.
        dict(name="naca_2048x1024_mixed", kind="step", flow="naca", nx=2048, ny=1024, re=1000.0, steps=1,
             precision="mixed", precond="chebyshev", degree=3, guess=0, cfl=0.5, tol=1e-11),
        # A stretched mesh (every row has its own coefficients), FP64.
        dict(name="stretched_320x200_fp64", kind="step", flow="stretched", nx=320, ny=200, re=100.0, steps=1,
             precision="fp64", precond="jacobi", degree=1, guess=0, cfl=0.5, tol=1e-11),
        # The lid-driven cavity: a closed box, whose Poisson system is singular.
        dict(name="cavity_192x192_fp64", kind="step", flow="cavity", nx=192, ny=192, re=400.0, steps=1,
             precision="fp64", precond="jacobi", degree=1, guess=0, cfl=0.5, tol=1e-11),
        # A parameter study: 64 cylinders and airfoils of uneven size in one batch, mixed precision.
        dict(name="batch_64_mixed", kind="batch", n=64, nx_lo=256, nx_hi=1024, precision="mixed",
             precond="chebyshev", degree=4, cfl=0.2, tol=1e-11),
        # A small FP64 batch.
        dict(name="batch_8_fp64", kind="batch", n=8, nx_lo=128, nx_hi=512, precision="fp64", precond="jacobi",
             degree=1, cfl=0.2, tol=1e-11),
        # The pressure solve alone, from a host code's arrays: an odd grid, cells that are not square.
        dict(name="solve_701x333_mixed", kind="solve", nx=701, ny=333, precision="mixed", precond="jacobi", degree=1,
             tol=1e-10),
        # The pressure solve of a host code that owns all device memory.
        dict(name="noalloc_250x121_fp64", kind="noalloc", nx=250, ny=121, precision="fp64", precond="jacobi", degree=1,
             tol=1e-10),
        # A burst of requests: queueing, set-up, stepping in the batch, results to the host.
        dict(name="serve_12_mixed", kind="serve", n=12, nx_lo=128, nx_hi=512, steps=6, precision="mixed",
             precond="chebyshev", degree=4, cfl=0.2, tol=1e-11),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "batch", "solve", "noalloc", "serve"])
    precision = rng.choice(["fp64", "mixed"])
    # Chebyshev with mixed precision (as every mixed workload is configured), Jacobi with both
    precond = rng.choice(["chebyshev", "chebyshev", "jacobi"]) if precision == "mixed" else "jacobi"
    degree = rng.choice([2, 3, 4]) if precond == "chebyshev" else 1
    solver = dict(precision=precision, precond=precond, degree=degree)
    # the explicit convection of small cut cells is stable at any size and Reynolds number of the
    # range at CFL 0.2 (at 0.5 some of them grow; the listed grids do not)
    cfl = 0.2
    if kind == "step":
        flow = rng.choice(["cylinder", "cylinder", "naca", "stretched", "cavity"])
        if flow == "cavity":
            nx = _log(rng, 48, 256)
            return dict(kind=kind, flow=flow, nx=nx, ny=nx, re=100.0 * rng.randint(1, 10), steps=rng.randint(1, 3), guess=0,
                        cfl=cfl, tol=1e-11, precision="fp64", precond="jacobi", degree=1)
        if flow == "stretched":
            nx = _log(rng, 64, 512)
            ny = int(nx * rng.uniform(0.55, 0.75))
        else:
            nx = _log(rng, 96, 2048 if precond == "chebyshev" else 1024)
            ny = nx // 2 + rng.choice([0, 0, 1, -3])
        return dict(kind=kind, flow=flow, nx=nx, ny=ny, re=float(rng.randint(40, 1000)), steps=rng.randint(1, 3) if nx < 512 else 1,
                    guess=rng.choice([0, 0, 32]), cfl=cfl, tol=1e-11, **solver)
    if kind == "batch":
        lo = _log(rng, 96, 320)
        return dict(kind=kind, n=rng.randint(2, 24), nx_lo=lo, nx_hi=_log(rng, lo, 704), cfl=cfl, tol=1e-11, **solver)
    if kind == "serve":
        return dict(kind=kind, n=rng.randint(2, 12), nx_lo=128, nx_hi=_log(rng, 160, 512), steps=rng.randint(4, 8), cfl=cfl, tol=1e-11,
                    **solver)
    nx = _log(rng, 64, 320 if kind == "noalloc" else 720)
    ny = int(nx * rng.uniform(0.4, 0.6))
    return dict(kind=kind, nx=nx, ny=ny, tol=1e-10, **solver)


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
def _solver(spec, case):
    spec.dt *= case.get("cfl", 0.5) / 0.5
    spec.precision, spec.precond, spec.cheb_degree = case["precision"], case["precond"], case["degree"]
    spec.tol_p = case["tol"]
    spec.guess_history = case.get("guess", 0)
    return spec


CIRCLE = dict(cx=0.0, cy=0.0, r=0.5)


def _step_spec(case):
    nx, ny = case["nx"], case["ny"]
    if case["flow"] == "cavity":
        spec = I.make_case("cavity", nx, ny, (0.0, 1.0, 0.0, 1.0), I.Geometry(), re=case["re"], cfl=0.5, lref=1.0,
                           bc=I.closed_box_bc(lid=1.0))
    elif case["flow"] == "stretched":
        h = 0.5 / (nx / 10.0)  # a fine patch of nx/4 cells over the body, growing outwards
        spec = I.stretched_cylinder(nx=nx, ny=ny, box=(-5.0, 15.0, -5.0, 5.0), fine=(nx // 4, nx // 4), h_fine=h,
                                    ratio=1.0 + 2.0 / nx, re=case["re"])
    elif case["flow"] == "naca":
        spec = I.make_case("naca", nx, ny, (-2.0, 6.0, -2.0, 2.0), I.Geometry(kind=I.GEOM_NACA, naca_tt=12, aoa_deg=4.0),
                           re=case["re"], cfl=0.5, lref=1.0)
    else:
        box = (-4.0, 12.0, -4.0, 4.0) if nx > 256 else (-2.0, 6.0, -2.0, 2.0)
        spec = I.make_case("cylinder", nx, ny, box, I.Geometry(kind=I.GEOM_CIRCLE, **CIRCLE), re=case["re"], cfl=0.5, lref=1.0)
    return _solver(spec, case)


def _solve_spec(case):
    box = (-2.0, 6.0, -2.0, 2.0)
    return _solver(I.make_case("solve", case["nx"], case["ny"], box, I.Geometry(kind=I.GEOM_CIRCLE, **CIRCLE), re=100.0, cfl=0.5,
                               lref=1.0), case)


def _mix(case, seed):
    """n cases of sizes spread over [nx_lo, nx_hi]; bodies, angles and Reynolds numbers from the seed."""
    out = []
    for k in range(case["n"]):
        f = k / max(case["n"] - 1, 1)
        nx = int(round(case["nx_lo"] * (case["nx_hi"] / case["nx_lo"]) ** f))
        # batch_cases alternates cylinders and airfoils by position
        spec = I.batch_cases(k % 2 + 1, seed=7919 * (seed % 100003) + 31 * k, nx_range=(nx, nx))[-1]
        out.append(_solver(spec, case))
    return out


def _noise(shape, seed, sigma=1e-3):
    return np.random.default_rng(seed).standard_normal(shape) * sigma


def _perturb(c, seed):
    """The seeded N(0, 1e-3) velocity perturbation on top of the start."""
    for k, (_, f) in enumerate(FIELDS[:2]):
        c.set_field(f, c.get_field(f) + _noise(c.shape, 2 * seed + k))


def _restart(cases, step):
    """Past the start-up of flows about bodies.  One step makes the perturbed uniform stream
    divergence-free; its pressure is that of the impulsive start, 1 / dt times the flow's, and is
    dropped as by a program that restarts from a velocity field; in the steps that follow the
    pressure builds up, and from then on a step solves for its change."""
    step(1)
    for c in cases:
        for f in (ccm.CCM_F_P, ccm.CCM_F_PHI):
            c.set_field(f, np.zeros(c.shape))
        ccm.lib().ccm_set_field(c.h, ccm.CCM_F_STEP, (ctypes.c_double * 1)(0.0), 1)
    step(3)


def _rhs(case, seed):
    """A divergence field as a solver meets it: smooth structures of several scales and grid noise."""
    rng = np.random.default_rng(seed)
    ny, nx = case["ny"] + 3, case["nx"] + 3
    x, y = np.linspace(0.0, 1.0, nx), np.linspace(0.0, 0.5, ny)
    out = 0.1 * rng.standard_normal((ny, nx))
    for _ in range(12):
        s, a = 0.01 + 0.1 * rng.random(), rng.standard_normal()
        out += a * np.outer(np.exp(-((y - 0.5 * rng.random()) / s) ** 2), np.exp(-((x - rng.random()) / s) ** 2))
    return out


class _Device:
    """A field of a case as a torch tensor on the case's own memory (ccm_field_device_ptr)."""

    def __init__(self, c, field):
        self.case = c  # the tensor keeps the memory's owner
        p, pitch = c.device_ptr(field)
        self.__cuda_array_interface__ = dict(shape=c.shape, strides=(8 * pitch, 8), typestr="<f8", data=(p, False), version=2)


def _views(c):
    """U, V, P at the faces and cells of the box."""
    ny, nx = c.spec.ny, c.spec.nx
    u, v, p = (torch.as_tensor(_Device(c, f), device="cuda") for _, f in FIELDS)
    return dict(u=u[1:ny + 1, 1:nx + 2], v=v[1:ny + 2, 1:nx + 1], p=p[1:ny + 1, 1:nx + 1])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":
        c = ccm.Case(_step_spec(case))
        _perturb(c, seed)
        if case["flow"] != "cavity":
            _restart([c], c.step)
        return dict(kind=kind, case=c, views=_views(c), steps=case["steps"])
    if kind == "batch":
        b = ccm.Batch(case["n"])
        cases = []
        for k, spec in enumerate(_mix(case, seed)):
            c = ccm.Case(spec)
            _perturb(c, 1000 * seed + k)
            b.add(c)
            cases.append(c)
        _restart(cases, b.step)
        return dict(kind=kind, batch=b, cases=cases, views=[_views(c) for c in cases])
    if kind == "solve":
        c = ccm.Case(_solve_spec(case))
        return dict(kind=kind, case=c, rhs=_rhs(case, seed), guess=np.zeros(c.shape), out=np.empty(c.shape))
    if kind == "noalloc":
        c = ccm.Case(_solve_spec(case))
        rows, cols = c.shape
        _, pitch = c.device_ptr(ccm.CCM_F_PHI)
        rhs = torch.zeros((rows, pitch), dtype=torch.float64, device="cuda")
        rhs[:, :cols] = torch.from_numpy(_rhs(case, seed)).cuda()
        return dict(kind=kind, case=c, rhs=rhs, phi=torch.zeros_like(rhs), stats=ccm.ccm_solve_stats())
    server = ccm.Server(150 << 30, max_batch=64, chunk_steps=4)
    return dict(kind=kind, server=server, specs=_mix(case, seed), steps=case["steps"])


# ---------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------
def run(state):
    kind = state["kind"]
    if kind == "step":
        state["case"].step(state["steps"])
        return state["views"]
    if kind == "batch":
        state["batch"].step(1)
        return {f: torch.cat([v[f].reshape(-1) for v in state["views"]]) for f, _ in FIELDS}
    if kind == "solve":
        c = state["case"]
        c.set_field(ccm.CCM_F_PHI, state["guess"])
        c.solve_pressure(state["rhs"])
        c.get_field(ccm.CCM_F_PHI, out=state["out"])
        return dict(phi=state["out"][1:-2, 1:-2])
    if kind == "noalloc":
        c = state["case"]
        state["phi"].zero_()
        status = ccm.lib().ccm_solve_pressure_noalloc(c.h, ctypes.c_void_p(state["rhs"].data_ptr()),
                                                      ctypes.c_void_p(state["phi"].data_ptr()), ctypes.byref(state["stats"]))
        if status != ccm.CCM_OK:
            raise ccm.CcmError(status, ccm.lib().ccm_last_error().decode())
        rows, cols = c.shape
        return dict(phi=state["phi"][1:rows - 2, 1:cols - 2])
    s = state["server"]
    ids = [s.submit(spec, nsteps=state["steps"]) for spec in state["specs"]]
    while s.run(1):
        pass
    out = []
    for rid, spec in zip(ids, state["specs"]):
        out.append({n: s.get_field(rid, f, spec.shape)[1:-2, 1:-2] for n, f in FIELDS})
        s.release(rid)
    return out


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------
def work(case):
    """Each input read once, each output written once, each operator applied once: how often an
    iteration has to pass over the grid is the solver's affair and not counted."""
    if case["kind"] in ("solve", "noalloc"):
        n = case["nx"] * case["ny"]
        # right-hand side, warm start, solution, and the row: diagonal and two face coefficients
        return dict(bytes=8.0 * 6 * n, flops=10.0 * n)
    if case["kind"] == "step":
        cells = case["nx"] * case["ny"]
    else:
        cells = sum(s.nx * s.ny for s in _mix(case, 0))
    steps = case.get("steps", 1)
    # state in and out: u, v, P, Phi, two levels of conv of two components; the operators'
    # apertures and weights (about 16 arrays); about 250 operations of the explicit stages
    return dict(bytes=8.0 * (8 + 6 + 16) * cells * steps, flops=250.0 * cells * steps)


# ---------------------------------------------------------------------------------------------
# the same results in 64 bits from plain array arithmetic
# ---------------------------------------------------------------------------------------------
def _cg(apply, b, diag, tol=1e-14, most=20000, zero_mean=None):
    """Jacobi-preconditioned CG on tensors (a list of them is one vector)."""
    dot = lambda p, q: sum((x * y).sum() for x, y in zip(p, q))  # noqa: E731
    fix = zero_mean or (lambda z: z)
    x = [torch.zeros_like(t) for t in b]
    r = [t.clone() for t in b]
    z = fix([t / d for t, d in zip(r, diag)])
    p, rz, bb = z, dot(r, z), float(dot(b, b))
    for it in range(most):
        q = apply(p)
        a = rz / dot(p, q)
        x = [s + a * t for s, t in zip(x, p)]
        r = [s - a * t for s, t in zip(r, q)]
        if it % 20 == 0 and float(dot(r, r)) <= tol * tol * bb:
            break
        z = fix([t / d for t, d in zip(r, diag)])
        new = dot(r, z)
        p = [s + (new / rz) * t for s, t in zip(z, p)]
        rz = new
    return x


def _wet_area(X0, X1, Y0, Y1, cx, cy, r):
    """Fluid area of boxes outside a circle, the boundary inside a box replaced by the chord
    between its crossings with the edges: the polygon of fluid corners and crossings."""
    cor = [(X0, Y0), (X1, Y0), (X1, Y1), (X0, Y1)]
    fl = [np.hypot(x - cx, y - cy) > r for x, y in cor]
    area = np.zeros(np.broadcast_shapes(X0.shape, Y0.shape))
    fx = fy = px = py = None  # the first and the last point of the polygon so far (nan: none)
    for k in range(4):
        (xa, ya), (xb, yb) = cor[k], cor[(k + 1) % 4]
        cross = fl[k] != fl[(k + 1) % 4]
        if k % 2 == 0:
            s = np.sqrt(np.maximum(r * r - (ya - cy) ** 2, 0.0))
            lo, hi = np.minimum(xa, xb), np.maximum(xa, xb)
            qx = np.where((cx - s >= lo) & (cx - s <= hi), cx - s, cx + s)
            qy = ya + 0.0 * qx
        else:
            s = np.sqrt(np.maximum(r * r - (xa - cx) ** 2, 0.0))
            lo, hi = np.minimum(ya, yb), np.maximum(ya, yb)
            qy = np.where((cy - s >= lo) & (cy - s <= hi), cy - s, cy + s)
            qx = xa + 0.0 * qy
        for on, x, y in ((fl[k], xa + 0.0 * area, ya + 0.0 * area), (cross, qx + 0.0 * area, qy + 0.0 * area)):
            if px is None:
                px, py = np.where(on, x, np.nan), np.where(on, y, np.nan)
                fx, fy = px.copy(), py.copy()
                continue
            area += np.where(on & ~np.isnan(px), px * y - py * x, 0.0)
            fx, fy = np.where(on & np.isnan(fx), x, fx), np.where(on & np.isnan(fy), y, fy)
            px, py = np.where(on, x, px), np.where(on, y, py)
    area += np.where(np.isnan(px), 0.0, px * fy - py * fx)
    return 0.5 * area


def _wet_length(a0, a1, off, r):
    """Fluid length of the segment [a0, a1] on the line at distance off from the circle's centre
    (a relative to the centre)."""
    s = np.sqrt(np.maximum(r * r - off ** 2, 0.0))
    f0, f1 = np.hypot(a0, off) > r, np.hypot(a1, off) > r
    c = np.where((-s >= a0) & (-s <= a1), -s, s)
    return np.where(f0 & f1, a1 - a0, np.where(f0, c - a0, np.where(f1, a1 - c, 0.0)))


def _solve_exact(case, seed):
    """K phi = rhs with the cut-cell coefficients A^2 / V about a circle; inflow west (no flux),
    phi = 0 beyond the other sides."""
    spec = _solve_spec(case)
    nx, ny, hx, hy, cx, cy, r = spec.nx, spec.ny, spec.hx, spec.hy, CIRCLE["cx"], CIRCLE["cy"], CIRCLE["r"]
    xf, yf = spec.x0 + np.arange(nx + 1) * hx, spec.y0 + np.arange(ny + 1) * hy
    xc, yc = xf[:-1] + 0.5 * hx, yf[:-1] + 0.5 * hy

    def face(A, V):
        return np.where(V > 1e-12 * hx * hy, A * A / np.where(V > 0, V, 1.0), 0.0)

    X, Y = xf[None, :], yf[:, None]
    cu = face(_wet_length(Y[:-1] - cy, Y[1:] - cy, X - cx, r), _wet_area(X - 0.5 * hx, X + 0.5 * hx, Y[:-1], Y[1:], cx, cy, r))
    cv = face(_wet_length(X[:, :-1] - cx, X[:, 1:] - cx, Y - cy, r),
              _wet_area(X[:, :-1], X[:, 1:], Y - 0.5 * hy, Y + 0.5 * hy, cx, cy, r))
    cu[:, 0] = 0.0
    assert xc.size == nx and yc.size == ny
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    cu, cv = torch.from_numpy(cu).to(dev), torch.from_numpy(cv).to(dev)
    diag = cu[:, :-1] + cu[:, 1:] + cv[:-1] + cv[1:]
    wet = diag > 0
    diag = torch.where(wet, diag, torch.ones_like(diag))
    b = torch.from_numpy(_rhs(case, seed)[1:-2, 1:-2].copy()).to(dev) * wet

    def apply(v):
        f = torch.nn.functional.pad(v[0], (1, 1, 1, 1))
        c = f[1:-1, 1:-1]
        return [torch.where(wet, diag * c - cu[:, :-1] * f[1:-1, :-2] - cu[:, 1:] * f[1:-1, 2:] - cv[:-1] * f[:-2, 1:-1]
                            - cv[1:] * f[2:, 1:-1], c)]

    x, = _cg(apply, [b], [diag])
    d, = _cg(apply, [b - apply([x])[0]], [diag], tol=1e-6)  # the correction of the true residual
    return dict(phi=(x + d).cpu().numpy())


def _cavity_exact(case, seed):
    """The projection steps of the lid-driven cavity on a uniform mesh: Adams-Bashforth
    convection in flux form, Crank-Nicolson viscosity visc(S) with S the symmetric strain, the
    pressure increment of mean zero, and the update P += Phi - (dt mu / 2 rho) lap Phi."""
    spec = _step_spec(case)
    n, m, hx, hy, mu, dt, rho = spec.nx, spec.ny, spec.hx, spec.hy, spec.mu, spec.dt, spec.rho
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    lid = spec.bc_ut[I.SIDE_N]
    nu_, nv_ = (_noise(spec.shape, 2 * seed + k) for k in range(2))
    u = torch.zeros((m, n + 1), dtype=torch.float64, device=dev)
    v = torch.zeros((m + 1, n), dtype=torch.float64, device=dev)
    u[:, 1:-1] = torch.from_numpy(nu_[1:m + 1, 2:n + 1].copy()).to(dev)
    v[1:-1] = torch.from_numpy(nv_[2:m + 1, 1:n + 1].copy()).to(dev)

    def ghosts(u, v, lid):
        """u with a row below and above, v with a column left and right (tangential reflection)."""
        return (torch.cat([-u[:1], u, 2.0 * lid - u[-1:]]), torch.cat([-v[:, :1], v, -v[:, -1:]], 1))

    def conv(u, v):
        U, V = ghosts(u, v, lid)
        un = 0.5 * (u[:, 1:] + u[:, :-1])             # at cells
        vn = 0.5 * (v[1:] + v[:-1])
        uy, vx = 0.5 * (U[1:] + U[:-1]), 0.5 * (V[:, 1:] + V[:, :-1])  # at nodes
        fu, fv, fn = hy * un * un, hx * vn * vn, uy * vx
        cu, cv = torch.zeros_like(u), torch.zeros_like(v)
        cu[:, 1:-1] = fu[:, 1:] - fu[:, :-1] + hx * (fn[1:, 1:-1] - fn[:-1, 1:-1])
        cv[1:-1] = fv[1:] - fv[:-1] + hy * (fn[1:-1, 1:] - fn[1:-1, :-1])
        return cu, cv

    def visc(u, v, lid):
        U, V = ghosts(u, v, lid)
        sxx, syy = (u[:, 1:] - u[:, :-1]) / hx, (v[1:] - v[:-1]) / hy
        sxy = 0.5 * ((U[1:] - U[:-1]) / hy + (V[:, 1:] - V[:, :-1]) / hx)
        wu, wv = torch.zeros_like(u), torch.zeros_like(v)
        wu[:, 1:-1] = hy * (sxx[:, 1:] - sxx[:, :-1]) + hx * (sxy[1:, 1:-1] - sxy[:-1, 1:-1])
        wv[1:-1] = hx * (syy[1:] - syy[:-1]) + hy * (sxy[1:-1, 1:] - sxy[1:-1, :-1])
        return wu, wv

    def grad(p):
        gu, gv = torch.zeros_like(u), torch.zeros_like(v)
        gu[:, 1:-1] = hy * (p[:, 1:] - p[:, :-1])
        gv[1:-1] = hx * (p[1:] - p[:-1])
        return gu, gv

    def div(u, v):
        return hy * (u[:, 1:] - u[:, :-1]) + hx * (v[1:] - v[:-1])

    vol, mass = hx * hy, rho / dt * hx * hy

    def helm(z):
        wu, wv = visc(z[0], z[1], 0.0)
        return [mass * z[0] - mu * wu, mass * z[1] - mu * wv]

    def poisson(z):
        gu, gv = grad(z[0])
        return [-div(gu, gv) / vol]

    p = torch.zeros((m, n), dtype=torch.float64, device=dev)
    one_u, one_v = torch.full_like(u, mass), torch.full_like(v, mass)
    diag = poisson([p])[0] + 2.0 * (hy / hx + hx / hy)
    mean0 = lambda z: [t - t.mean() for t in z]  # noqa: E731
    old = None
    for _ in range(case["steps"]):
        cu, cv = conv(u, v)
        ou, ov = old or (cu, cv)
        gu, gv = grad(p)
        wu, wv = visc(u, v, lid)
        lu, lv = visc(torch.zeros_like(u), torch.zeros_like(v), lid)
        ru = mass * u - rho * (1.5 * cu - 0.5 * ou) - gu + mu * (wu + lu)
        rv = mass * v - rho * (1.5 * cv - 0.5 * ov) - gv + mu * (wv + lv)
        old = (cu, cv)
        us, vs = _cg(helm, [ru, rv], [one_u, one_v])
        phi, = _cg(poisson, mean0([-(rho / dt) * div(us, vs)]), [diag], zero_mean=mean0)
        gu, gv = grad(phi)
        u, v = us - dt / rho * gu / vol, vs - dt / rho * gv / vol
        p = p + phi + 0.5 * dt * mu / rho * poisson([phi])[0] / vol
    return dict(u=u.cpu().numpy(), v=v.cpu().numpy(), p=p.cpu().numpy())


def exact(case, seed):
    if case["kind"] in ("solve", "noalloc"):
        return _solve_exact(case, seed)
    if case["kind"] == "step" and case["flow"] == "cavity":
        return _cavity_exact(case, seed)
    return None  # a step about a body takes the whole cut-cell discretisation
