"""Performance cases of the LW-ACM library.

Each case is what a program does with the public binding
(paper_1111_2142_gb300/lwacm.py): it holds the initial fields on the GPU and a
context with its workspace, then one pass hands the fields to the context
(set_fields), advances a number of time steps and reads the result (zero-copy
views of the state, gradients, or the series of global quantities that was
monitored on the way). Every pass starts from the same fields, so it can be
repeated. Sizes, viscosities and options are those of the benchmark, the tests and
the paper's runs, and generic ragged ones.

exact() restates the method in plain torch in FP64 (link by link, with rolled
arrays and autograd for gradients) and shares no code with the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1111_2142_gb300 import lwacm as lw

BCS = {"periodic": lw.PERIODIC, "cavity": lw.CAVITY, "channel": lw.CHANNEL}
STORAGES = {"f32": lw.F32, "bf16": lw.BF16, "f16": lw.F16}
L2_BYTES = 64 << 20  # a state below this stays on the chip between steps


# ---- cases -------------------------------------------------------------------------


def _steps_case(dims, steps, **kw):
    """A single domain advanced `steps` steps; defaults: plain scheme, periodic, FP32."""
    case = dict(kind="steps", nx=dims[0], ny=dims[1], nz=dims[2] if len(dims) > 2 else 1, steps=steps,
                lattice=19 if len(dims) > 2 else 9, bc="periodic", storage="f32", nu=0.01, u0=0.02,
                nu_p=0.0, gamma=0.0, alpha=0.0, semi=False, force=0.0, stochastic=False, monitor=0)
    case.update(kw)
    return case


def listed():
    return [
        # the paper's 2D Taylor-Green run at its small size: a step is one short launch
        dict(name="tgv2d_64", **_steps_case((64, 64), 256, u0=0.01)),
        # the 128^2 double shear layer with both improvements of the scheme (omega_p and
        # the bulk viscosity): thousands of short steps in a run, a tenth of them here
        dict(name="shear2d_128", **_steps_case((128, 128), 320, nu=5.12e-4, u0=0.04, nu_p=170 * 5.12e-4, gamma=0.4)),
        # a force that changes every step (the forced Taylor-Green vortex): the program sets
        # the field and takes one step, so nothing is replayed from a graph
        dict(name="driven2d_96", kind="driven", lattice=9, nx=96, ny=96, nz=1, steps=16, nu=0.1, u0=0.04),
        # the 2D lid-driven cavity at Re 1000: walls, a state that stays in L2
        dict(name="cavity2d_1024", **_steps_case((1024, 1024), 128, bc="cavity", nu=0.1024, u0=0.1)),
        # a large 2D domain: bound by memory traffic or by instructions, not by launches
        dict(name="periodic2d_4096", **_steps_case((4096, 4096), 16)),
        # an ensemble of 256 2D domains of 32 to 512 nodes a side, each with its viscosity
        dict(name="ensemble2d_256", kind="ensemble", lattice=9, domains=256, smin=32, smax=512, dims_seed=1, steps=32,
             tile=0, mode=0, u0=0.02),
        # the headline workload with its kinetic-energy curve every 10 steps
        dict(name="tgv3d_256", **_steps_case((256, 256, 256), 20, nu=0.005, monitor=10)),
        # 3D rows longer than 256 nodes with BF16 storage
        dict(name="bf16_3d_384", **_steps_case((384, 256, 256), 16, nu=0.005, u0=0.05, storage="bf16")),
        # the paper's 60^3 diagonally driven cavity, its global quantities read now and then
        dict(name="cavity3d_60", **_steps_case((60, 60, 60), 128, bc="cavity", nu=60 * 0.1 / 700, u0=0.1, monitor=64)),
        # a 3D box of sides as a user's geometry gives them: no multiple of anything
        dict(name="ragged3d_201", **_steps_case((201, 131, 150), 24)),
        # a temperature carried along by a 3D flow
        dict(name="scalar3d_256", **_steps_case((256, 256, 128), 16, nu=0.02, alpha=0.03)),
        # gradients of a 3D run with respect to its start and the viscosity
        dict(name="adjoint3d_128", kind="adjoint", lattice=19, nx=128, ny=128, nz=128, steps=24, bc="periodic", nu=0.01,
             u0=0.02),
    ]


def draw(rng):
    """One more case of the listed ones' kinds, its sizes over their whole range."""
    logu = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))  # noqa: E731
    nu = round(math.exp(rng.uniform(math.log(0.003), math.log(0.1))), 5)
    kind = rng.choice(["small2d", "variant2d", "driven", "walls2d", "large2d", "ensemble", "rows3d", "storage3d", "walls3d",
                       "ragged3d", "variant3d", "adjoint"])
    if kind == "small2d":
        return _steps_case((logu(20, 260), logu(20, 260)), rng.choice([64, 128, 200, 256]), nu=nu)
    if kind == "variant2d":
        opt = rng.choice([dict(nu_p=0.1), dict(gamma=0.4), dict(nu_p=0.08, gamma=0.3), dict(force=1e-6), dict(semi=True)])
        return _steps_case((logu(48, 2100), logu(48, 2100)), rng.choice([24, 48, 96]), nu=nu, **opt)
    if kind == "driven":
        return dict(kind="driven", lattice=9, nx=logu(32, 800), ny=logu(32, 800), nz=1, steps=rng.choice([8, 16, 24]),
                    nu=nu, u0=0.04)
    if kind == "walls2d":
        return _steps_case((logu(64, 2000), logu(64, 2000)), rng.choice([32, 64, 96]), nu=nu, u0=0.08,
                           bc=rng.choice(["cavity", "channel"]), storage=rng.choice(["f32", "f32", "bf16"]))
    if kind == "large2d":
        return _steps_case((logu(1000, 4200), logu(1000, 4200)), rng.choice([8, 12, 16]), nu=nu,
                           storage=rng.choice(["f32", "f32", "f16"]))
    if kind == "ensemble":
        return dict(kind="ensemble", lattice=9, domains=logu(8, 256), smin=rng.choice([24, 32, 48]),
                    smax=rng.choice([128, 256, 480]), dims_seed=rng.randrange(1000), steps=rng.choice([8, 16, 32]),
                    tile=rng.choice([0, 0, 2]), mode=rng.choice([0, 0, 1]), u0=0.02)
    if kind == "rows3d":
        nx = rng.choice([128, 256, 4 * rng.randrange(18, 64)])
        ny, nz = logu(24, 256), logu(24, 256)
        return _steps_case((nx, ny, nz), rng.choice([8, 16, 20]), nu=nu, force=rng.choice([0.0, 1e-6]),
                           monitor=rng.choice([0, 4]))
    if kind == "storage3d":
        nx = rng.choice([128, 256, 384, 8 * rng.randrange(9, 48)])
        return _steps_case((nx, logu(32, 256), logu(32, 200)), rng.choice([8, 12, 16]), nu=nu, u0=0.05,
                           storage=rng.choice(["bf16", "f16"]), stochastic=rng.choice([False, False, True]))
    if kind == "walls3d":
        return _steps_case((logu(24, 200), logu(24, 200), logu(24, 200)), rng.choice([16, 32]), nu=nu, u0=0.08,
                           bc=rng.choice(["cavity", "cavity", "channel"]), monitor=rng.choice([0, 8]))
    if kind == "ragged3d":
        return _steps_case((logu(20, 320), logu(20, 200), logu(20, 200)), rng.choice([8, 16, 24]), nu=nu,
                           storage=rng.choice(["f32", "f32", "f32", "bf16"]))
    if kind == "variant3d":
        opt = rng.choice([dict(alpha=0.03), dict(alpha=0.03), dict(nu_p=0.1), dict(semi=True)])
        nx = rng.choice([128, 256, logu(40, 256)])
        return _steps_case((nx, logu(32, 200), logu(32, 160)), rng.choice([8, 12, 16]), nu=nu, **opt)
    if rng.random() < 0.4:
        return dict(kind="adjoint", lattice=9, nx=logu(48, 800), ny=logu(48, 800), nz=1, steps=rng.choice([16, 24, 40]),
                    bc=rng.choice(["periodic", "cavity"]), nu=nu, u0=0.02)
    return dict(kind="adjoint", lattice=19, nx=rng.choice([128, logu(24, 160)]), ny=logu(24, 128), nz=logu(24, 128),
                steps=rng.choice([9, 16, 24]), bc=rng.choice(["periodic", "periodic", "cavity"]), nu=nu, u0=0.02)


# ---- inputs ------------------------------------------------------------------------


def _waves(rng, shape, amp):
    """A product wave of random low wave numbers and phases over shape (z, y, x order)
    and its factors: per axis (sin, cos, wave number) as broadcastable arrays."""
    out = []
    for a, n in enumerate(shape):
        k = 2 * math.pi * int(rng.integers(1, 4)) / n
        view = [1] * len(shape)
        view[a] = n
        t = (torch.arange(n, dtype=torch.float64, device="cuda") * k + float(rng.uniform(0, 2 * math.pi))).view(view)
        out.append((torch.sin(t), torch.cos(t), k))
    return out


def _flow(rng, shape, u0):
    """A smooth divergence-free velocity of a few Taylor-Green cells of random wave
    numbers and phases, with the density deviation that goes with it: (d, ux, uy[, uz])."""
    dim = len(shape)
    u = [torch.zeros(shape, dtype=torch.float64, device="cuda") for _ in range(dim)]  # x, y[, z]
    d = torch.zeros(shape, dtype=torch.float64, device="cuda")
    planes = [(0, 1)] if dim == 2 else [(0, 1), (1, 2), (2, 0)]
    for i, j in planes:
        w = _waves(rng, shape, u0)
        ax, ay = w[dim - 1 - i], w[dim - 1 - j]  # factors of axes i and j
        rest = 1.0
        for a in range(dim):
            if a not in (i, j):
                rest = w[dim - 1 - a][1]
        amp = u0 / (len(planes) * max(ax[2], ay[2]))
        u[i] += amp * ay[2] * ax[0] * ay[1] * rest
        u[j] -= amp * ax[2] * ax[1] * ay[0] * rest
        d += 0.75 * u0 * u0 / len(planes) * ((2 * ax[1] ** 2 - 1) + (2 * ay[1] ** 2 - 1)) * rest
    return [t.to(torch.float32).contiguous() for t in [d] + u]


def _shape(case):
    return (case["ny"], case["nx"]) if case["lattice"] == 9 else (case["nz"], case["ny"], case["nx"])


def _lid(case):
    if case.get("bc", "periodic") == "periodic":
        return None
    if case["lattice"] == 9 or case["bc"] == "channel":
        return (0.1, 0.0) if case["lattice"] == 9 else (0.05, 0.0, 0.0)
    return (math.sqrt(2) / 20, math.sqrt(2) / 20, 0.0)


def _force(case):
    g = case.get("force", 0.0)
    return None if not g else ((g, 0.0) if case["lattice"] == 9 else (g, 0.0, -0.5 * g))


def _ensemble_dims(case):
    rng = np.random.default_rng(case["dims_seed"])
    lo, hi = math.log(case["smin"]), math.log(case["smax"])
    dims = [tuple(int(round(math.exp(v))) for v in rng.uniform(lo, hi, 2)) for _ in range(case["domains"])]
    return dims, [float(v) for v in rng.uniform(0.002, 0.05, case["domains"])]


def _inputs(case, seed):
    """The initial fields (and what else varies with the seed), from the seed alone."""
    rng = np.random.default_rng(seed)
    if case["kind"] == "ensemble":
        dims, _ = _ensemble_dims(case)
        doms = [_flow(rng, (ny, nx), case["u0"]) for nx, ny in dims]
        return {"fields": [torch.cat([f[k].reshape(-1) for f in doms]) for k in range(3)]}
    shape = _shape(case)
    got = {"fields": _flow(rng, shape, case["u0"])}
    if case["kind"] == "driven":
        base = _flow(rng, shape, 1e-5)
        ph = float(rng.uniform(0, 2 * math.pi))
        got["g"] = [[(b * math.cos(0.1 * t + ph)).contiguous() for b in base[1:]] for t in range(case["steps"])]
    if case["kind"] == "adjoint":
        got["lam"] = _flow(rng, shape, 1.0)
    if case.get("alpha"):
        w = _waves(rng, shape, 1.0)
        t = torch.ones(shape, dtype=torch.float64, device="cuda")
        for s, c, _ in w:
            t = t * s
        got["T"] = (1.0 + 0.5 * t).to(torch.float32).contiguous()
    return got


def prepare(case, seed):
    state = dict(case=case, **_inputs(case, seed))
    if case["kind"] == "ensemble":
        dims, nus = _ensemble_dims(case)
        state["sim"] = lw.LwacmBatch(lw.D2Q9, dims, nus, mode=case["mode"], tile=case["tile"])
        return state
    kw = {}
    if case["kind"] == "steps":
        kw = dict(storage=STORAGES[case["storage"]], force=_force(case), bulk_gamma=case["gamma"] or None,
                  scalar_alpha=case["alpha"] or None, semi_implicit=case["semi"], stochastic_rounding=case["stochastic"])
    if case["kind"] == "driven":
        kw = dict(force_field=True)
    sim = lw.Lwacm(case["lattice"], case["nx"], case["ny"], case["nz"], case["nu"], BCS[case.get("bc", "periodic")],
                   lid=_lid(case), **kw)
    if case.get("nu_p"):
        sim.set_option(lw.OPT_NU_P, case["nu_p"])
    if case["kind"] == "steps":  # a program that steps often captures its step graph ahead
        sim.set_fields(*state["fields"])
        sim.prepare(case["monitor"] or case["steps"])
    if case["kind"] == "adjoint":
        for t in state["fields"]:
            t.requires_grad_(True)
        state["nu"] = torch.tensor(case["nu"], dtype=torch.float32, requires_grad=True)
    if case["kind"] == "steps" and (case["alpha"] or case["gamma"]):
        state["extra"] = torch.empty(_shape(case), dtype=torch.float32, device="cuda")
    state["sim"] = sim
    return state


# ---- one pass ----------------------------------------------------------------------

SERIES = ("mass", "jx", "jy", "jz", "ke", "umax", "mpar", "mperp")


def run(state):
    case, sim = state["case"], state["sim"]
    if case["kind"] == "adjoint":
        outs = lw.run(sim, case["steps"], state["nu"], *state["fields"])
        grads = torch.autograd.grad(outs, [*state["fields"], state["nu"]], grad_outputs=state["lam"])
        return {"fields": [t.detach() for t in outs], "grads": list(grads)}
    sim.set_fields(*state["fields"])
    if case["kind"] == "driven":
        for g in state["g"]:
            sim.set_force_field(*g)
            sim.step(1)
        return {"fields": list(sim.fields())}
    if case["kind"] == "ensemble":
        sim.step(case["steps"])
        return {"fields": list(sim.fields())}
    if case["alpha"]:
        sim.set_scalar(state["T"])
    out = {}
    if case["monitor"]:
        series = []
        for _ in range(case["steps"] // case["monitor"]):
            sim.step(case["monitor"])
            q = sim.diagnostics()
            series.append([q[k] for k in SERIES])
        out["series"] = np.array(series, dtype=np.float32)
    else:
        sim.step(case["steps"])
    out["fields"] = list(sim.fields())
    if "extra" in state:  # the scalar or the trace, copied on the device through the C ABI
        get = lw.load().lwacm_get_scalar if case["alpha"] else lw.load().lwacm_get_trace
        status = get(sim._h, state["extra"].data_ptr(), lw.F32, lw.DEVICE)
        if status != lw.OK:
            raise lw.LwacmError(status, "reading the scalar or the trace")
        out["extra"] = state["extra"]
    return out


# ---- work --------------------------------------------------------------------------


def work(case):
    """Bytes: the inputs read once and the results written once, and, where a state does
    not stay on the chip between steps, the state read and written once in each step.
    Flops: the moment form's per node and step (D2Q9 62, D3Q19 146, the variants' and
    the adjoint's extra operations on top)."""
    three_d = case["lattice"] == 19
    if case["kind"] == "ensemble":
        n = sum(a * b for a, b in _ensemble_dims(case)[0])
    else:
        n = case["nx"] * case["ny"] * case["nz"]
    nf, flops = (4, 146) if three_d else (3, 62)
    esize = 2 if case.get("storage", "f32") != "f32" else 4
    extra = 1 if case.get("alpha") or case.get("gamma") else 0
    flops += (60 if case.get("alpha") else 0) + (40 if case.get("gamma") else 0) + (20 if case.get("nu_p") else 0)
    flops += 60 if case.get("semi") else 0
    steps = case["steps"]
    once = n * nf * (4 + esize) + n * 4 * ((2 if case.get("alpha") else 0) + (1 if case.get("gamma") else 0))
    per_step = 2 * n * (nf + extra) * esize
    moved = once if n * (nf + extra) * esize < L2_BYTES else once + (steps - 1) * per_step
    if case["kind"] == "driven":
        moved += steps * n * 2 * 4
    if case["kind"] == "adjoint":
        # forward, then a sweep that reads the state and moves the adjoint state each step
        moved = 2 * moved + (0 if n * nf * 4 < L2_BYTES else steps * n * nf * 4)
        flops = flops + 2 * flops
    return {"bytes": float(moved), "flops": float(flops) * n * steps}


# ---- the method in 64 bits -----------------------------------------------------------


def _links(Q):
    if Q == 9:
        c = [(x, y, 0) for x in (-1, 0, 1) for y in (-1, 0, 1)]
        w = {0: 4 / 9, 1: 1 / 9, 2: 1 / 36}
    else:
        c = [(x, y, z) for x in (-1, 0, 1) for y in (-1, 0, 1) for z in (-1, 0, 1) if abs(x) + abs(y) + abs(z) < 3]
        w = {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}
    return [(v, w[sum(map(abs, v))]) for v in c]


def _shift(t, c):
    """t at the upwind node x - c."""
    dims, by = [], []
    for a in range(t.dim()):
        if c[a]:
            dims.append(t.dim() - 1 - a)
            by.append(c[a])
    return torch.roll(t, by, dims) if dims else t


def _dot(c, u):
    e = 0.0
    for a, ua in enumerate(u):
        if c[a]:
            e = e + ua if c[a] > 0 else e - ua
    return e


def _beyond(shape, c, axes):
    """Nodes whose upwind source along c lies beyond a walled face, and beyond the top
    of each axis, as boolean arrays (None where no such node exists)."""
    hit, top = None, {}
    for a in axes:
        if not c[a]:
            continue
        n = shape[len(shape) - 1 - a]
        view = [1] * len(shape)
        view[len(shape) - 1 - a] = n
        at = torch.zeros(n, dtype=torch.bool, device="cuda")
        at[0 if c[a] > 0 else n - 1] = True
        at = at.view(view).expand(shape)
        hit = at if hit is None else hit | at
        if c[a] < 0:
            top[a] = at
    return hit, top


def _step(f, case, nu, g=None, tr=None, T=None):
    """One time step in FP64: f = (d, ux, uy[, uz]); returns the new f, trace and scalar."""
    d, u = f[0], f[1:]
    links, dim = _links(case["lattice"]), len(u)
    rho, s, a = 1 + d, 18 * nu, 1 - 6 * nu
    sq = sum(c * c for c in u)
    bc = case.get("bc", "periodic")
    walled = [] if bc == "periodic" else ([1] if bc == "channel" else list(range(dim)))
    lid_axis = 1 if bc == "channel" else dim - 1
    lid = _lid(case)
    gamma, nu_p = case.get("gamma", 0.0), case.get("nu_p", 0.0)
    sdelta = 18 * (nu_p - nu) if nu_p else 0.0

    def factor(v, ci, dev):  # the product form's factor in one direction and its change with the trace
        return (1 - 1 / 3 - v * v, -dev) if ci == 0 else ((1 / 3 + v * v + ci * v) / 2, dev / 2)

    def star(c, w, d_, u_):  # pre-combined link value less its weight
        e = _dot(c, u_)
        q = sum(k * k for k in u_)
        v = w * (d_ + (1 + d_) * (s * e + 4.5 * e * e - 1.5 * q))
        odd = None
        if gamma:
            h = gamma * tr / 2
            A, ax = factor(u_[0], c[0], h)
            B, ay = factor(u_[1], c[1], h)
            A0, ax0 = factor(-u_[0], c[0], h)
            B0, ay0 = factor(-u_[1], c[1], h)
            one = (1 + d_) * ((A + ax) * (B + ay) - A * B)
            two = (1 + d_) * ((A0 + ax0) * (B0 + ay0) - A0 * B0)
            odd = (one - two) / 2
            v = v + one - a * odd
        return v, e, odd

    dsum, jsum, dp, trace, Tn = 0.0, [0.0] * dim, 0.0, 0.0, 0.0
    at = 1 - 6 * case["alpha"] if T is not None else 0.0
    for c, w in links:
        v, e, odd = star(c, w, d, u)
        gi = _shift(v, c)
        if walled and any(c[k] for k in walled):
            hit, top = _beyond(d.shape, c, walled)
            own = star(tuple(-k for k in c), w, d, u)[0]
            gi = torch.where(hit, own, gi)
            if lid_axis in top:
                gi = gi + top[lid_axis].double() * (w * 36 * nu * _dot(c, lid))
        dsum = dsum + gi
        for k in range(dim):
            if c[k]:
                jsum[k] = jsum[k] + gi if c[k] > 0 else jsum[k] - gi
        if sdelta and any(c):
            dp = dp + _shift(w * rho * e, c) + (_shift(odd, c) / 3 if odd is not None else 0.0)
        if gamma:
            trace = trace + (sum(k * k for k in c) - 2 / 3) * gi
        if T is not None:
            Tn = Tn + _shift(w * ((1 - at) * (T + 4.5 * e * e - 1.5 * sq) + 3 * T * e), c)
    if T is not None:
        Tn = Tn + at * T
    dn = dsum + sdelta * dp
    force = _force(case)
    j = [a * rho * u[k] + jsum[k] for k in range(dim)]
    if force is not None:
        j = [j[k] + rho * force[k] for k in range(dim)]
    if g is not None:
        j = [j[k] + rho * g[k] for k in range(dim)]
    un = [j[k] / (1 + dn) for k in range(dim)]
    trn = trace / (1 + dsum) - sum(k * k for k in un) if gamma else None
    if case.get("semi"):
        s = s + sdelta
        dn = sum(_shift(star(c, w, d, un)[0], c) for c, w in links)
    return [dn] + un, trn, (Tn if T is not None else None)


def _quantities(f):
    rho, u = 1 + f[0], list(f[1:]) + [torch.zeros_like(f[0])] * (4 - len(f))
    sq = sum(c * c for c in u)
    two = len(f) == 3
    vals = [f[0].sum()] + [(rho * c).sum() for c in u] + [0.5 * (rho * sq).sum(), sq.max().sqrt()]
    vals += [torch.zeros_like(vals[0])] * 2 if two else [0.5 * ((u[0] + u[1]) ** 2).sum(), 0.5 * ((u[0] - u[1]) ** 2).sum()]
    return [float(v) for v in vals]


def exact(case, seed):
    got = _inputs(case, seed)
    f = [t.double() for t in got["fields"]]
    if case["kind"] == "ensemble":
        dims, nus = _ensemble_dims(case)
        outs, off = [[], [], []], 0
        for (nx, ny), nu in zip(dims, nus):
            part = [t[off:off + nx * ny].view(ny, nx) for t in f]
            off += nx * ny
            for _ in range(case["steps"]):
                part = _step(part, case, nu)[0]
            for k in range(3):
                outs[k].append(part[k].reshape(-1))
        return {"fields": [torch.cat(o) for o in outs]}
    if case["kind"] == "adjoint":
        from torch.utils.checkpoint import checkpoint
        leaves = [t.requires_grad_(True) for t in f]
        nu = torch.tensor(float(np.float32(case["nu"])), dtype=torch.float64, device="cuda", requires_grad=True)
        now = leaves
        for _ in range(case["steps"]):
            now = checkpoint(lambda *a: tuple(_step(list(a[:-1]), case, a[-1])[0]), *now, nu, use_reentrant=False)
        grads = torch.autograd.grad(now, [*leaves, nu], grad_outputs=[t.double() for t in got["lam"]])
        return {"fields": [t.detach() for t in now], "grads": [t.detach() for t in grads[:-1]] + [grads[-1].cpu()]}
    tr = torch.zeros_like(f[0]) if case.get("gamma") else None
    T = got["T"].double() if "T" in got else None
    series, out = [], {}
    for t in range(case["steps"]):
        f, tr, T = _step(f, case, case["nu"], g=[k.double() for k in got["g"][t]] if "g" in got else None, tr=tr, T=T)
        if case.get("monitor") and (t + 1) % case["monitor"] == 0:
            series.append(_quantities(f))
    if case.get("monitor"):
        out["series"] = np.array(series, dtype=np.float64)
    out["fields"] = list(f)
    if T is not None or tr is not None:
        out["extra"] = T if T is not None else tr
    return out
