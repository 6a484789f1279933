"""The measured work: runs of the coupled lattice-Boltzmann + WENO solver as its users make them.

A pass is one job through the public Python API: initialise a handle from fields on the
device, advance it a few dozen to a few hundred steps, and take the fields (and the masses a
tank experiment records) back.  A long run is the same steps many times over, so a job's time
is that of its steps plus one initialisation and one read-out.  The plan that a program keeps
between jobs -- the handle and its workspace -- is made in ``prepare``.

``exact`` restates the method (D2Q9 / D3Q19 BGK with Guo forcing and half-way bounce-back,
flux-split or upwind WENO with central diffusion and settling, SSP-RK3, first-order upwind
sugar) in 64-bit torch operations on whole fields.
"""
import math
import random

import torch

from paper_2106_07694_gb300 import autograd, lbm_wenoc as lw

DEVICE = "cuda" if torch.cuda.is_available() else "cpu"

TAU, KAPPA, U_CAP, PHI0 = 0.6, 1e-3, 0.1, 1.19e-3
# the two-layer tank (particles over a sugar solution): glass beads of 3 g/l over
# rho_f = 1008.4 kg/m3, mapped to lattice units as in the two-layer workload
SUGAR = dict(gravity=5.53e-3, density_contrast=1.808e-3, sugar=True, sugar_contrast=8.4e-3,
             sugar_diffusivity=1.7e-5, phi0=PHI0, vs_sugar=5.53e-3)
CLASS_VS = (5e-4, 1e-3, 2e-3)


def listed():
    return [
        # the smallest lattice in FP64: what a new model term is checked on against a 64-bit
        # reference before it is trusted in FP32
        dict(name="check_128x256_f64", kind="sim", nx=128, ny=256, nz=0, steps=40, dtype="f64", flow=0.0),
        # the smallest lattice in FP32, stepped ten at a time with the deposit and the mass
        # below mid-height read in between (the m_b(t) and flux curves): launches and latency
        dict(name="monitor_128x256", kind="monitor", nx=128, ny=256, nz=0, steps=10, reads=12, dtype="f32", flow=0.0),
        # a laboratory-sized tank with the flow already turning over, resumed from given
        # velocities
        dict(name="tank_512x1024", kind="sim", nx=512, ny=1024, nz=0, steps=100, dtype="f32", flow=0.02),
        # a tank whose sides are no round numbers: ragged strips, odd rows
        dict(name="ragged_1260x701", kind="sim", nx=1260, ny=701, nz=0, steps=60, dtype="f32", flow=0.02),
        # the headline lattice
        dict(name="main_2048x4096", kind="sim", nx=2048, ny=4096, nz=0, steps=32, dtype="f32", flow=0.02),
        # the paper's two-layer experiment: particles over a heavier sugar layer
        dict(name="sugar_1024x2048", kind="sim", nx=1024, ny=2048, nz=0, steps=40, dtype="f32", flow=0.01, sugar=True),
        # the paper's own order of WENO in place of the fifth-order default
        dict(name="weno3_1536x2048", kind="sim", nx=1536, ny=2048, nz=0, steps=32, dtype="f32", flow=0.02,
             scheme="weno3"),
        # three particle sizes settling at their own speeds
        dict(name="classes_1024x1536", kind="sim", nx=1024, ny=1536, nz=0, steps=24, dtype="f32", flow=0.01, classes=3),
        # a 3D tank, D3Q19, at the full benchmark size: the largest job
        dict(name="main_256x256x512", kind="sim", nx=256, ny=256, nz=512, steps=12, dtype="f32", flow=0.02),
        # the paper's simulation as it ran it, on a small ragged box: D3Q19, sugar, third-order WENO
        dict(name="paper_120x90x200", kind="sim", nx=120, ny=90, nz=200, steps=24, dtype="f32", flow=0.01, sugar=True,
             scheme="weno3"),
        # the parameter sweep as one job: instances of different sizes and physics together
        dict(name="sweep_64", kind="sweep", count=64, sizes=0, steps=16),
        # an inversion's inner loop: deposited mass and its gradient through autograd
        dict(name="gradient_512x1024", kind="gradient", nx=512, ny=1024, steps=100),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _sides2d(rng, nodes):
    nx = max(32, min(4096, int(math.sqrt(nodes * _log(rng, 0.3, 1.5)) / 4) * 4))  # nx is a multiple of four
    return nx, max(33, min(8192, int(nodes / nx)))


def draw(rng):
    kind = rng.choice(["sim2d", "sim2d", "sim2d", "variant2d", "variant2d", "sim3d", "sim3d", "f64", "monitor",
                       "sweep", "gradient"])
    if kind in ("sim2d", "variant2d"):
        nx, ny = _sides2d(rng, _log(rng, 3e4, 8e6))
        case = dict(kind="sim", nx=nx, ny=ny, nz=0, steps=rng.randint(8, 30), dtype="f32", flow=rng.uniform(0.005, 0.03))
        if kind == "variant2d":
            case.update(rng.choice([dict(sugar=True), dict(scheme="weno3"), dict(scheme="sign"), dict(classes=2),
                                    dict(classes=3), dict(sugar=True, scheme="weno3")]))
        return case
    if kind == "sim3d":
        nodes = _log(rng, 1e5, 1.6e7)
        nz = max(16, int((nodes * _log(rng, 1.0, 4.0)) ** (1 / 3)))
        nx = max(16, int(math.sqrt(nodes / nz * _log(rng, 0.6, 1.6)) / 4) * 4)
        ny = max(16, int(nodes / (nx * nz)))
        case = dict(kind="sim", nx=nx, ny=ny, nz=nz, steps=rng.randint(4, 12), dtype="f32", flow=rng.uniform(0.005, 0.03))
        case.update(rng.choice([{}, {}, dict(sugar=True), dict(scheme="weno3"), dict(sugar=True, scheme="weno3")]))
        return case
    if kind == "f64":
        nx, ny = _sides2d(rng, _log(rng, 1e4, 2e5))
        return dict(kind="sim", nx=nx, ny=ny, nz=0, steps=rng.randint(8, 40), dtype="f64", flow=rng.uniform(0.0, 0.03))
    if kind == "monitor":
        nx, ny = _sides2d(rng, _log(rng, 1e4, 2e5))
        return dict(kind="monitor", nx=nx, ny=ny, nz=0, steps=rng.randint(1, 20), reads=rng.randint(2, 12), dtype="f32",
                    flow=rng.uniform(0.0, 0.02))
    if kind == "sweep":
        return dict(kind="sweep", count=rng.randint(3, 48), sizes=rng.randint(1, 10**6), steps=rng.randint(4, 16))
    nx, ny = _sides2d(rng, _log(rng, 2e4, 5e5))
    return dict(kind="gradient", nx=nx, ny=ny, steps=rng.randint(20, 90))


# ---- inputs

def _shape(case):
    return (case["nx"], case["ny"], case["nz"]) if case["nz"] else (case["nx"], case["ny"])


def _physics(case):
    kw = dict(tau=TAU, gravity=1e-5, density_contrast=1.0, settling_velocity=1e-3, diffusivity=KAPPA)
    if case.get("sugar"):
        kw.update(SUGAR)
    if case.get("scheme") == "weno3":
        kw.update(weno3=True)
    if case.get("scheme") == "sign":
        kw.update(sign_split=True)
    if case.get("classes"):
        kw.update(class_vs=CLASS_VS[:case["classes"]])
    return kw


def _front(shape, gen, frac, dtype, background=0.05):
    """A particle layer over a dilute background: a tanh front at `frac` of the height, rippled by
    a few modes, with 1e-3 of noise at every node."""
    nv = shape[-1]
    v = torch.arange(nv, device=DEVICE, dtype=torch.float32) + 0.5
    x = torch.arange(shape[0], device=DEVICE, dtype=torch.float32) * (2 * math.pi / shape[0])
    ph = torch.rand(4, generator=gen, device=DEVICE) * 2 * math.pi
    ripple = 1.5 * torch.cos(3 * x + ph[0]) + 1.0 * torch.cos(5 * x + ph[1])
    if len(shape) == 3:
        y = torch.arange(shape[1], device=DEVICE, dtype=torch.float32) * (2 * math.pi / shape[1])
        h = (v - frac * nv)[:, None, None] + ripple[None, None, :] + 1.5 * torch.cos(2 * y + ph[2])[None, :, None]
    else:
        h = (v - frac * nv)[:, None] + ripple[None, :]
    c = background + (1 - background) * 0.5 * (1 + torch.tanh(h / 2))
    c = c + 1e-3 * (2 * torch.rand(c.shape, generator=gen, device=DEVICE) - 1)
    return c.to(dtype).contiguous()


def _rolls(shape, gen, amplitude, dtype):
    """Divergence-free convection rolls of the given largest speed (None when at rest)."""
    if not amplitude:
        return None
    nx, nv = shape[0], shape[-1]
    ph = torch.rand(2, generator=gen, device=DEVICE) * 2 * math.pi
    v = (torch.arange(nv, device=DEVICE, dtype=torch.float32) + 0.5) * (math.pi / nv)

    def pair(n, m, phase):
        k = 2 * math.pi * m / n
        s = amplitude / (2 * max(k, math.pi / nv)) * (1 if len(shape) == 3 else 2)
        a = torch.arange(n, device=DEVICE, dtype=torch.float32) * k + phase
        return (s * (math.pi / nv)) * torch.sin(2 * v)[:, None] * torch.sin(a), (-s * k) * (torch.sin(v) ** 2)[:, None] * torch.cos(a)

    ux, uv = pair(nx, 2, ph[0])
    if len(shape) == 2:
        return torch.stack([ux, uv]).to(dtype).contiguous()
    uy, uw = pair(shape[1], 1, ph[1])
    grid = (nv, shape[1], nx)
    u = torch.stack([ux[:, None, :].expand(grid), uy[:, :, None].expand(grid), uv[:, None, :] + uw[:, :, None]])
    return u.to(dtype).contiguous()


def _sim_inputs(case, seed):
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(seed)
    dtype = torch.float64 if case["dtype"] == "f64" else torch.float32
    shape = _shape(case)
    frac = 0.5 if case.get("sugar") else 0.75
    k = case.get("classes", 1)
    c = [_front(shape, gen, frac, dtype) / k for _ in range(k)]
    u = _rolls(shape, gen, case["flow"], dtype)
    S = None
    if case.get("sugar"):  # the lower layer, without noise
        v = torch.arange(shape[-1], device=DEVICE, dtype=torch.float32) + 0.5
        prof = 0.5 * (1 - torch.tanh((v - frac * shape[-1]) / 2))
        S = prof.reshape((-1,) + (1,) * (len(shape) - 1)).expand(c[0].shape).to(dtype).contiguous()
    return c, u, S


def _sweep_members(case):
    """Lattices from 256 x 512 to 1024 x 2048, buoyancy and settling speed over the paper's ranges."""
    r = random.Random(case["sizes"])
    out = []
    for _ in range(case["count"]):
        nx = 64 * r.randint(4, 16)
        out.append(dict(shape=(nx, 2 * nx), tau=TAU, gravity=_log(r, 2e-6, 1e-4), density_contrast=1.0,
                        settling_velocity=_log(r, 2e-4, 4e-3), diffusivity=KAPPA))
    return out


def _sweep_inputs(case, seed):
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(seed)
    return [_front(m["shape"], gen, 0.75, torch.float32) for m in _sweep_members(case)]


GRADIENT = dict(tau=TAU, gravity=2e-3, density_contrast=1.0, diffusivity=0.02, lf_alpha=0.25, u_cap=0.2)
GRADIENT_VS = 0.05


def _gradient_inputs(case, seed):
    """A stirred suspension, rough at the scale of the nodes."""
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(seed)
    return 0.5 + 0.4 * (2 * torch.rand((case["ny"], case["nx"]), generator=gen, device=DEVICE) - 1)


# ---- one pass

def prepare(case, seed):
    if case["kind"] == "gradient":
        return dict(case=case, c0=_gradient_inputs(case, seed).requires_grad_(),
                    vs=torch.tensor(GRADIENT_VS, dtype=torch.float64, requires_grad=True))
    if case["kind"] == "sweep":
        members = _sweep_members(case)
        n = [m["shape"][0] * m["shape"][1] for m in members]
        return dict(case=case, batch=lw.Batch(members), c0=_sweep_inputs(case, seed), nodes=n,
                    rho=torch.empty(sum(n), device="cuda"), u=torch.empty(2 * sum(n), device="cuda"),
                    c=torch.empty(sum(n), device="cuda"))
    c, u, S = _sim_inputs(case, seed)
    return dict(case=case, sim=lw.Simulation(_shape(case), fp64=case["dtype"] == "f64", **_physics(case)), c=c, u=u, S=S)


def run(state):
    case = state["case"]
    if case["kind"] == "gradient":
        c0, vs = state["c0"], state["vs"]
        c0.grad = vs.grad = None
        J = autograd.deposited_mass(c0, vs, case["steps"], (case["nx"], case["ny"]), **GRADIENT)
        J.backward()
        return dict(J=J.item(), dc0=c0.grad, dvs=vs.grad.item())
    if case["kind"] == "sweep":
        b = state["batch"]
        for inst, c0 in zip(b.instances, state["c0"]):
            inst.init(c0)
        b.step(case["steps"])
        at = 0
        deposits = []
        for inst, n in zip(b.instances, state["nodes"]):
            lw.lbm_wenoc_fields(inst.handle, state["rho"][at:at + n], state["u"][2 * at:2 * (at + n)],
                                state["c"][at:at + n])
            deposits.append(inst.deposit)
            at += n
        return dict(rho=state["rho"], u=state["u"], c=state["c"], deposits=torch.tensor(deposits, dtype=torch.float32))
    sim, c, u, S = state["sim"], state["c"], state["u"], state["S"]
    sim.init(c[0], u)
    for k in range(1, len(c)):
        sim.set_class(k, c[k])
    if len(c) > 1:
        sim.set_class(0, c[0])
    if S is not None:
        sim.set_sugar(S)
    out = {}
    if case["kind"] == "monitor":
        mid = case["ny"] // 2
        out["series"] = []
        for _ in range(case["reads"]):
            sim.step(case["steps"])
            out["series"].append([sim.deposit, sim.mass_below(mid)])
    else:
        sim.step(case["steps"])
    out["rho"], out["u"], out["c"] = sim.fields("cuda")
    if S is not None:
        out["S"] = sim.sugar("cuda")
    if len(c) > 1:
        out["classes"] = [sim.class_field(k, "cuda") for k in range(len(c))]
    out["deposit"] = sim.deposit
    return out


# ---- what a pass cannot do without

def _step_work(q, dim, es, scheme="", sugar=False, classes=1):
    """Bytes and operations of one node and step: the populations and the concentrations once
    in and once out; moments, collision and forcing about 29 operations a population; the
    reconstructions, split, diffusion, divergence and combination of the three stages."""
    nbytes = es * (2 * q + 2 * classes + (2 if sugar else 0))
    face = {"": 2 * 70, "weno3": 2 * 21, "sign": 70}[scheme]
    transport = 3 * (dim * (face + 10) + 5)
    return nbytes, 29 * q + classes * transport + (12 * dim if sugar else 0)


def work(case):
    if case["kind"] == "sweep":
        n = sum(m["shape"][0] * m["shape"][1] for m in _sweep_members(case))
        b, f = _step_work(9, 2, 4)
        return dict(bytes=n * (case["steps"] * b + 4 * 5), flops=n * case["steps"] * f)
    if case["kind"] == "gradient":
        n = case["nx"] * case["ny"]
        b, f = _step_work(9, 2, 4)
        # forward, then back: the adjoint populations and c once in and out and the step's state
        # read; each face's reconstructions with their derivatives, about 2.5 times the forward's
        return dict(bytes=n * (case["steps"] * (2 * b + 24) + 8), flops=n * case["steps"] * (f + 2.5 * f))
    n = case["nx"] * case["ny"] * max(1, case["nz"])
    es = 8 if case["dtype"] == "f64" else 4
    q, dim = (19, 3) if case["nz"] else (9, 2)
    b, f = _step_work(q, dim, es, case.get("scheme", ""), bool(case.get("sugar")), case.get("classes", 1))
    steps = case["steps"] * case.get("reads", 1)
    fields = es * (2 + (2 if case["flow"] else 1) * dim + 1)
    return dict(bytes=n * (steps * b + fields), flops=n * steps * f)


# ---- the method in 64 bits, on whole fields

_C2 = [(0, 0), (1, 0), (-1, 0), (0, 1), (0, -1), (1, 1), (-1, -1), (1, -1), (-1, 1)]
_C3 = [c for c in [(x, y, z) for x in (-1, 0, 1) for y in (-1, 0, 1) for z in (-1, 0, 1)] if 0 < sum(map(abs, c)) < 3]
_C3 = [(0, 0, 0)] + _C3


def _weights(cs):
    rest, one, two = (4 / 9, 1 / 9, 1 / 36) if len(cs) == 9 else (1 / 3, 1 / 18, 1 / 36)
    return [(rest, one, two)[sum(map(abs, c))] for c in cs]


def _weno5(a, b, c, d, e):
    w0 = 0.1 / (1e-6 + 13 / 12 * (a - 2 * b + c) ** 2 + 0.25 * (a - 4 * b + 3 * c) ** 2) ** 2
    w1 = 0.6 / (1e-6 + 13 / 12 * (b - 2 * c + d) ** 2 + 0.25 * (b - d) ** 2) ** 2
    w2 = 0.3 / (1e-6 + 13 / 12 * (c - 2 * d + e) ** 2 + 0.25 * (3 * c - 4 * d + e) ** 2) ** 2
    q = w0 * (2 * a - 7 * b + 11 * c) + w1 * (-b + 5 * c + 2 * d) + w2 * (2 * c + 5 * d - e)
    return q / (6 * (w0 + w1 + w2))


def _weno3(a, b, c, d, e):
    w0, w1 = 2 / (1e-6 + (d - c) ** 2) ** 2, 1 / (1e-6 + (c - b) ** 2) ** 2
    return (w0 * (c + d) + w1 * (3 * c - b)) / (2 * (w0 + w1))


def _extend(a, axis, wall, odd=False):
    """Three more nodes on each side: the periodic images, or the mirror images behind a wall."""
    n = a.shape[axis]
    lo, hi = a.narrow(axis, 0, 3), a.narrow(axis, n - 3, 3)
    if wall:
        lo, hi = lo.flip(axis), hi.flip(axis)
        return torch.cat([-lo, a, -hi] if odd else [lo, a, hi], axis)
    return torch.cat([hi, a, lo], axis)


def _rate(c, u, vs, par):
    """-div of the advective, settling and diffusive flux of c (axes of the arrays: vertical first)."""
    dim, alpha, scheme = c.dim(), par["alpha"], par["scheme"]
    weno = _weno3 if scheme == "weno3" else _weno5
    L = 0
    for d in range(dim):
        axis, wall = dim - 1 - d, d == dim - 1
        n = c.shape[axis]
        C = _extend(c, axis, wall)
        W = _extend(u[d], axis, wall, odd=True)
        if wall:
            W = W - (_extend(vs, axis, True) if isinstance(vs, torch.Tensor) and vs.dim() else vs)
        at = lambda a, k: a.narrow(axis, k, n + 1)  # noqa: E731  stencil node k of every face
        if scheme == "sign":
            h = W / alpha * C
            left = at(W, 2) + at(W, 3) >= 0
            F = alpha * torch.where(left, weno(*(at(h, k) for k in range(5))), weno(*(at(h, 5 - k) for k in range(5))))
        else:
            p, m = 0.5 * (W / alpha + 1) * C, 0.5 * (W / alpha - 1) * C
            F = alpha * (weno(*(at(p, k) for k in range(5))) + weno(*(at(m, 5 - k) for k in range(5))))
        F = F - par["kappa"] * (at(C, 3) - at(C, 2))
        if wall:
            floor = -(vs * c).narrow(axis, 0, 1)
            F = torch.cat([floor, F.narrow(axis, 1, n - 1), torch.zeros_like(floor)], axis)
        L = L + F.narrow(axis, 0, n) - F.narrow(axis, 1, n)
    return L


def _stream(g, cs):
    dim = len(cs[0])
    opp = {c: i for i, c in enumerate(cs)}
    out = []
    for i, c in enumerate(cs):
        back = g[opp[tuple(-k for k in c)]]
        a = g[i]
        for d in range(dim - 1):
            if c[d]:
                a = torch.roll(a, c[d], dims=dim - 1 - d)
        n = a.shape[0]
        if c[-1] > 0:
            a = torch.cat([back[:1], a[:n - 1]])
        elif c[-1] < 0:
            a = torch.cat([a[1:], back[n - 1:]])
        out.append(a)
    return out


def _moments(g, c, S, cs, par):
    dim = len(cs[0])
    rho = 1 + sum(g)
    Fv = -par["A"] * c
    if S is not None:
        Fv = Fv - par["gS"] * S * (1 - par["phi0"] * c)
    F = [0.0] * (dim - 1) + [Fv]
    u = [(sum(x * c_[d] for x, c_ in zip(g, cs) if c_[d]) + 0.5 * F[d]) / rho for d in range(dim)]
    return rho, u, Fv


def _advance(g, cls, S, dep, cs, par):
    """One coupled step of the populations g, the class fields cls and the sugar S."""
    w, dim, tau = _weights(cs), len(cs[0]), par["tau"]
    tot = sum(cls[1:], cls[0])
    rho, u, Fv = _moments(g, tot, S, cs, par)
    uu, uF = sum(x * x for x in u), u[-1] * Fv
    post = []
    for x, ci, wi in zip(g, cs, w):
        cu = sum((u[d] * ci[d] for d in range(dim) if ci[d]), torch.zeros_like(rho))
        eq = wi * ((rho - 1) + rho * (3 * cu + 4.5 * cu * cu - 1.5 * uu))
        src = (1 - 0.5 / tau) * wi * (3 * (ci[-1] * Fv - uF) + 9 * cu * (ci[-1] * Fv))
        post.append(x - (x - eq) / tau + src)
    g = _stream(post, cs)
    new, dep = [], list(dep)
    for k, c in enumerate(cls):
        vs = par["vs"][k] * (1 - par["ks"] * S) if S is not None else par["vs"][k]
        c1 = c + _rate(c, u, vs, par)
        c2 = 0.75 * c + 0.25 * (c1 + _rate(c1, u, vs, par))
        c3 = c / 3 + 2 / 3 * (c2 + _rate(c2, u, vs, par))
        dep[k] = dep[k] + ((vs[0] if S is not None else vs) * (c[0] / 6 + c1[0] / 6 + 2 / 3 * c2[0])).sum()
        new.append(c3)
    if S is not None:
        s = S
        for d in range(dim):
            axis, n = dim - 1 - d, S.shape[dim - 1 - d]
            if d == dim - 1:
                lo = torch.cat([S.narrow(axis, 0, 1), S.narrow(axis, 0, n - 1)], axis)
                hi = torch.cat([S.narrow(axis, 1, n - 1), S.narrow(axis, n - 1, 1)], axis)
            else:
                lo, hi = torch.roll(S, 1, axis), torch.roll(S, -1, axis)
            s = s - torch.where(u[d] > 0, u[d] * (S - lo), u[d] * (hi - S)) + par["Ds"] * (hi - 2 * S + lo)
        S = s
    return g, new, S, dep


def _rest(c, u, cs):
    """Equilibrium populations (less their weights) at density one."""
    w, dim = _weights(cs), len(cs[0])
    if u is None:
        return [torch.zeros_like(c) for _ in cs]
    uu = sum(u[d] * u[d] for d in range(dim))
    out = []
    for ci, wi in zip(cs, w):
        cu = sum((u[d] * ci[d] for d in range(dim) if ci[d]), torch.zeros_like(c))
        out.append(wi * (3 * cu + 4.5 * cu * cu - 1.5 * uu))
    return out


def _par(kw, scheme="", vs=None):
    vs = list(kw.get("class_vs") or (kw.get("settling_velocity"),)) if vs is None else vs
    return dict(tau=kw["tau"], A=kw["gravity"] * kw["density_contrast"], vs=vs, kappa=kw["diffusivity"], scheme=scheme,
                alpha=kw.get("lf_alpha") or max(vs) + U_CAP, gS=kw["gravity"] * kw.get("sugar_contrast", 0.0),
                phi0=kw.get("phi0", 0.0), ks=kw.get("vs_sugar", 0.0), Ds=kw.get("sugar_diffusivity", 0.0))


def _forward(cls, u, S, steps, par, every=0, level=0):
    dim = cls[0].dim()
    cs = _C2 if dim == 2 else _C3
    cls = [c.double() for c in cls]
    g = _rest(cls[0], None if u is None else u.double(), cs)
    S = None if S is None else S.double()
    dep, series = [0.0] * len(cls), []
    for t in range(steps):
        g, cls, S, dep = _advance(g, cls, S, dep, cs, par)
        if every and (t + 1) % every == 0:
            d = float(sum(dep))
            series.append([d, float(cls[0][:level].sum()) + d])
    rho, v, _ = _moments(g, sum(cls[1:], cls[0]), S, cs, par)
    return rho, torch.stack(v), cls, S, dep, series


def _exact_gradient(case, seed):
    from torch.utils.checkpoint import checkpoint
    c0 = _gradient_inputs(case, seed).double().requires_grad_()
    vs = torch.tensor(GRADIENT_VS, dtype=torch.float64, device=DEVICE, requires_grad=True)
    par = _par(dict(GRADIENT, settling_velocity=GRADIENT_VS))

    def step(g, c, dep, vs):
        g, (c,), _, (dep,) = _advance(list(g.unbind(0)), [c], None, [dep], _C2, dict(par, vs=[vs]))
        return torch.stack(g), c, dep

    g, c = torch.stack(_rest(c0.detach(), None, _C2)), c0
    dep = torch.zeros((), dtype=torch.float64, device=DEVICE)
    for _ in range(case["steps"]):
        g, c, dep = checkpoint(step, g, c, dep, vs, use_reentrant=False)
    dep.backward()
    return dict(J=dep.item(), dc0=c0.grad, dvs=vs.grad.item())


def exact(case, seed):
    if case["kind"] == "gradient":
        return _exact_gradient(case, seed)
    with torch.no_grad():
        if case["kind"] == "sweep":
            rho, u, c, dep = [], [], [], []
            for m, c0 in zip(_sweep_members(case), _sweep_inputs(case, seed)):
                r, v, (a,), _, (d,), _ = _forward([c0], None, None, case["steps"], _par(m))
                rho.append(r.reshape(-1))
                u.append(v.reshape(-1))
                c.append(a.reshape(-1))
                dep.append(float(d))
            return dict(rho=torch.cat(rho), u=torch.cat(u), c=torch.cat(c), deposits=torch.tensor(dep, dtype=torch.float64))
        cls, u, S = _sim_inputs(case, seed)
        reads = case.get("reads", 0)
        rho, v, cls, S, dep, series = _forward(cls, u, S, case["steps"] * max(1, reads),
                                               _par(_physics(case), case.get("scheme", "")),
                                               every=case["steps"] if reads else 0, level=case["ny"] // 2)
    out = dict(rho=rho, u=v, c=sum(cls[1:], cls[0]), deposit=float(sum(dep)))
    if reads:
        out["series"] = series
    if S is not None:
        out["S"] = S
    if len(cls) > 1:
        out["classes"] = cls
    return out
