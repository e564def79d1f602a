"""Measured workloads of the framework, through its public entry points.

Three kinds of case, each what a user's program does between two looks at a run:

* ``steps``: ``steps`` fused time steps of one cavity (``lbm.Cavity.step``), then the wall Nusselt numbers and the
  state read back into pinned host memory (``nusselt``, ``get_state``); every pass goes on from where the last ended;
* ``batch``: the same for a sweep of cavities stepped together (``lbm.Batch``, plan chosen by ``tune``);
* ``adjoint``: the gradient of the hot-wall Nusselt number (``autograd.hot_wall_nusselt`` and its ``backward``).

Runs start from a smooth convective flow (a few vortices and a stratified temperature drawn from the seed), as a run
restarted from a stored state does.  What leaves the library as a Python float is returned in the precision of the run's
storage; the relaxation times beside 16-bit populations, which follow from them, in 16 bits too.
"""
import math

import numpy as np
import torch

from paper_2011_15073_gb300 import autograd, inputs, lbm

MA, PR, POROSITY = 0.1, 6.2, 0.6
POPS = {"f64": torch.float64, "f32": torch.float32, "f32d": torch.float32, "f16s": torch.float16,
        "f16d": torch.float16, "bf16s": torch.bfloat16, "bf16d": torch.bfloat16}
FLOPS = 330   # of one node and step: both transforms and their inverses, both collisions, the viscosity and the drag


def _case(name, nx, ny, steps, prec, n=0.6, Da=1e-2, Ra=1e5, kind="steps", **more):
    c = dict(name=name, kind=kind, nx=nx, ny=ny, steps=steps, prec=prec, n=n, Da=Da, Ra=Ra, porous_model=1, clamp_mode=1,
             layout=0, tau_iters=0, field=False, ncases=1, ckpt_every=0)
    c.update(more)
    return c


def listed():
    return [
        # the plain method, as a first run or a test does it: 64 x 64, Newtonian, FP64; launches and latency count
        _case("plain 64 f64", 64, 64, 200, "f64", n=1.0, Da=1e-1, Ra=1e3, clamp_mode=0),
        # the paper's grid, drag and literal law, FP64 as its tables are reproduced
        _case("paper 160 f64", 160, 160, 200, "f64", Da=1e-3, porous_model=0, clamp_mode=0),
        # one parameter study's cavity between two convergence checks
        _case("study 256 f32d", 256, 256, 1000, "f32d", n=0.8, Ra=1e4),
        # a cavity that is not square and of odd sizes, with a measured (per-node) permeability
        _case("darcy 701x499 f32", 701, 499, 400, "f32", n=0.8, Ra=1e4, field=True),
        # an ordinary grid of a resolved run
        _case("resolved 1024 f32d", 1024, 1024, 400, "f32d"),
        # FP64 reference on a resolved, ragged grid
        _case("reference 1000x1100 f64", 1000, 1100, 25, "f64", Da=1e-2),
        # node-local implicit relaxation time, which stores no tau
        _case("implicit 2048 f32", 2048, 2048, 300, "f32", tau_iters=2),
        # half the memory: the in-place layout
        _case("in place 2048 f32d", 2048, 2048, 300, "f32d", layout=1),
        # the benchmark's cavity, the largest: FP32 deviations, and FP16 with stochastic rounding
        _case("benchmark 4096 f32d", 4096, 4096, 500, "f32d", Da=1e-3),
        _case("benchmark 4096 f16s", 4096, 4096, 500, "f16s", Da=1e-3),
        # the paper's (n, Da, Ra) sweep as one batch of cavities of 128^2 to 512^2, without its first, which amplifies
        # any rounding (nearly at rest, on the clamp of the law)
        _case("sweep 26 f32d", 0, 0, 100, "f32d", kind="batch", ncases=26, first=1),
        # design: gradient with respect to a permeability field, n and Ra
        _case("adjoint 256 f32", 256, 256, 400, "f32", n=0.8, Ra=1e4, kind="adjoint", field=True, ckpt_every=100),
    ]


def draw(rng):
    kind = rng.choice(["steps"] * 8 + ["batch", "adjoint"])
    Da = 10.0 ** rng.uniform(-3, -1)
    if kind == "batch":
        k = rng.randint(3, 26)
        return _case("", 0, 0, rng.randint(40, 100), "f32d", kind=kind, ncases=k,
                     first=rng.randint(1, 27 - k))
    if kind == "adjoint":
        nx, ny = rng.randint(96, 288), rng.randint(96, 288)
        steps = rng.randint(150, 400)
        return _case("", nx, ny, steps, "f32", n=rng.choice([0.8, 1.0]), Ra=1e4, kind=kind, field=True,
                     ckpt_every=rng.randint(40, 150))
    prec = rng.choice(["f32d", "f32d", "f32", "f64", "f16s"])
    nx = round(math.exp(rng.uniform(math.log(48), math.log(1400 if prec == "f64" else 4096))))
    ny = min(4096, max(48, round(nx * math.exp(rng.uniform(-0.7, 0.7)))))
    if prec == "f16s":   # the 16-bit storage is for large grids, and was studied at these Darcy numbers
        prec, Da = ("f16s", 10.0 ** rng.uniform(-2, -1)) if nx >= 600 else ("f32d", Da)
    if rng.random() < 0.4:
        nx, ny = nx // 16 * 16, ny // 16 * 16
    most = 3e7 if prec == "f64" else 2e9
    steps = int(min(1000, max(10, most / (nx * ny))))
    # the groups of the studies: thickening fluids and small Rayleigh numbers on the small grids, whose tau they keep moderate
    n = rng.choice([0.6, 0.8, 1.0, 1.4] if nx < 300 else [0.6, 0.8, 1.0])
    Ra = 10.0 ** (rng.uniform(3, 4) if nx < 128 else rng.uniform(4, 5) if nx < 600 else 5)
    return _case("", nx, ny, steps, prec, n=n, Da=Da, Ra=Ra, field=rng.random() < 0.2,
                 layout=1 if prec == "f32d" and rng.random() < 0.25 else 0,
                 tau_iters=2 if prec != "f64" and rng.random() < 0.2 else 0)


# ------------------------------------------------------------------ inputs
def _cavities(case):
    """(nx, ny, n, Da, Ra) of each cavity."""
    if case["kind"] == "batch":
        k = case.get("first", 0)
        return [(c["N"], c["N"], c["n"], c["Da"], c["Ra"]) for c in inputs.sweep_cases()[k:k + case["ncases"]]]
    return [(case["nx"], case["ny"], case["n"], case["Da"], case["Ra"])]


def _opts(case):
    return dict(prec=case["prec"], clamp_mode=case["clamp_mode"], porous_model=case["porous_model"],
                layout=case["layout"], tau_iters=case["tau_iters"])


def _rest(i, heat):
    """Rest value of population i: the weight, times the mean temperature for the heat."""
    if heat:
        return (2.0 if i == 0 else 1.0) / 12.0
    return 4.0 / 9.0 if i == 0 else (1.0 / 9.0 if i < 5 else 1.0 / 36.0)


E = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
OPP = [0, 3, 4, 1, 2, 7, 8, 5, 6]
DEV = "cuda"


def _flow(nx, ny, seed):
    """A smooth convective flow: (u_x, u_y, T) in lattice units, FP64 on the device."""
    r = np.random.default_rng(seed)
    X = ((torch.arange(nx, device=DEV, dtype=torch.float64) + 0.5) / nx)[None, :]
    Y = ((torch.arange(ny, device=DEV, dtype=torch.float64) + 0.5) / ny)[:, None]
    ux, uy = torch.zeros(ny, nx, device=DEV, dtype=torch.float64), torch.zeros(ny, nx, device=DEV, dtype=torch.float64)
    T = (1.0 - X).expand(ny, nx).clone()
    most = max(1, min(12, min(nx, ny) // 24))
    for m in range(1, most + 1):
        a, b = r.uniform(-1, 1) * 0.02 / m, r.uniform(-1, 1) * 0.15 / m
        l = int(r.integers(1, most + 1))
        # stream function a sin^2(m pi X) sin^2(l pi Y) / (pi m): at rest on the walls
        sx, sy = torch.sin(m * math.pi * X), torch.sin(l * math.pi * Y)
        ux += a * l / m * sx * sx * torch.sin(2 * l * math.pi * Y)
        uy -= a * torch.sin(2 * m * math.pi * X) * sy * sy
        T += b * sx * torch.cos(l * math.pi * Y)
    return ux, uy, T


def _populations(flow, eps, i, heat):
    ux, uy, T = flow
    eu = E[i][0] * ux + E[i][1] * uy
    if heat:
        return T * (1 / 3 if i == 0 else 1 / 6) + (T * eu * 0.5 if i else 0.0)
    return _rest(i, False) * (1.0 + 3.0 * eu + (4.5 * eu * eu - 1.5 * (ux * ux + uy * uy)) / eps)


def _start(case, nx, ny, seed, prec, tau0):
    """The native state (as lbm_state_bytes describes it) of that flow at equilibrium, as bytes in pinned memory."""
    n, dt = nx * ny, POPS[prec]
    tt = torch.float64 if prec == "f64" else torch.float32
    es = torch.empty((), dtype=dt).element_size()
    dev = torch.empty(14 * n * es + n * torch.empty((), dtype=tt).element_size(), dtype=torch.uint8, device=DEV)
    flow = _flow(nx, ny, seed)
    planes = dev[:14 * n * es].view(dt).view(14, ny, nx)
    for q in range(14):
        heat, i = q >= 9, q % 9
        v = _populations(flow, POROSITY if case["porous_model"] else 1.0, i, heat)
        if prec not in ("f64", "f32"):
            v = (v - _rest(i, heat)) * (32768.0 if prec == "f16s" else 1.0)
        planes[q] = v.to(dt)
    dev[14 * n * es:].view(tt).fill_(tau0)
    host = torch.empty(dev.numel(), dtype=torch.uint8, pin_memory=True)
    host.copy_(dev)
    return host


def _darcy(nx, ny, seed):
    return inputs.darcy_field(seed, nx, ny)


def prepare(case, seed):
    if case["kind"] == "adjoint":
        return dict(case=case, Da=torch.from_numpy(_darcy(case["nx"], case["ny"], seed)).to(DEV, torch.float32))
    s = dict(case=case, host=[])
    if case["kind"] == "batch":
        s["run"] = lbm.Batch([dict(nx=a, ny=b, n=n, Da=Da, Ra=Ra, Pr=PR, porosity=POROSITY) for a, b, n, Da, Ra in _cavities(case)],
                             **_opts(case))
        s["ctx"] = [s["run"].case_ctx(i) for i in range(case["ncases"])]
    else:
        nx, ny, n, Da, Ra = _cavities(case)[0]
        s["run"] = lbm.Cavity(nx, ny, n, Da, Ra, PR, POROSITY, **_opts(case))
        if case["field"]:
            s["run"].set_darcy_field(_darcy(nx, ny, seed))
        s["ctx"] = [s["run"].ctx]
    for k, (nx, ny, *_) in enumerate(_cavities(case)):
        host = _start(case, nx, ny, seed * 32 + k, case["prec"], lbm.get_lattice(s["ctx"][k]).tau0)
        lbm.set_state(s["ctx"][k], host)
        s["host"].append(host)   # the state is read back into the same buffer
    if case["kind"] == "batch":
        s["run"].tune(20)
    return s


# -------------------------------------------------------------------- run
def _out(case, host, nx, ny):
    dt = POPS[case["prec"]]
    es = torch.empty((), dtype=dt).element_size()
    at = 14 * nx * ny * es
    out = {"populations": host[:at].view(dt).view(14, ny, nx)}
    if not case["tau_iters"]:   # with an implicit tau none is stored
        tau = host[at:].view(torch.float64 if es == 8 else torch.float32).view(ny, nx)
        out["tau"] = tau.to(dt) if es == 2 else tau
    return out


def run(state):
    case = state["case"]
    if case["kind"] == "adjoint":
        Da = state["Da"].clone().requires_grad_()
        n = torch.tensor(case["n"], dtype=torch.float32, requires_grad=True)
        Ra = torch.tensor(case["Ra"], dtype=torch.float32, requires_grad=True)
        J = autograd.hot_wall_nusselt(Da, n, Ra, Pr=PR, porosity=POROSITY, steps=case["steps"], ckpt_every=case["ckpt_every"],
                                      prec=case["prec"], clamp_mode=case["clamp_mode"])
        J.backward()
        return {"J": J.detach().float(), "dDa": Da.grad, "dn": n.grad, "dRa": Ra.grad}
    r = state["run"]
    r.step(case["steps"])
    hot, cold = r.nusselt()[:2]
    for ctx, host in zip(state["ctx"], state["host"]):
        lbm.get_state(ctx, host)
    nu = np.stack([np.atleast_1d(hot), np.atleast_1d(cold)]).astype(np.float64 if case["prec"] == "f64" else np.float32)
    return {"nu": nu, "states": [_out(case, host, c[0], c[1]) for host, c in zip(state["host"], _cavities(case))]}


def work(case):
    nodes = sum(c[0] * c[1] for c in _cavities(case))
    es = torch.empty((), dtype=POPS[case["prec"]]).element_size()
    state = 14 * es + (0 if case["tau_iters"] else (8 if es == 8 else 4))
    if case["kind"] == "adjoint":   # a forward pass, its recomputation and the reverse; the field read, its gradient written
        return {"bytes": nodes * 8.0, "flops": nodes * case["steps"] * 4.0 * FLOPS}
    return {"bytes": nodes * (2.0 * state + (es if case["field"] else 0)), "flops": nodes * case["steps"] * float(FLOPS)}


# ------------------------------------------------------------------ exact
# The scheme in plain FP64 torch: pull streaming with half-way walls, the D2Q9 multiple-relaxation-time collision with the
# porous force and the modified power law, the D2Q5 one for the heat, in moment space.
M9 = [[1] * 9, [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1], [0, 1, 0, -1, 0, 1, -1, -1, 1],
      [0, -2, 0, 2, 0, 1, -1, -1, 1], [0, 0, 1, 0, -1, 1, 1, -1, -1], [0, 0, -2, 0, 2, 1, 1, -1, -1],
      [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1]]
N5 = [[1] * 5, [0, 1, 0, -1, 0], [0, 0, 1, 0, -1], [-4, 1, 1, 1, 1], [0, 1, -1, 1, -1]]


class _Exact:
    def __init__(self, case, nx, ny, n, Da, Ra):
        f = lambda v: torch.as_tensor(v, device=DEV, dtype=torch.float64)   # noqa: E731
        self.nx, self.ny, self.clamp, self.iters = nx, ny, case["clamp_mode"], case["tau_iters"]
        n, Ra = f(n), f(Ra)
        U = MA / math.sqrt(3.0)
        self.n, self.nu_ref = n, PR / Ra ** ((2.0 - n) / 2.0) * U * nx
        self.scale, self.K = nx / U, f(Da) * nx * nx
        self.eps = POROSITY if case["porous_model"] else 1.0
        self.Fe = 1.75 / math.sqrt(150.0 * POROSITY ** 3) if case["porous_model"] else 0.0
        self.gbeta, self.wT = PR * U * U / nx, 1.0 / (3.0 * U * nx / torch.sqrt(Ra) + 0.5)
        self.tau0 = 3.0 * self.nu_ref * (1.0 if self.clamp == 0 else 0.01 ** (n - 1.0)) + 0.5
        self.M, self.N = f(M9), f(N5)
        self.Mi, self.Ni = torch.linalg.inv(self.M), torch.linalg.inv(self.N)

    def pull(self, F, heat):
        ny, nx = self.ny, self.nx
        out = [F[0]]
        for i in range(1, 5 if heat else 9):
            (ex, ey), back = E[i], F[OPP[i]]
            to = (slice(max(ey, 0), ny + min(ey, 0)), slice(max(ex, 0), nx + min(ex, 0)))
            of = (slice(max(-ey, 0), ny + min(-ey, 0)), slice(max(-ex, 0), nx + min(-ex, 0)))
            v = (1.0 / 3.0 if ex > 0 else 0.0) - back if heat and ex else back.clone()   # hot wall T = 1 on the left, cold T = 0
            v[to] = F[i][of]
            out.append(v)
        return torch.stack(out)

    def velocity(self, v, vmag, nu):
        c0 = 0.5 + self.eps * nu / (4.0 * self.K)
        den = c0 + torch.sqrt(c0 * c0 + self.eps * self.Fe / (2.0 * torch.sqrt(self.K)) * vmag)
        return v[0] / den, v[1] / den, vmag / den

    def law(self, gs):
        if self.clamp:
            return gs.clamp(0.01, 1e6) ** (self.n - 1.0)
        D = gs.clamp(0.01, 1e6) ** (self.n - 1.0)
        return torch.where(gs < 0.01, torch.ones_like(D), D)

    def strain(self, m, rho, ux, uy, tau):
        u2 = ux * ux + uy * uy
        A = 1.4 / 6.0 * (m[1] + 2.0 * rho - 3.0 * rho * u2 / self.eps)
        B = 0.5 / tau * (m[7] - rho * (ux * ux - uy * uy) / self.eps)
        C = (m[8] - rho * ux * uy / self.eps) / tau
        return A, B, C

    def step(self, F, G, tau):
        f, g = self.pull(F, False), self.pull(G, True)
        m, h = torch.tensordot(self.M, f, 1), torch.tensordot(self.N, g, 1)
        rho, T, eps = m[0], h[0], self.eps
        Gy = self.gbeta * (T - 0.5)
        v = (m[3] / rho, m[5] / rho + 0.5 * eps * Gy)
        v2 = v[0] * v[0] + v[1] * v[1]
        vmag = torch.where(v2 > 0, v2, torch.ones_like(v2)).sqrt() * (v2 > 0)
        if self.iters:
            tau = self.tau0
            for _ in range(self.iters):
                ux, uy, _m = self.velocity(v, vmag, (tau - 0.5) / 3.0)
                A, B, C = self.strain(m, rho, ux, uy, tau)
                s = A * A + B * B + C * C
                gs = 3.0 / rho * torch.sqrt(s) * self.scale
                phi = 3.0 * self.nu_ref * self.law(gs) + 0.5
                J = 1.0 + (self.n - 1.0) * (B * B + C * C) / s * (phi - 0.5) / phi
                tau = torch.where((gs > 0.01) & (gs < 1e6), tau * (phi / tau) ** (1.0 / J), phi)
        nu = (tau - 0.5) / 3.0
        ux, uy, umag = self.velocity(v, vmag, nu)
        drag = -eps * nu / self.K - eps * self.Fe / torch.sqrt(self.K) * umag
        Fx, Fy = drag * ux, drag * uy + eps * Gy
        A, B, C = self.strain(m, rho, ux, uy, tau)
        s = A * A + B * B + C * C
        new = 3.0 * self.nu_ref * self.law(3.0 / rho * torch.where(s > 0, s, torch.ones_like(s)).sqrt() * (s > 0) * self.scale) + 0.5
        w, re, uF = 1.0 / new, rho / eps, ux * Fx + uy * Fy
        u2 = 3.0 * re * (ux * ux + uy * uy)
        post = [rho,
                m[1] - 1.4 * (m[1] + 2.0 * rho - u2) + 0.3 * 6.0 * re * uF,
                m[2] - 1.4 * (m[2] - rho + u2) - 0.3 * 6.0 * re * uF,
                rho * (ux + 0.5 * Fx), m[4] - 1.2 * (m[4] + rho * ux) - 0.4 * rho * Fx,
                rho * (uy + 0.5 * Fy), m[6] - 1.2 * (m[6] + rho * uy) - 0.4 * rho * Fy,
                m[7] - w * (m[7] - re * (ux * ux - uy * uy)) + (1.0 - 0.5 * w) * 2.0 * re * (ux * Fx - uy * Fy),
                m[8] - w * (m[8] - re * ux * uy) + (1.0 - 0.5 * w) * re * (ux * Fy + uy * Fx)]
        heat = [T, h[1] - self.wT * (h[1] - T * ux), h[2] - self.wT * (h[2] - T * uy), h[3] - 1.5 * (h[3] + 2.0 / 3.0 * T),
                h[4] - 1.5 * h[4]]
        return torch.tensordot(self.Mi, torch.stack(post), 1), torch.tensordot(self.Ni, torch.stack(heat), 1), new

    def nusselt(self, G):
        T = self.pull(G, True).sum(0)
        return (-self.nx * (9.0 * T[:, 0] - T[:, 1] - 8.0) / 3.0).mean(), (self.nx * (9.0 * T[:, -1] - T[:, -2]) / 3.0).mean()


def _exact_gradient(case, seed):
    from torch.utils.checkpoint import checkpoint
    nx, ny = case["nx"], case["ny"]
    leaf = lambda v: torch.as_tensor(v, device=DEV).to(torch.float32).double().requires_grad_()   # noqa: E731
    Da, n, Ra = leaf(_darcy(nx, ny, seed)), leaf(case["n"]), leaf(case["Ra"])
    x = _Exact(case, nx, ny, n, Da, Ra)
    zero = torch.zeros(ny, nx, device=DEV, dtype=torch.float64)
    F, G = torch.stack([zero + _rest(i, False) for i in range(9)]), torch.stack([zero + _rest(i, True) for i in range(5)])
    tau = zero + x.tau0

    def some(F, G, tau, k):
        for _ in range(k):
            F, G, tau = x.step(F, G, tau)
        return F, G, tau

    left = case["steps"]
    while left:
        k = min(left, 20)
        F, G, tau = checkpoint(some, F, G, tau, k, use_reentrant=False)
        left -= k
    J = x.nusselt(G)[0]
    J.backward()
    return {"J": J.detach(), "dDa": Da.grad, "dn": n.grad, "dRa": Ra.grad}


def exact(case, seed):
    if case["kind"] == "adjoint":
        return _exact_gradient(case, seed)
    got, nus = [], []
    for k, (nx, ny, n, Da, Ra) in enumerate(_cavities(case)):
        prec = case["prec"]
        x = _Exact(case, nx, ny, n, torch.as_tensor(_darcy(nx, ny, seed), device=DEV) if case["field"] else Da, Ra)
        at = 14 * nx * ny * torch.empty((), dtype=POPS[prec]).element_size()
        host = _start(case, nx, ny, seed * 32 + k, prec, float(x.tau0))
        P = host[:at].view(POPS[prec]).view(14, ny, nx).to(DEV).double()
        tau = host[at:].view(torch.float64 if prec == "f64" else torch.float32).view(ny, nx).to(DEV).double()
        rest = torch.tensor([_rest(q % 9, q >= 9) for q in range(14)], device=DEV, dtype=torch.float64)[:, None, None]
        by = 32768.0 if prec == "f16s" else 1.0
        if prec not in ("f64", "f32"):
            P = P / by + rest
        F, G = P[:9], P[9:]
        for _ in range(case["steps"]):
            F, G, tau = x.step(F, G, tau)
        P = torch.cat([F, G])
        if prec not in ("f64", "f32"):
            P = (P - rest) * by
        out = {"populations": P.cpu()}
        nus.append([float(v) for v in x.nusselt(G)])
        if not case["tau_iters"]:
            out["tau"] = tau.cpu()
        got.append(out)
    return {"nu": np.array(nus).T.copy(), "states": got}
