"""The work that users of the porous lattice Boltzmann library have it do, as
cases that can be timed and compared: what a program has in hand (`prepare`),
one pass through the public entry points (`run`), what a pass cannot do without
(`work`) and the same results in 64 bits from plain torch (`exact`).

A case names a task and its sizes:

  flow       one porosity field: rest state, `steps` time steps, rho and u
             (a job of a parameter study; `Solver.run_jobs` chains such jobs)
  monitored  the same with rho, u and the convergence figures every `every` steps
  porosity   a porosity that varies in time: a new field every `every` steps
  batch      many uneven channels advanced together, rho and u of each
  gradient   outlet flux and its gradient with respect to the porosity

All sizes, relaxation times and drag laws come from the workloads of the
benchmark and the tests or lie between them.  Launch shapes are the autotuner's,
as a program that runs more than a few steps picks them.
"""
import math

import numpy as np
import torch

import paper_1406_6438_gb300 as V
from paper_1406_6438_gb300.adjoint import outlet_flux

D_P = 21.33                # particle diameter of the Ergun drag


def _flow(name, q, nx, ny, nz=1, walls=0, tau=0.6, steps=100, **more):
    return dict(name=name, task="flow", q=q, nx=nx, ny=ny, nz=nz, walls=walls, tau=tau,
                steps=steps, **more)


def listed():
    return [
        # the porous Poiseuille channel, one short run of a parameter study: the
        # whole state fits in a few SMs, so launches and latency count
        _flow("channel_128x64", 9, 128, 64, walls=2, tau=0.8, steps=2000, k_mode=2, K=4.096),
        # the validation case of the method: Couette flow between plates that lie
        # on nodes (non-equilibrium extrapolation), odd row count, low porosity
        _flow("couette_80x81", 9, 80, 81, walls=2, tau=0.8, steps=1000, k_mode=2, K=64.0,
              lo=0.1, hi=0.12, g=0.0, wall_kind=1, plate=0.00125),
        # a middle-sized channel (the gradient workload's grid, forward only):
        # the state stays in L2, a launch is as long as the work it starts
        _flow("channel_512x512", 9, 512, 512, walls=2, tau=0.8, steps=400),
        # ragged sizes and a moving upper wall (bounce-back), fixed K and F_eps
        _flow("moving_wall_1501x733", 9, 1501, 733, walls=2, tau=0.9, steps=150, k_mode=1,
              K=4.0, F_eps=0.3, plate=0.01),
        # the benchmark's plain step: 4096^2 periodic, far larger than L2
        _flow("periodic_4096", 9, 4096, 4096, steps=100),
        # a run that watches its own convergence
        dict(name="monitored_2048", task="monitored", q=9, nx=2048, ny=2048, nz=1, walls=2,
             tau=0.7, steps=60, every=10),
        # porosity varying in time (two-fluid coupling): a new field every 10 steps
        dict(name="porosity_1536x1000", task="porosity", q=9, nx=1536, ny=1000, nz=1, walls=0,
             tau=0.6, steps=60, every=10),
        # the porous duct in 3-D at the benchmark's size
        _flow("duct_256", 19, 256, 256, 256, walls=6, steps=50, lo=0.35, hi=0.95, g=2e-5),
        # a smaller duct of ragged sizes
        _flow("duct_150x110x90", 19, 150, 110, 90, walls=6, tau=0.8, steps=80, lo=0.35, hi=0.95,
              g=2e-5),
        # many small channels of a parameter study in one go
        dict(name="batch_256", task="batch", domains=256, nx_lo=64, nx_hi=1024, ny_lo=32,
             ny_hi=512, steps=40),
        # reverse mode: the gradient workload's channel, a short rollout
        dict(name="gradient_512x512", task="gradient", q=9, nx=512, ny=512, nz=1, walls=2,
             tau=0.8, steps=200, every=100),
        # reverse mode in 3-D
        dict(name="gradient_3d_96x64x48", task="gradient", q=19, nx=96, ny=64, nz=48, walls=6,
             tau=0.7, steps=40, every=20),
    ]


MOST_CELLS = 1 << 24       # the largest listed grid
MOST_UPDATES = 1.2e9       # cells x steps of a drawn case, at most


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _steps(rng, cells, lo, hi):
    """Steps of a drawn case, so that it stays below the largest listed ones."""
    return max(lo, min(_log_int(rng, lo, hi), int(MOST_UPDATES / cells)))


def draw(rng):
    kind = rng.choice(["flow2", "flow2", "flow2", "flow3", "flow3", "plates", "monitored",
                       "porosity", "batch", "gradient"])
    tau = round(rng.uniform(0.55, 1.0), 3)
    if kind == "batch":
        nx_hi, ny_hi = rng.randint(100, 1024), rng.randint(60, 512)
        return dict(task="batch", domains=rng.randint(16, 256), nx_lo=min(64, nx_hi), nx_hi=nx_hi,
                    ny_lo=32, ny_hi=ny_hi, steps=rng.randint(10, 40))
    if kind == "plates":
        nx, ny = rng.randint(60, 130), rng.randint(41, 90)
        return dict(task="flow", q=9, nx=nx, ny=ny, nz=1, walls=2, tau=tau,
                    steps=rng.randint(200, 1000), k_mode=2, K=round(rng.uniform(4.0, 64.0), 2),
                    lo=0.1, hi=0.12, g=0.0, wall_kind=1, plate=0.00125)
    if kind == "gradient":
        if rng.random() < 0.3:
            nx, ny, nz = rng.randint(20, 96), rng.randint(16, 64), rng.randint(12, 48)
            steps = rng.randint(10, 40)
            return dict(task="gradient", q=19, nx=nx, ny=ny, nz=nz, walls=6, tau=tau, steps=steps,
                        every=rng.randint(5, steps))
        nx, ny = _log_int(rng, 64, 512), _log_int(rng, 48, 512)
        steps = rng.randint(40, 200)
        return dict(task="gradient", q=9, nx=nx, ny=ny, nz=1, walls=rng.choice([0, 2]), tau=tau,
                    steps=steps, every=rng.randint(10, 100))
    if kind == "flow3":
        nx, ny, nz = (_log_int(rng, 24, 256) for _ in range(3))
        if rng.random() < 0.4:
            nx = max(32, nx // 32 * 32)
        return dict(task="flow", q=19, nx=nx, ny=ny, nz=nz, walls=rng.choice([0, 2, 4, 6, 6]),
                    tau=tau, steps=_steps(rng, 2 * nx * ny * nz, 20, 200), lo=0.35, hi=0.95, g=2e-5)
    nx, ny = _log_int(rng, 96, 4096), _log_int(rng, 64, 4096)
    if rng.random() < 0.3:
        nx = max(128, nx // 128 * 128)
    steps = _steps(rng, nx * ny, 20, 1000)
    if kind == "monitored":
        return dict(task="monitored", q=9, nx=nx, ny=ny, nz=1, walls=rng.choice([0, 2]), tau=tau,
                    steps=min(steps, 100), every=rng.choice([5, 10, 25]))
    if kind == "porosity":
        nx, ny = min(nx, 2000), min(ny, 2000)
        return dict(task="porosity", q=9, nx=nx, ny=ny, nz=1, walls=rng.choice([0, 2]), tau=tau,
                    steps=60, every=rng.choice([5, 10, 20]))
    case = dict(task="flow", q=9, nx=nx, ny=ny, nz=1, walls=rng.choice([0, 0, 2]), tau=tau,
                steps=steps)
    if case["walls"]:
        case.update(rng.choice([dict(), dict(k_mode=1, K=4.0, F_eps=0.3, plate=0.01),
                                dict(k_mode=2, K=4.0), dict(drag_mode=1)]))
    return case


# ------------------------------------------------------------------ inputs --

def _params(c, nx=None, ny=None, tau=None):
    """The library's parameters of one domain, floats rounded to float32 once."""
    r = lambda v: float(np.float32(v))  # noqa: E731
    return dict(q=c.get("q", 9), nx=nx or c["nx"], ny=ny or c["ny"], nz=c.get("nz", 1),
                wall_mask=c.get("walls", 2), tau=r(tau or c["tau"]),
                g=(r(c.get("g", 5e-5 if c.get("walls", 2) == 0 else 2e-5)), 0.0, 0.0),
                drag_mode=c.get("drag_mode", 2), k_mode=c.get("k_mode", 0), d_p=r(D_P),
                K=r(c.get("K", 1.0)), F_eps=r(c.get("F_eps", 0.0)),
                u_wall=(r(c.get("plate", 0.0)), 0.0, 0.0), wall_kind=c.get("wall_kind", 0))


def _noise(shape, lo, hi, gen, sigma=16.0):
    """Gaussian-smoothed periodic white noise mapped onto [lo, hi], float32."""
    spec = torch.fft.fftn(torch.randn(shape, generator=gen, dtype=torch.float64, device="cuda"))
    for ax, n in enumerate(shape):
        k = 2.0 * math.pi * torch.fft.fftfreq(n, dtype=torch.float64, device="cuda")
        spec *= torch.exp(-0.5 * (sigma * k) ** 2).view([n if a == ax else 1 for a in range(3)])
    s = torch.fft.ifftn(spec).real
    s = (s - s.min()) / (s.max() - s.min()).clamp_min(1e-300)
    return (lo + (hi - lo) * s).to(torch.float32)


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)


def _eps(c, seed):
    return _noise((c["nz"], c["ny"], c["nx"]), c.get("lo", 0.4), c.get("hi", 1.0), _gen(seed))


def _eps_series(c, seed):
    """A slowly varying field: the first one drifting towards another one."""
    a, b = _eps(c, seed), _eps(c, seed + 7919)
    n = -(-c["steps"] // c["every"])
    return [torch.lerp(a, b, 0.3 * k / n).contiguous() for k in range(n)]


def _domains(c, seed):
    """Sizes (the batch's own, the same for every seed), relaxation times and
    porosity fields (by seed) of a batch."""
    r = np.random.default_rng([c["domains"], c["nx_hi"], c["ny_hi"]])
    nxs = r.integers(c["nx_lo"], c["nx_hi"] + 1, c["domains"])
    nys = r.integers(c["ny_lo"], c["ny_hi"] + 1, c["domains"])
    taus = np.random.default_rng(seed).uniform(0.55, 1.0, c["domains"])
    gen = _gen(seed)
    return [(_params(dict(g=1e-5), int(x), int(y), t), _noise((1, int(y), int(x)), 0.4, 1.0, gen))
            for x, y, t in zip(nxs, nys, taus)]


def prepare(case, seed):
    task = case["task"]
    if task == "batch":
        doms = _domains(case, seed)
        b = V.Batch([p for p, _ in doms])
        for d, (_, e) in enumerate(doms):
            b.set_eps(d, e.view(-1))
        b.autotune()
        return dict(case=case, batch=b)
    p = _params(case)
    s = V.Solver(p)
    eps = _eps_series(case, seed) if task == "porosity" else [_eps(case, seed)]
    s.set_eps(eps[0].view(-1))
    s.autotune()
    rho = torch.empty(s.params.shape, dtype=torch.float32, device="cuda")
    u = torch.empty((s.params.dim,) + s.params.shape, dtype=torch.float32, device="cuda")
    return dict(case=case, solver=s, eps=eps, rho=rho, u=u)


def run(state):
    c = state["case"]
    n = c["steps"]
    if c["task"] == "batch":
        b = state["batch"]
        b.step(n)
        out = [b.moments(d) for d in range(b.n)]
        return (torch.cat([r.view(-1) for r, _ in out]), torch.cat([u.view(-1) for _, u in out]))
    s, eps = state["solver"], state["eps"]
    if c["task"] == "gradient":
        e = eps[0].requires_grad_(True)
        J = outlet_flux(e, s, n, c["every"])
        (g,) = torch.autograd.grad(J, e)
        return J.detach(), g
    s.set_eps_async(eps[0].view(-1))
    if c["task"] == "monitored":
        return s.step_monitored(n, c["every"])
    if c["task"] == "porosity":
        for k, e in enumerate(eps):
            if k:
                s.update_eps(e.view(-1))
            s.step(min(c["every"], n - k * c["every"]))
    else:
        s.step(n)
    return s.moments(state["rho"], state["u"])


# -------------------------------------------------------------------- work --

# floating-point operations of one cell update (moments, velocity, equilibrium,
# sources, relaxation; a multiply-add counts two), forward and transposed
FLOPS = {9: 200, 19: 420}
REVERSE_FLOPS = {9: 420, 19: 900}


def work(case):
    """Each input (porosity) read once, each result (rho, u, the flow state that
    the handle keeps) written once; the operations of all the steps."""
    if case["task"] == "batch":
        r = np.random.default_rng([case["domains"], case["nx_hi"], case["ny_hi"]])
        nxs = r.integers(case["nx_lo"], case["nx_hi"] + 1, case["domains"])
        nys = r.integers(case["ny_lo"], case["ny_hi"] + 1, case["domains"])
        n = int((nxs * nys).sum())
        # the state is the input of the pass here
        return dict(bytes=n * 4.0 * (2 * 9 + 1 + 3), flops=float(FLOPS[9]) * n * case["steps"])
    q = case["q"]
    n = case["nx"] * case["ny"] * case["nz"]
    updates = float(n) * case["steps"]
    if case["task"] == "gradient":
        # the flux is a number and the gradient one value per cell
        return dict(bytes=n * 8.0, flops=updates * (FLOPS[q] + REVERSE_FLOPS[q]))
    fields = -(-case["steps"] // case["every"]) if case["task"] == "porosity" else 1
    return dict(bytes=n * 4.0 * (fields + q + 3 + (q == 19)), flops=updates * FLOPS[q])


# ------------------------------------------------------- the same in 64 bits --

_E9 = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0),
       (-1, -1, 0), (1, -1, 0)]
_E19 = [(0, 0, 0)] + [tuple(s if a == ax else 0 for a in range(3)) for ax in range(3)
                      for s in (1, -1)]
_E19 += [tuple({a: s, b: t}.get(ax, 0) for ax in range(3)) for a, b in ((0, 1), (0, 2), (1, 2))
         for s, t in ((1, 1), (-1, -1), (1, -1), (-1, 1))]


class _Flow64:
    """The method in double precision: collide, then stream, on f_i [q, cells]."""

    def __init__(self, p):
        self.p = p
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        e = _E9 if p["q"] == 9 else _E19
        D = 2 if p["q"] == 9 else 3
        t64 = dict(dtype=torch.float64, device=dev)
        w = [(4 / 9, 1 / 9, 1 / 36) if D == 2 else (1 / 3, 1 / 18, 1 / 36)][0]
        self.w = torch.tensor([w[sum(map(abs, v))] for v in e], **t64).view(-1, 1)
        self.E = torch.tensor([v[:D] for v in e], **t64)
        self.g = torch.tensor(p["g"][:D], **t64).view(-1, 1)
        self.uw = torch.tensor(p["u_wall"][:D], **t64).view(-1, 1)
        nx, ny, nz = p["nx"], p["ny"], p["nz"]
        wy, wz = p["wall_mask"] >> 1 & 1, p["wall_mask"] >> 2 & 1
        n = nx * ny * nz
        cell = torch.arange(n, device=dev).view(nz, ny, nx)
        x, y, z = (torch.arange(k, device=dev) for k in (nx, ny, nz))
        plates = p["wall_kind"] == 1
        moving = any(p["u_wall"]) and not plates
        pull, ahead, self.gain = [], [], {}
        for i, (ex, ey, ez) in enumerate(e):
            opp = e.index((-ex, -ey, -ez))

            def at(sign):
                ys, zs = y + sign * ey, z + sign * ez
                out = torch.zeros((nz, ny, nx), dtype=torch.bool, device=dev)
                if wy:
                    out |= ((ys < 0) | (ys >= ny)).view(1, -1, 1)
                if wz:
                    out |= ((zs < 0) | (zs >= nz)).view(-1, 1, 1)
                xs = (x + sign * ex) % nx
                return out, cell[zs % nz][:, ys % ny][:, :, xs]
            past, src = at(-1)
            pull.append(torch.where(past, opp * n + cell, i * n + src).reshape(-1))
            past, dst = at(1)
            ahead.append(torch.where(past, cell, dst).reshape(-1))
            if moving and ey < 0:
                # bounced off the moving upper wall alone (not a z wall too)
                top = (y == ny - 1).view(1, -1, 1).expand(nz, ny, nx).clone()
                if wz and ez:
                    top &= ((z - ez >= 0) & (z - ez < nz)).view(-1, 1, 1)
                c = 6.0 * float(self.w[i]) * float((self.E[i].view(-1, 1) * self.uw).sum())
                self.gain[i] = (top.reshape(-1).nonzero().view(-1), c)
        self.pull = torch.stack(pull).view(-1)
        self.ahead = ahead
        self.shape = (nz, ny, nx)
        self.plate = None
        if plates:
            row = lambda k: cell[:, k].reshape(-1)  # noqa: E731
            zero = torch.zeros_like(self.uw)
            self.plate = [(row(0), row(1), zero), (row(ny - 1), row(ny - 2), self.uw)]

    def porosity(self, eps):
        """What depends on the porosity alone: eps, grad eps, drag coefficients."""
        p = self.p
        e = eps.reshape(-1)
        grad = 0
        for i in range(1, len(self.ahead)):
            grad = grad + 3.0 * self.w[i] * self.E[i].view(-1, 1) * e[self.ahead[i]]
        nu = (p["tau"] - 0.5) / 3.0
        if p["k_mode"] == 0:
            a = 150.0 * nu * (1 - e) ** 2 / (e * p["d_p"] ** 2)
            b = 1.75 * (1 - e) / p["d_p"]
        else:
            a = nu * e ** 2 / p["K"]
            F = p["F_eps"] if p["k_mode"] == 1 else 1.75 / torch.sqrt(150.0 * e ** 3)
            b = e ** 3 * F / math.sqrt(p["K"])
        on = (p["drag_mode"] > 0, p["drag_mode"] > 1)
        return e, grad, a * on[0], b * on[1]

    def macro(self, f, por):
        e, grad, al, be = por
        R = f.sum(0)
        rho = R / e
        Pc = rho * grad / 3.0
        m = self.E.T @ f + 0.5 * Pc + 0.5 * R * self.g
        m2 = (m * m).sum(0)
        mm = torch.where(m2 > 0, torch.sqrt(torch.where(m2 > 0, m2, 1.0)), 0.0)
        a = R + 0.5 * al
        u = 2.0 * m / (a + torch.sqrt(a * a + 2.0 * be * mm))
        u2 = (u * u).sum(0)
        un = torch.where(u2 > 0, torch.sqrt(torch.where(u2 > 0, u2, 1.0)), 0.0)
        return R, rho, u, Pc + R * self.g - (al + be * un) * u

    def feq(self, R, u):
        eu = self.E @ u
        return self.w * R * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * (u * u).sum(0)), eu

    def step(self, f, por):
        tau = self.p["tau"]
        R, _, u, Vs = self.macro(f, por)
        feq, eu = self.feq(R, u)
        S = (1.0 - 0.5 / tau) * self.w * (3.0 * (self.E @ Vs - (u * Vs).sum(0)) +
                                          9.0 * eu * (self.E @ Vs))
        fs = f - (f - feq) / tau + S
        if self.plate:
            for b, _, ub in self.plate:
                fs[:, b] = f[:, b] - (f[:, b] - self.feq(f[:, b].sum(0), ub)[0]) / tau
        fn = fs.reshape(-1)[self.pull].view(fs.shape)
        for i, (top, c) in self.gain.items():
            fn[i, top] = fn[i, top] + c * por[0][top]
        self.on_plates(fn, por)
        return fn

    def on_plates(self, f, por):
        """Plate nodes: equilibrium of the plate plus the neighbour's remainder."""
        for b, nb, ub in self.plate or ():
            R, rho, u, _ = self.macro(f[:, nb], [t[..., nb] for t in por])
            f[:, b] = self.feq(por[0][b] * rho, ub)[0] + f[:, nb] - self.feq(R, u)[0]

    def rest(self, por):
        f = self.w * por[0]
        self.on_plates(f, por)
        return f

    def moments(self, f, por):
        _, rho, u, _ = self.macro(f, por)
        return rho.view(self.shape), u.view((-1,) + self.shape)


def _exact_gradient(c, eps):
    from torch.utils.checkpoint import checkpoint
    m = _Flow64(_params(c))
    e = eps.double().requires_grad_(True)
    por = m.porosity(e)
    f = m.rest(por)
    for k in range(0, c["steps"], 10):
        def some(f, *por, n=min(10, c["steps"] - k)):
            for _ in range(n):
                f = m.step(f, por)
            return f
        f = checkpoint(some, f, *por, use_reentrant=False)
    R, _, u, _ = m.macro(f, por)
    J = (R * u[0]).view(m.shape)[:, :, -1].sum()
    return J.detach(), torch.autograd.grad(J, e)[0]


def exact(case, seed):
    if case["task"] == "gradient":
        return _exact_gradient(case, _eps(case, seed))
    with torch.no_grad():
        if case["task"] == "batch":
            rho, u = [], []
            for p, eps in _domains(case, seed):
                m = _Flow64(p)
                por = m.porosity(eps.double())
                f = m.rest(por)
                for _ in range(case["steps"]):
                    f = m.step(f, por)
                r, v = m.moments(f, por)
                rho.append(r.reshape(-1))
                u.append(v.reshape(-1))
            return torch.cat(rho), torch.cat(u)
        m = _Flow64(_params(case))
        fields = _eps_series(case, seed) if case["task"] == "porosity" else [_eps(case, seed)]
        por = m.porosity(fields[0].double())
        f = m.rest(por)
        every = case.get("every", case["steps"])
        last, stats = None, [0.0, 0.0, 0.0, 0.0]
        for k in range(case["steps"]):
            if case["task"] == "porosity" and k and k % every == 0:
                por = m.porosity(fields[k // every].double())
            if case["task"] == "monitored" and ((k + 1) % every == 0 or k + 1 == case["steps"]):
                # moments of the state that this step reads, as the library reports them
                rho, u = m.moments(f, por)
                du = u if last is None else u - last
                size = lambda v: float((v * v).sum(0).max().sqrt())  # noqa: E731
                stats = [max(stats[0], size(du)), max(stats[1], size(u)), 0.0, stats[3] + 1.0]
                last = u
            f = m.step(f, por)
        if case["task"] == "monitored":
            return rho, u, torch.tensor(stats, dtype=torch.float64)
        return m.moments(f, por)
