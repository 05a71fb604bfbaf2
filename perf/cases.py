"""What is measured: whole calls and single stages of the open-cavity EnVar library, through its Python binding.

A case is one call (or the few calls that belong together) of a user's program on a handle it keeps: an EnVar,
Gauss-Newton or adjoint gradient iteration, one trial run of a line search, an uneven batch, the eigenvector
ensemble, the H^1 smoothing.  Horizons are short (a few time steps per run instead of thousands): the cost of a
run is its number of steps times the cost of a step.

`exact` restates the discretisation in 64 bits with torch: MAC grid, central advection and diffusion, AB2,
incremental projection with a direct pressure solve, window costs, EnVar gradient.  It shares no code with the library.
"""
import math

import numpy as np
import torch

import paper_2605_23812_gb300 as pkg

CAVITY = (-1.2, 2.5, -1.0, 1.0)
PAPER = (-1.2, 2.5, -1.0, 0.5)
REGION = (-0.5, 1.0, -0.2, 0.3)
SLIP_SPAN = (-0.4, 1.75)
EPS = 1e-2
# pressure-solve parameters: the library's defaults with a higher refinement cap (small grids, and grids whose coarsest
# multigrid level stays large), and what the tuner picks on the larger grids
DEFAULT = {"max_outer": 40}
TUNED = {"max_outer": 10, "max_inner": 2, "nu_pre": 3, "nu_post": 3, "coarse_sweeps": 1, "inner_rtol": 1e-3, "nu_coarse": 2}


def listed():
    def run(name, call, prec, cost, nx, ny, re, n, steps, solver="tuned", **kw):
        return dict({"name": name, "kind": "run", "call": call, "prec": prec, "cost": cost, "nx": nx, "ny": ny, "re": re,
                     "n": n, "steps": steps, "window": steps // 2, "solver": solver, "paper": False}, **kw)

    return [
        # the smallest useful ensemble: a first look at a coarse grid, a test; latency and launches count
        run("mixed_64x32_n2", "step", "mixed", "domain", 64, 32, 1000.0, 2, 20, "default"),
        # the plain method's configuration: one FP64 member at a time
        run("plain_fp64_128x64_n8", "step", "plain", "domain", 128, 64, 1000.0, 8, 10, "default"),
        # the FP64 ensemble that a mixed run is judged against
        run("fp64_256x128_n16", "step", "fp64", "domain", 256, 128, 4000.0, 16, 10),
        # a Gauss-Newton iteration on the sensor cost
        run("gn_256x128_n32", "gn", "mixed", "sensors", 256, 128, 4000.0, 32, 25),
        # the benchmark's EnVar iteration: quasi-periodic configuration, 33 runs
        run("step_512x256_n32", "step", "mixed", "domain", 512, 256, 7500.0, 32, 30),
        # the paper's own flow: its box, free-slip segments, forcing in y, sensor cost
        run("paper_592x240_n16", "step", "mixed", "sensors", 592, 240, 6250.0, 16, 20, "default", paper=True),
        # the chaotic configuration: the largest grid, 65 runs
        run("chaotic_1024x512_n64", "step", "mixed", "domain", 1024, 512, 15000.0, 64, 10),
        # one run of one member: a trial of the line searches (L-BFGS, adjoint loop)
        {"name": "trial_512x256", "kind": "trial", "prec": "mixed", "nx": 512, "ny": 256, "re": 7500.0, "steps": 20,
         "window": 10, "solver": "tuned"},
        # the uneven batch: three grids, horizons 1 : 2 : 4
        {"name": "batch_96", "kind": "batch", "prec": "mixed", "grids": "256x128x31,512x256x47,1024x512x15", "steps": 5},
        # the reference gradient: discrete adjoint with binomial checkpoints (fewer than the steps)
        {"name": "adjoint_128x64", "kind": "adjoint", "nx": 128, "ny": 64, "re": 1000.0, "steps": 24, "window": 12,
         "snapshots": 8, "solver": "tuned"},
        # the eigenvector ensemble, made once per control problem
        {"name": "eigen_256x128_n32", "kind": "eigen", "nx": 256, "ny": 128, "n": 32},
        # the adjoint loop's gradient regularisation
        {"name": "h1_512x256", "kind": "h1", "nx": 512, "ny": 256},
    ]


def _log(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def _grid(rng, lo, hi):
    """nx, ny: multiples of 16 (odd multiples among them), about two to one as the box is, cells from lo to hi."""
    cells = _log(rng, lo, hi)
    nx = max(32, 16 * round(math.sqrt(cells * 2.0 * _log(rng, 0.8, 1.25)) / 16))
    return nx, max(16, 16 * round(cells / nx / 16))


def _solver(nx, ny, small="tuned"):
    """The tuner's choice needs a small coarsest level (it sweeps there once); small: what a small grid's handle uses."""
    a, b = nx, ny
    while a % 2 == 0 and b % 2 == 0 and a >= 8 and b >= 4:
        a, b = a // 2, b // 2
    return "default" if a * b > 16 else small if nx * ny < 65536 else "tuned"


def draw(rng):
    """One more case: ensembles mostly, over grid, ensemble size, precision, cost and horizon; the single stages at times."""
    kind = rng.choice(["mixed", "mixed", "mixed", "mixed", "fp64", "plain", "trial", "batch", "adjoint", "eigen", "h1"])
    re = round(_log(rng, 300.0, 15000.0))
    if kind in ("mixed", "fp64", "plain"):
        nx, ny = _grid(rng, 32 * 16, {"mixed": 1024 * 512, "fp64": 256 * 128, "plain": 128 * 64}[kind])
        most = {"mixed": 65 * 1024 * 512, "fp64": 17 * 256 * 128, "plain": 9 * 128 * 64}[kind]
        n = max(2, min(64 if kind != "plain" else 8, round(_log(rng, 2, 66)), most // (nx * ny) - 1))
        steps = max(4, min(40, round(_log(rng, 5, 42)), 10 * most // (nx * ny * (n + 1))))
        cost = rng.choice(["domain", "domain", "sensors"])
        return {"kind": "run", "call": "gn" if cost == "sensors" and rng.random() < 0.5 else "step", "prec": kind, "cost": cost,
                "nx": nx, "ny": ny, "re": float(re), "n": n, "steps": steps, "window": max(2, steps // rng.choice([1, 2, 3])),
                "solver": _solver(nx, ny, rng.choice(["tuned", "default"])), "paper": rng.random() < 0.2}
    if kind == "trial":
        nx, ny = _grid(rng, 64 * 32, 1024 * 512)
        steps = rng.randrange(8, 25)
        return {"kind": "trial", "prec": "mixed", "nx": nx, "ny": ny, "re": float(re), "steps": steps, "window": steps // 2, "solver": _solver(nx, ny, rng.choice(["tuned", "default"]))}
    if kind == "batch":
        a, b = _grid(rng, 64 * 32, 256 * 128), _grid(rng, 128 * 64, 512 * 256)
        return {"kind": "batch", "prec": "mixed", "grids": "%dx%dx%d,%dx%dx%d" % (*a, rng.randrange(3, 32), *b, rng.randrange(3, 32)), "steps": rng.randrange(4, 11)}
    if kind == "adjoint":
        nx, ny = _grid(rng, 32 * 16, 160 * 80)
        steps = rng.randrange(8, 33)
        return {"kind": "adjoint", "nx": nx, "ny": ny, "re": float(re), "steps": steps, "window": max(2, steps // 2), "snapshots": rng.randrange(3, 12), "solver": _solver(nx, ny, rng.choice(["tuned", "default"]))}
    if kind == "eigen":
        nx, ny = _grid(rng, 96 * 48, 256 * 128)
        return {"kind": "eigen", "nx": nx, "ny": ny, "n": rng.randrange(4, 33)}
    nx, ny = _grid(rng, 64 * 32, 512 * 256)
    return {"kind": "h1", "nx": nx, "ny": ny}


# ---------------------------------------------------------------------------------------------- inputs from the seed
def _axes(nx, ny, box):
    x0, x1, y0, y1 = box
    dx, dy = (x1 - x0) / nx, (y1 - y0) / ny
    return dx, dy, x0 + (np.arange(nx) + 0.5) * dx, y0 + (np.arange(ny) + 0.5) * dy


def _control(nx, ny, box):
    """Control rectangle (first column, row, columns, rows) and the mask of its fluid cells."""
    _, _, xc, yc = _axes(nx, ny, box)
    i = np.flatnonzero((xc >= REGION[0]) & (xc <= REGION[1]))
    j = np.flatnonzero((yc >= REGION[2]) & (yc <= REGION[3]))
    fluid = (yc[j][:, None] > 0) | ((xc[i] > 0) & (xc[i] < 1))[None, :]
    return i[0], j[0], len(i), len(j), fluid


def _flow(nx, ny, box, delta, seed):
    """A developed-like state: the inflow profile above the lip, a shear-layer wave and a cavity vortex from a
    streamfunction (divergence-free), and 1e-3 noise on every face."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kw = {"dtype": torch.float64, "device": "cuda"}
    dx, dy, _, yc = _axes(nx, ny, box)
    x = (box[0] + torch.arange(nx + 1, **kw) * dx)[None, :]
    y = (box[2] + torch.arange(ny + 1, **kw) * dy)[:, None]
    a = torch.rand(6, generator=gen, **kw)
    inside = ((x > 0) & (x < 1) & (y < 0)) | (y > 0)
    psi = (0.01 + 0.01 * a[0]) * torch.sin((5 + 4 * a[1]) * x + 6.28 * a[2]) * torch.exp(-((y - 0.15) / 0.1) ** 2) * (y > 0)
    psi = psi + (0.02 + 0.02 * a[3]) * (torch.sin(math.pi * x) * torch.sin(math.pi * y)) ** 2 * inside * (y < 0)
    prof = torch.tensor([math.erf(v / delta) if v > 0 else 0.0 for v in yc], **kw)
    u = prof[:, None] + (psi[1:] - psi[:-1]) / dy + 1e-3 * torch.randn(ny, nx + 1, generator=gen, **kw)
    v = -(psi[:, 1:] - psi[:, :-1]) / dx + 1e-3 * torch.randn(ny + 1, nx, generator=gen, **kw)
    return u, v


def _fields(nx, ny, box, count, y_only, seed):
    """Smooth Gaussian random forcing fields on the control cells, one column each: (n_ctrl, count)."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kw = {"dtype": torch.float64, "device": "cuda"}
    dx, dy, _, _ = _axes(nx, ny, box)
    _, _, nrx, nry, fluid = _control(nx, ny, box)

    def factor(m, h):
        d = (torch.arange(m, **kw)[:, None] - torch.arange(-8, m + 8, **kw)[None, :]) * h
        g = torch.exp(-2 * d * d / 0.05**2)
        return g / g.square().sum(1, keepdim=True).sqrt()

    z = torch.randn(2 * count, nry + 16, nrx + 16, generator=gen, **kw)
    f = 0.1 * factor(nry, dy) @ z @ factor(nrx, dx).T
    e = f[:, torch.from_numpy(fluid).cuda()].reshape(count, 2, -1)
    if y_only:
        e[:, 0] = 0.0
    return e.reshape(count, -1).T.contiguous()


def _weights(n, seed):
    return 0.1 * np.random.default_rng(seed).standard_normal(n)


def _setup(c):
    return (PAPER, 1e-6) if c.get("paper") else (CAVITY, 0.1)


def _handle(c, **kw):
    box, delta = _setup(c)
    prec = {"mixed": pkg.MIXED, "fp64": pkg.FP64_BATCHED, "plain": pkg.FP64_PLAIN}[c["prec"]]
    cost = pkg.COST_SENSORS if c.get("cost") == "sensors" else pkg.COST_DOMAIN
    cfg = pkg.default_config(c["nx"], c["ny"], y1=box[3], Re=c["re"], n_steps=c["steps"], n_window=c["window"], inlet_delta=delta,
                             precision=prec, cost_mode=cost, lip_slip=int(bool(c.get("paper"))), forcing_y_only=int(bool(c.get("paper"))),
                             **(TUNED if c["solver"] == "tuned" else DEFAULT), **kw)
    return pkg.Ensemble(cfg)


def _subs(c):
    """The batch's handles as run cases: horizons 1 : 2 : 4 times the first."""
    for k, g in enumerate(c["grids"].split(",")):
        nx, ny, n = (int(v) for v in g.split("x"))
        steps = c["steps"] * 2**k
        yield {"prec": c["prec"], "cost": "domain", "nx": nx, "ny": ny, "re": (4000.0, 7500.0, 15000.0)[k], "n": n, "steps": steps,
               "window": steps // 2, "solver": _solver(nx, ny), "call": "step"}


def _eigen_prior(seed):
    a = np.random.default_rng(seed).random(2)
    return 0.08 + 0.04 * a[0], 0.045 + 0.01 * a[1]


def prepare(case, seed):
    c = case
    if c["kind"] in ("run", "trial", "adjoint"):
        box, delta = _setup(c)
        c = dict(c, prec="plain") if c["kind"] == "adjoint" else c
        ens = _handle(c, n_members=c.get("n", 1))
        ens.set_initial_state(*_flow(c["nx"], c["ny"], box, delta, seed))
        if c["kind"] == "run":
            ens.set_ensemble(_fields(c["nx"], c["ny"], box, c["n"], c["paper"], seed + 1))
            return {"case": c, "ens": ens, "w": _weights(c["n"], seed + 2)}
        return {"case": c, "ens": ens, "f": _fields(c["nx"], c["ny"], box, 1, False, seed + 1)[:, 0].contiguous()}
    if c["kind"] == "batch":
        hs, ws = [], []
        for k, s in enumerate(_subs(c)):
            ens = _handle(s, n_members=s["n"])
            ens.set_initial_state(*_flow(s["nx"], s["ny"], CAVITY, 0.1, seed + 10 * k))
            ens.set_ensemble(_fields(s["nx"], s["ny"], CAVITY, s["n"], False, seed + 10 * k + 1))
            hs.append(ens)
            ws.append(_weights(s["n"], seed + 10 * k + 2))
        return {"case": c, "hs": hs, "ws": ws, "batch": pkg.Batch(hs)}
    sigma, a = _eigen_prior(seed) if c["kind"] == "eigen" else (0.1, 0.05)
    ens = pkg.Ensemble(pkg.default_config(c["nx"], c["ny"], n_members=c.get("n", 1), n_steps=2, n_window=1, sigma=sigma, corr_len=a,
                                          precision=pkg.FP64_PLAIN if c["kind"] == "h1" else pkg.MIXED))
    if c["kind"] == "eigen":
        return {"case": c, "ens": ens}
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return {"case": c, "ens": ens, "g": torch.randn(ens.n_ctrl, generator=gen, dtype=torch.float64, device="cuda")}


def _results(ens, member):
    u, v, p = ens.get_state(member)
    return {"J": ens.cost()[0], "u": u, "v": v, "p": p}


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "run":
        ens = state["ens"]
        w, j0 = ens.step(0.5, state["w"]) if c["call"] == "step" else ens.gn_step(1.0, state["w"])
        out = {"w": w, "J0": j0, **_results(ens, c["n"] if c["prec"] == "plain" else 0)}
        if c["call"] == "gn":
            out["H"] = ens.gn_hessian()
        return out
    if kind == "trial":
        j = state["ens"].forward_control(state["f"])
        return {"J": j, **dict(zip("uvp", state["ens"].get_state(0)))}
    if kind == "batch":
        state["batch"].forward(state["ws"])
        return [{"g": e.gradient(), **_results(e, 0)} for e in state["hs"]]
    if kind == "adjoint":
        j, g = state["ens"].adjoint_gradient(state["f"], c["snapshots"])
        return {"J": j, "g": g}
    if kind == "eigen":
        lam = state["ens"].use_eigen_ensemble()
        return {"lam": lam, "E": state["ens"].get_ensemble()}
    return state["ens"].h1_smooth(state["g"])


def work(case):
    """Bytes: per step and member the state read and written once (velocity, pressure, previous tendency and pressure
    increment, in the handle's types) on the fluid cells; flops: predictor, right-hand side and correction, and per step
    one multigrid-preconditioned solve of two V-cycles.  Stages: inputs and outputs once, and their products."""
    c = case
    if c["kind"] == "batch":
        parts = [work(dict(s, kind="run", paper=False)) for s in _subs(c)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    _, _, xc, yc = _axes(c["nx"], c["ny"], _setup(c)[0])
    fluid = float(((yc[:, None] > 0) | ((xc > 0) & (xc < 1))[None, :]).sum())
    _, _, nrx, nry, ctl = _control(c["nx"], c["ny"], _setup(c)[0])
    ncc = float(ctl.sum())
    if c["kind"] in ("run", "trial", "adjoint"):
        mixed = c.get("prec") == "mixed"
        steps = c["steps"] * (c["n"] + 1 if c["kind"] == "run" else 1) * (3 if c["kind"] == "adjoint" else 1)
        return {"bytes": steps * fluid * (64 if mixed else 96), "flops": steps * fluid * 450.0}
    if c["kind"] == "eigen":
        lanczos = 2.0 * c["n"]
        return {"bytes": 8.0 * 2 * ncc * c["n"], "flops": lanczos * (2.0 * nrx * nry * (nrx + nry) + 4.0 * lanczos * ncc)}
    return {"bytes": 8.0 * 4 * ncc, "flops": 2 * 100 * 20 * ncc}


# ---------------------------------------------------------------------------------------------- 64-bit restatement
class _Flow:
    """The discretised flow on one grid, batched over members, in float64 torch (differentiable in the forcing)."""

    def __init__(self, c):
        box, delta = _setup(c)
        self.c, self.nx, self.ny = c, c["nx"], c["ny"]
        nx, ny = self.nx, self.ny
        self.dx, self.dy, xc, yc = _axes(nx, ny, box)
        self.box, self.dt, self.nu = box, 0.3 * min(self.dx, self.dy), 1.0 / c["re"]
        f = (yc[:, None] > 0) | ((xc > 0) & (xc < 1))[None, :]
        dev = lambda a: torch.as_tensor(np.ascontiguousarray(a)).cuda()  # noqa: E731
        uu, ub = np.zeros((ny, nx + 1), bool), np.zeros((ny, nx + 1), bool)
        uu[:, 1:-1], ub[:, 1:-1] = f[:, 1:] & f[:, :-1], ~f[:, 1:] & ~f[:, :-1]
        vu, vb = np.zeros((ny + 1, nx), bool), np.zeros((ny + 1, nx), bool)
        vu[1:-1], vb[1:-1] = f[1:] & f[:-1], ~f[1:] & ~f[:-1]
        slip = np.zeros_like(ub)
        if c.get("paper"):
            xf = box[0] + np.arange(nx + 1) * self.dx
            slip[:-1] = ub[:-1] & uu[1:] & ((xf < SLIP_SPAN[0]) | (xf > SLIP_SPAN[1]))[None, :]
        # what a u face sees north / south (v face: east / west): +1 its own value, -1 its mirror, 0 the neighbour's
        sn, ss = np.zeros(uu.shape), np.zeros(uu.shape)
        sn[-1], ss[0] = 1.0, -1.0
        sn[:-1] = np.where(slip[1:], 1.0, np.where(ub[1:], -1.0, 0.0))
        ss[1:] = np.where(slip[:-1], 1.0, np.where(ub[:-1], -1.0, 0.0))
        se, sw = np.zeros(vu.shape), np.zeros(vu.shape)
        se[:, -1], sw[:, 0] = 1.0, -1.0
        se[:, :-1] = np.where(vb[:, 1:], -1.0, 0.0)
        sw[:, 1:] = np.where(vb[:, :-1], -1.0, 0.0)
        self.f, self.uu, self.vu = dev(f), dev(uu), dev(vu)
        self.sn, self.ss, self.se, self.sw = dev(sn), dev(ss), dev(se), dev(sw)
        self.inlet, self.out = dev(f[:, 0]), dev(f[:, -1])
        self.uin = dev(np.array([math.erf(y / delta) for y in yc]) * f[:, 0])
        self._poisson(f)

    def _poisson(self, f):
        """Direct solve: channel and cavity are rectangles that the cosine transform diagonalises; the faces between them
        and the constants are a low-rank update (Woodbury)."""
        nx, ny = self.nx, self.ny
        kw = {"dtype": torch.float64, "device": "cuda"}
        self.cx, self.cy = self.dy / self.dx, self.dx / self.dy
        self.jl = jl = int(np.flatnonzero(f.all(1))[0])
        cols = np.flatnonzero(f[0])
        self.ca, self.cb = ca, cb = int(cols[0]), int(cols[-1]) + 1

        def basis(n):
            k = torch.arange(n, **kw)
            q = torch.cos(math.pi * k[None, :] * (k[:, None] + 0.5) / n) * math.sqrt(2.0 / n)
            q[:, 0] = 1.0 / math.sqrt(n)
            return q, 2.0 - 2.0 * torch.cos(math.pi * k / n)

        self.rects = []
        for j0, j1, i0, i1 in ((jl, ny, 0, nx), (0, jl, ca, cb)):
            (qy, ly), (qx, lx) = basis(j1 - j0), basis(i1 - i0)
            lam = self.cy * ly[:, None] + self.cx * lx[None, :]
            lam[0, 0] = 1.0
            self.rects.append((j0, j1, i0, i1, qy, qx, lam))
        nc = cb - ca
        U = torch.zeros(nc + 3, ny, nx, **kw)
        r = torch.arange(nc, device="cuda")
        U[r, jl, ca + r], U[r, jl - 1, ca + r] = 1.0, -1.0
        fl = torch.as_tensor(f).cuda()
        for k, (j0, j1, i0, i1, *_) in enumerate(self.rects):
            U[nc + k, j0:j1, i0:i1] = 1.0 / math.sqrt((j1 - j0) * (i1 - i0))
        U[nc + 2][fl] = 1.0 / math.sqrt(float(f.sum()))
        D = torch.cat([torch.full((nc,), self.cy, **kw), torch.tensor([-1.0, -1.0, 1.0], **kw)])
        self.U = U.reshape(nc + 3, -1)
        self.W = torch.cat([self._fast(u[None]).reshape(1, -1) for u in U])
        self.K = torch.linalg.inv(torch.diag(1.0 / D) + self.U @ self.W.T)

    def _fast(self, b):
        x = torch.zeros_like(b)
        for j0, j1, i0, i1, qy, qx, lam in self.rects:
            x[:, j0:j1, i0:i1] = qy @ ((qy.T @ b[:, j0:j1, i0:i1] @ qx) / lam) @ qx.T
        return x

    def _apply(self, x):
        gx = torch.where(self.uu[:, 1:-1], self.cx * (x[:, :, 1:] - x[:, :, :-1]), 0.0)
        gy = torch.where(self.vu[1:-1], self.cy * (x[:, 1:] - x[:, :-1]), 0.0)
        pad = torch.nn.functional.pad
        return pad(gx, (1, 0)) - pad(gx, (0, 1)) + pad(gy, (0, 0, 1, 0)) - pad(gy, (0, 0, 0, 1))

    def solve(self, b):
        def once(r):
            y = self._fast(r)
            t = (y.reshape(len(r), -1) @ self.U.T) @ self.K.T
            return y - (t @ self.W).reshape(y.shape)

        x = once(b)
        return torch.where(self.f, x + once(b - self._apply(x)), 0.0)

    def load(self, u, v):
        u = torch.where(self.uu, u, 0.0)
        u[:, -1] = 0.0
        u0 = u.clone()
        u0[:, 0] = self.uin
        return u0, torch.where(self.vu, v, 0.0)

    def faces(self, f):
        """Control vectors (rows of f) to forces on the u and v faces: half from each neighbouring control cell."""
        ia, ja, nrx, nry, mask = _control(self.nx, self.ny, self.box)
        m = torch.from_numpy(mask).cuda()
        rect = torch.zeros(len(f), 2, nry, nrx, dtype=torch.float64, device="cuda")
        at = m.flatten().nonzero()[:, 0]
        rect = rect.reshape(len(f), 2, -1).index_copy(2, at, f.reshape(len(f), 2, -1)).reshape(rect.shape)
        pad = torch.nn.functional.pad
        cell = pad(rect, (ia, self.nx - ia - nrx, ja, self.ny - ja - nry))
        return 0.5 * (pad(cell[:, 0], (1, 0)) + pad(cell[:, 0], (0, 1))), 0.5 * (pad(cell[:, 1], (0, 0, 1, 0)) + pad(cell[:, 1], (0, 0, 0, 1)))

    def tendency(self, u, v):
        pad = torch.nn.functional.pad
        i4x, i4y = 0.25 / self.dx, 0.25 / self.dy
        nx2, ny2 = self.nu / self.dx**2, self.nu / self.dy**2
        uc, ue, uw = u[:, :, 1:-1], u[:, :, 2:], u[:, :, :-2]
        sn, ss = self.sn[:, 1:-1], self.ss[:, 1:-1]
        un = torch.where(sn != 0, sn * uc, pad(uc[:, 1:], (0, 0, 0, 1)))
        us = torch.where(ss != 0, ss * uc, pad(uc[:, :-1], (0, 0, 1, 0)))
        vn, vs = v[:, 1:, 1:] + v[:, 1:, :-1], v[:, :-1, 1:] + v[:, :-1, :-1]
        ru = nx2 * (ue - 2 * uc + uw) + ny2 * (un - 2 * uc + us) - ((uc + ue) ** 2 - (uw + uc) ** 2) * i4x - ((uc + un) * vn - (us + uc) * vs) * i4y
        vc, vN, vS = v[:, 1:-1], v[:, 2:], v[:, :-2]
        se, sw = self.se[1:-1], self.sw[1:-1]
        ve = torch.where(se != 0, se * vc, pad(vc[:, :, 1:], (0, 1)))
        vw = torch.where(sw != 0, sw * vc, pad(vc[:, :, :-1], (1, 0)))
        ue2, uw2 = u[:, 1:, 1:] + u[:, :-1, 1:], u[:, 1:, :-1] + u[:, :-1, :-1]
        rv = nx2 * (ve - 2 * vc + vw) + ny2 * (vN - 2 * vc + vS) - (ue2 * (vc + ve) - uw2 * (vw + vc)) * i4x - ((vc + vN) ** 2 - (vS + vc) ** 2) * i4y
        return pad(ru, (1, 1)), pad(rv, (0, 0, 1, 1))

    def simulate(self, u0, v0, f, each):
        """Runs the members with control vectors f (rows); each(n, u, v) after step n = 1 ..; returns u, v, p."""
        fu, fv = self.faces(f)
        M, dt = len(f), self.dt
        u, v = self.load(u0.clone(), v0.clone())
        u, v = u.expand(M, -1, -1), v.expand(M, -1, -1)
        # the outlet keeps the raw values of the initial state
        u = torch.cat([u[:, :, :-1], torch.where(self.out, u0[:, -1], 0.0).expand(M, -1)[:, :, None]], 2)
        p = torch.zeros(M, self.ny, self.nx, dtype=torch.float64, device="cuda")
        old = None
        for n in range(1, self.c["steps"] + 1):
            ub = torch.where(self.out, u[:, :, -1] - dt * (u[:, :, -1] - u[:, :, -2]) / self.dx, 0.0)
            ub = torch.where(self.out, ub + (self.uin.sum() - ub.sum(1, keepdim=True)) / self.out.sum(), 0.0)
            ru, rv = self.tendency(u, v)
            a, b = (ru, rv) if old is None else (1.5 * ru - 0.5 * old[0], 1.5 * rv - 0.5 * old[1])
            old = (ru, rv)
            pad = torch.nn.functional.pad
            gx = pad((p[:, :, 1:] - p[:, :, :-1]) / self.dx, (1, 1))
            gy = pad((p[:, 1:] - p[:, :-1]) / self.dy, (0, 0, 1, 1))
            us = torch.where(self.uu, u + dt * (a + fu - gx), 0.0)
            us = torch.cat([self.uin.expand(M, -1)[:, :, None], us[:, :, 1:-1], ub[:, :, None]], 2)
            vs = torch.where(self.vu, v + dt * (b + fv - gy), 0.0)
            div = self.dy * (us[:, :, 1:] - us[:, :, :-1]) + self.dx * (vs[:, 1:] - vs[:, :-1])
            x = self.solve(torch.where(self.f, -div / dt, 0.0))
            u = us - torch.where(self.uu, dt * pad((x[:, :, 1:] - x[:, :, :-1]) / self.dx, (1, 1)), 0.0)
            v = vs - torch.where(self.vu, dt * pad((x[:, 1:] - x[:, :-1]) / self.dy, (0, 0, 1, 1)), 0.0)
            p = p + torch.where(self.f, x - x.sum((1, 2), keepdim=True) / self.f.sum(), 0.0)
            each(n, u, v)
        return u, v, p

    def centred(self, u, v):
        return torch.where(self.f, 0.5 * (u[:, :, 1:] + u[:, :, :-1]), 0.0), torch.where(self.f, 0.5 * (v[:, 1:] + v[:, :-1]), 0.0)

    def sensors(self, u, v):
        """(u, v) at (k/5, 0), k = 1 .. 4, bilinear on the faces: (M, 8)."""
        got = []
        for k in range(4):
            for a, ox, oy in ((u, 0.0, 0.5), (v, 0.5, 0.0)):
                fi, fj = (0.2 * (k + 1) - self.box[0]) / self.dx - ox, (0.0 - self.box[2]) / self.dy - oy
                i, j = math.floor(fi), math.floor(fj)
                tx, ty = fi - i, fj - j
                row = lambda r: (1 - tx) * a[:, r, i] + tx * a[:, r, i + 1]  # noqa: E731,B023
                got.append((1 - ty) * row(j) + (ty * row(j + 1) if ty > 0 else 0.0))
        return torch.stack(got, 1)


def _exact_run(c, seed):
    """Costs, gradient and the last states of the N + 1 runs, members in parts of at most 2^24 cells."""
    box, delta = _setup(c)
    F, n, nw = _Flow(c), c["n"], c["window"]
    u0, v0 = _flow(c["nx"], c["ny"], box, delta, seed)
    E = _fields(c["nx"], c["ny"], box, n, c.get("paper"), seed + 1)
    w = torch.as_tensor(_weights(n, seed + 2)).cuda()
    f = torch.cat([(E @ w)[None], (E @ w)[None] + EPS * E.T])
    domain = c["cost"] == "domain"
    J, Yd, H, last, ref = [], [], [], {}, []
    part = max(1, (1 << 24) // (c["nx"] * c["ny"]))
    for m0 in range(0, n + 1, part):
        fm = f[m0:m0 + part]
        s1, s2, d1, d2, series = 0.0, 0.0, 0.0, 0.0, []

        def each(k, u, v):
            nonlocal s1, s2, d1, d2
            if k <= c["steps"] - nw:
                return
            if not domain:
                series.append(F.sensors(u, v))
                return
            q = torch.stack(F.centred(u, v), 1)
            t = k - (c["steps"] - nw) - 1
            if m0 == 0:
                ref.append(q[0].clone())
            # about the first sample and about member 0: small numbers, so that the sums of squares lose nothing
            e, d = q - ref[0], q - ref[t]
            s1, s2, d1, d2 = s1 + e, s2 + e * e, d1 + d, d2 + d * d

        u, v, p = F.simulate(u0, v0, fm, each)
        if m0 == 0:
            last[0] = (u[0].clone(), v[0].clone(), p[0].clone())
        last[m0 + len(fm) - 1] = (u[-1].clone(), v[-1].clone(), p[-1].clone())
        if domain:
            h = F.dx * F.dy / (2.0 * nw)
            J.append(h * (s2 - s1 * s1 / nw).sum((1, 2, 3)))
            Yd.append(h * (d2 - d1 * d1 / nw).sum((1, 2, 3)))
        else:
            s = torch.stack(series, 1)
            H.append((s - s.mean(1, keepdim=True)).reshape(len(fm), -1))
    if domain:
        J, Yd = torch.cat(J), torch.cat(Yd)
        g = (J[1:] - J[0] - Yd[1:]) / EPS + (n - 1) * w
        Y = None
    else:
        H = torch.cat(H)
        J, Y = 0.5 * H.square().sum(1), (H[1:] - H[0]) / EPS
        g = Y @ H[0] + (n - 1) * w
    return J, g, w, Y, last


def _say(J, state):
    return {"J": J.cpu().numpy(), **dict(zip("uvp", state))}


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "run":
        J, g, w, Y, last = _exact_run(c, seed)
        n = c["n"]
        out = _say(J, last[n if c["prec"] == "plain" else 0])
        out["J0"] = float(J[0] + 0.5 * (n - 1) * (w @ w))
        if c["call"] == "gn":
            H = Y @ Y.T + (n - 1) * torch.eye(n, dtype=torch.float64, device="cuda")
            return {**out, "H": H.cpu().numpy(), "w": (w - torch.linalg.solve(H, g)).cpu().numpy()}
        return {**out, "w": (w - 0.5 * g / max(n - 1, 1)).cpu().numpy()}
    if kind == "batch":
        got = []
        for k, s in enumerate(_subs(c)):
            J, g, _, _, last = _exact_run(s, seed + 10 * k)
            got.append({"g": g.cpu().numpy(), **_say(J, last[0])})
        return got
    if kind in ("trial", "adjoint"):
        box, delta = _setup(c)
        F = _Flow(c)
        f = _fields(c["nx"], c["ny"], box, 1, False, seed + 1).T.contiguous().requires_grad_(kind == "adjoint")
        q = []
        with torch.set_grad_enabled(kind == "adjoint"):
            u, v, p = F.simulate(*_flow(c["nx"], c["ny"], box, delta, seed), f,
                                 lambda k, u, v: q.append(torch.stack(F.centred(u, v))) if k > c["steps"] - c["window"] else None)
            q = torch.stack(q)
            J = F.dx * F.dy / (2.0 * c["window"]) * (q - q.mean(0)).square().sum()
            if kind == "adjoint":
                return {"J": float(J.detach()), "g": torch.autograd.grad(J, f)[0][0]}
        return {"J": float(J), "u": u[0], "v": v[0], "p": p[0]}
    kw = {"dtype": torch.float64, "device": "cuda"}
    dx, dy, _, _ = _axes(c["nx"], c["ny"], CAVITY)
    ia, ja, nrx, nry, mask = _control(c["nx"], c["ny"], CAVITY)
    m = torch.from_numpy(mask).cuda()
    if kind == "eigen":
        sigma, a = _eigen_prior(seed)
        j, i = (t.to(torch.float64) for t in m.nonzero(as_tuple=True))
        B = sigma**2 * torch.exp(-(((i[:, None] - i) * dx) ** 2 + ((j[:, None] - j) * dy) ** 2) / a**2)
        lam, V = torch.linalg.eigh(B)
        r = torch.arange(c["n"], device="cuda") // 2
        lam, V = lam.flip(0)[r], V.flip(1)[:, r]
        V = V * torch.sign(V.gather(0, V.abs().argmax(0, keepdim=True)))
        E = torch.zeros(2, len(i), c["n"], **kw)
        k = torch.arange(c["n"], device="cuda")
        E[k % 2, :, k] = (V * (lam * (c["n"] - 1)).sqrt()).T
        return {"lam": lam.cpu().numpy(), "E": E.reshape(-1, c["n"])}
    # (I - l^2 Lap) x = (1 + l^2) g, no flux through the control set's boundary: CG in 64 bits
    gen = torch.Generator(device="cuda").manual_seed(seed)
    l2 = 0.02**2
    b = torch.zeros(2, nry, nrx, **kw)
    b[:, m] = (1 + l2) * torch.randn(2 * int(m.sum()), generator=gen, **kw).reshape(2, -1)
    ox, oy = (m[:, 1:] & m[:, :-1]).to(torch.float64) * (l2 / dx**2), (m[1:] & m[:-1]).to(torch.float64) * (l2 / dy**2)
    pad = torch.nn.functional.pad

    def A(x):
        gx, gy = ox * (x[:, :, 1:] - x[:, :, :-1]), oy * (x[:, 1:] - x[:, :-1])
        return x + pad(gx, (1, 0)) - pad(gx, (0, 1)) + pad(gy, (0, 0, 1, 0)) - pad(gy, (0, 0, 0, 1))

    x, r = torch.zeros_like(b), b.clone()
    p, rr = r.clone(), r.square().sum()
    for _ in range(2000):
        if rr <= 1e-30 * b.square().sum():
            break
        q = A(p)
        al = rr / (p * q).sum()
        x, r = x + al * p, r - al * q
        new = r.square().sum()
        p, rr = r + new / rr * p, new
    return x[:, m].reshape(-1)
