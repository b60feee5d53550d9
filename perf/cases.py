"""The work a user of this library has it do, as cases that can be timed and checked.

A case is a dict of plain values. Its "run" names the shape of the user's program:

  solve   one initial-value problem on one simulation: set the weights, advance, read them back
          (FEL: with the field history; "moments": with the FP64 diagnostics at the end)
  host    the same from and to NumPy arrays
  watch   a run that is looked at while it goes: a few steps, then the diagnostics, several times
  batch   many small simulations advanced together, then all of them read back
  serve   requests of mixed size and length through the request server, until it has drained

Every pass starts from its own initial weights, so that passes do not depend on each other. Meshes and
physics are those of inputs.py and the tests: the pendulum of Sec. IV.A, the linear oscillator turned by
pi/10 per step, and the 1-D FEL of Sec. IV.B, with the drift-kick-drift and the RK4 integrator.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2007_12227_gb300 import inputs as I
from paper_2007_12227_gb300 import vlasov as V

PI = math.pi
TENT, CUBIC = V.VP_BASIS_TENT, V.VP_BASIS_CUBIC_BSPLINE


def listed():
    return [
        # the paper's proof-of-concept size: a small FP64 run with the tent deposit, in and out through
        # NumPy, where launches and latency are everything
        dict(name="pendulum_128_fp64_tent", run="host", physics="pendulum", nx=128, np=128, fp64=True,
             basis="tent", lumped=False, steps=100),
        # the headline mesh on the plan that the autotuner gives
        dict(name="pendulum_8192_tuned", run="solve", physics="pendulum", nx=8192, np=8192, fp64=False,
             basis="cubic", lumped=False, steps=10, tuned=True, moments=False),
        # weights that stay non-negative: the lumped projection, the deposit alone
        dict(name="pendulum_4096_lumped", run="solve", physics="pendulum", nx=4096, np=4096, fp64=False,
             basis="cubic", lumped=True, steps=20, tuned=False, moments=False),
        # an ordinary mesh of no special size on the default plan, with the diagnostics at the end
        dict(name="pendulum_1000x901", run="solve", physics="pendulum", nx=1000, np=901, fp64=False,
             basis="cubic", lumped=False, steps=50, tuned=False, moments=True),
        # a mesh with odd rows (no vector access fits them), still small enough to leave the chip idle
        dict(name="pendulum_357x300", run="solve", physics="pendulum", nx=357, np=300, fp64=False,
             basis="cubic", lumped=False, steps=50, tuned=False, moments=False),
        # the FEL run of the benchmark on the default plan, with its field history
        dict(name="fel_4096x2048", run="solve", physics="fel", nx=4096, np=2048, fp64=False,
             basis="cubic", lumped=False, steps=20, tuned=False, moments=False),
        # double precision, as a check on an FP32 run needs it
        dict(name="pendulum_1024_fp64", run="solve", physics="pendulum", nx=1024, np=1024, fp64=True,
             basis="cubic", lumped=False, steps=10, tuned=False, moments=False),
        # the linear oscillator of Sec. IV.A, one revolution: strong shear of both axes in every step
        dict(name="rotation_640x512", run="solve", physics="rotation", nx=640, np=512, fp64=False,
             basis="cubic", lumped=False, steps=20, tuned=False, moments=False),
        # the paper's own FEL integrator
        dict(name="fel_rk4_512x256_fp64", run="solve", physics="fel_rk4", nx=512, np=256, fp64=True,
             basis="cubic", lumped=False, steps=10, tuned=False, moments=False),
        # a run with its diagnostics (mass, energy, entropy) written down every few steps
        dict(name="pendulum_2048_watched", run="watch", physics="pendulum", nx=2048, np=2048, fp64=False,
             basis="cubic", lumped=False, steps=5, looks=6),
        # a parameter scan: ragged pendulum and FEL instances as one batch on a graph
        dict(name="batch_40", run="batch", count=40, nmin=64, nmax=1024, steps=20, mix=1),
        # requests of mixed size and length through the server
        dict(name="serve_12", run="serve", count=12, nmin=128, nmax=1024, smin=50, smax=400, mix=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["host", "solve", "solve", "solve", "fp64", "fel", "rotation", "rk4", "watch", "batch",
                       "serve"])
    if kind == "host":
        return dict(run="host", physics="pendulum", nx=_log(rng, 64, 512), np=_log(rng, 64, 512), fp64=True,
                    basis=rng.choice(["tent", "cubic"]), lumped=False, steps=rng.randint(50, 150))
    if kind == "solve":
        return dict(run="solve", physics="pendulum", nx=_log(rng, 200, 8192), np=_log(rng, 200, 8192), fp64=False,
                    basis="cubic", lumped=rng.random() < 0.3, steps=rng.randint(4, 10), tuned=rng.random() < 0.2,
                    moments=rng.random() < 0.3)
    if kind == "fp64":
        return dict(run="solve", physics="pendulum", nx=_log(rng, 128, 1024), np=_log(rng, 128, 1024), fp64=True,
                    basis=rng.choice(["tent", "cubic"]), lumped=False, steps=rng.randint(4, 10), tuned=False,
                    moments=False)
    if kind == "fel":
        return dict(run="solve", physics="fel", nx=_log(rng, 256, 4096), np=_log(rng, 256, 4096), fp64=False,
                    basis="cubic", lumped=rng.random() < 0.2, steps=rng.randint(4, 20), tuned=False,
                    moments=rng.random() < 0.3)
    if kind == "rotation":
        return dict(run="solve", physics="rotation", nx=_log(rng, 400, 1500), np=_log(rng, 300, 1500),
                    fp64=rng.random() < 0.3, basis="cubic", lumped=False, steps=rng.randint(4, 20), tuned=False,
                    moments=False)
    if kind == "rk4":
        return dict(run="solve", physics="fel_rk4", nx=_log(rng, 128, 1024), np=_log(rng, 128, 1024),
                    fp64=rng.random() < 0.5, basis="cubic", lumped=False, steps=rng.randint(4, 10), tuned=False,
                    moments=False)
    if kind == "watch":
        return dict(run="watch", physics=rng.choice(["pendulum", "fel"]), nx=_log(rng, 256, 4096),
                    np=_log(rng, 256, 4096), fp64=False, basis="cubic", lumped=rng.random() < 0.3,
                    steps=rng.randint(2, 5), looks=rng.randint(3, 6))
    if kind == "batch":
        return dict(run="batch", count=rng.randint(16, 48), nmin=64, nmax=_log(rng, 256, 1024),
                    steps=rng.randint(10, 20), mix=rng.randint(2, 1 << 20))
    return dict(run="serve", count=rng.randint(6, 12), nmin=128, nmax=_log(rng, 256, 1024), smin=50,
                smax=rng.randint(100, 400), mix=rng.randint(2, 1 << 20))


# ------------------------------------------------------------------ inputs
def _problem(physics, nx, np_, rng):
    """Grid, pusher and the parameters of the initial density, from the seeded rng."""
    if physics == "pendulum":
        grid = I.Grid(nx, np_, -PI, PI, -4.0, 4.0)
        push = I.Pusher(I.PUSH_KDK, I.POT_PENDULUM, 1.0, 1.0, 0.02)
        dens = [(rng.uniform(0.5, 1.5), rng.uniform(-0.3, 0.3), rng.uniform(0.3, 0.7), 0.4),
                (rng.uniform(0.5, 1.5), rng.uniform(-0.3, 0.3), rng.uniform(2.3, 2.6), 0.2)]
    elif physics == "rotation":
        grid = I.Grid(nx, np_, -4.0, 4.0, -4.0, 4.0)
        push = I.Pusher(I.PUSH_ROTATION, I.POT_HARMONIC, 1.0, 1.0, PI / 10)
        dens = [(1.0, rng.uniform(0.8, 1.2), rng.uniform(-0.2, 0.2), rng.uniform(0.3, 0.4))]
    else:
        grid = I.Grid(nx, np_, 0.0, 2 * PI, -4.0, 4.0)
        kind = I.PUSH_FEL if physics == "fel" else I.PUSH_FEL_RK4
        push = I.Pusher(kind, I.POT_FREE, 1.0, 1.0, 0.01, math.exp(rng.uniform(math.log(5e-4), math.log(5e-3))), 0.0)
        # thermal spread, modulation depth and phase
        dens = (rng.uniform(0.05, 0.2), rng.uniform(0.5e-4, 2e-4), rng.uniform(0.0, 2 * PI))
    return grid, push, dens


def _nodes(grid):
    x = grid.x0 + torch.arange(grid.nx, dtype=torch.float64, device="cuda") * ((grid.x1 - grid.x0) / grid.nx)
    p = grid.p0 + torch.arange(grid.np, dtype=torch.float64, device="cuda") * ((grid.p1 - grid.p0) / (grid.np - 1))
    return x, p


def _density(physics, grid, dens, dtype):
    """Nodal weights [np][nx] on the GPU, normalised to unit mass."""
    x, p = _nodes(grid)
    if physics in ("pendulum", "rotation"):
        L = grid.x1 - grid.x0
        f = torch.zeros(grid.np, grid.nx, dtype=torch.float64, device="cuda")
        for c, xc, pc, s in dens:
            dx = torch.remainder(x - xc + 0.5 * L, L) - 0.5 * L
            f += c * torch.exp(-0.5 * ((p - pc) / s) ** 2)[:, None] * torch.exp(-0.5 * (dx / s) ** 2)[None, :]
    else:
        sp, eps, ph = dens
        f = torch.exp(-0.5 * (p / sp) ** 2)[:, None] * (1.0 + eps * torch.cos(x - ph))[None, :]
    hx, hp = (grid.x1 - grid.x0) / grid.nx, (grid.p1 - grid.p0) / (grid.np - 1)
    return (f / (f.sum() * hx * hp)).to(dtype)


def _members(case):
    """Sizes and physics of a batch's or a server's members: half pendulum, half FEL."""
    rng = random.Random(case["mix"])
    out = []
    for k in range(case["count"]):
        n = _log(rng, case["nmin"], case["nmax"])
        steps = _log(rng, case["smin"], case["smax"]) if "smin" in case else case["steps"]
        out.append(("fel" if k % 2 else "pendulum", n, steps))
    return out


def _inputs(case, seed):
    """(physics, grid, pusher, steps, weights) of each simulation of the case."""
    rng = random.Random(seed)
    if case["run"] in ("batch", "serve"):
        members = [(ph, n, n, steps) for ph, n, steps in _members(case)]
        dtype = torch.float32
    else:
        members = [(case["physics"], case["nx"], case["np"], case["steps"])]
        dtype = torch.float64 if case["fp64"] else torch.float32
    out = []
    for ph, nx, np_, steps in members:
        grid, push, dens = _problem(ph, nx, np_, rng)
        out.append((ph, grid, push, steps, _density(ph, grid, dens, dtype)))
    return out


def prepare(case, seed):
    got = _inputs(case, seed)
    st = dict(case=case)
    if case["run"] == "serve":
        st["stream"] = torch.cuda.Stream()   # a created stream: the server's batches replay graphs on it
        arena = sum(24 * g.nx * g.np + (1 << 20) for _, g, _, _, _ in got)
        st["server"] = V.Server(arena, stream=st["stream"])
        st["requests"] = [(g, pu, n, f.cpu().numpy()) for _, g, pu, n, f in got]
        return st
    if case["run"] == "batch":
        st["stream"] = torch.cuda.Stream()
        torch.cuda.synchronize()   # the simulations are built on that stream
        st["sims"] = [V.Sim(g, CUBIC, pu, stream=st["stream"], history_cap=256) for _, g, pu, _, _ in got]
        st["f"] = [f for *_, f in got]
        st["out"] = [torch.empty_like(f) for f in st["f"]]
        for s, f in zip(st["sims"], st["f"]):
            s.set_f(f)
        st["batch"] = V.Batch(st["sims"], stream=st["stream"])
        return st
    ph, grid, push, _, f = got[0]
    basis = TENT if case["basis"] == "tent" else CUBIC
    proj = V.VP_PROJ_LUMPED if case["lumped"] else V.VP_PROJ_GALERKIN
    prec = V.VP_FP64 if case["fp64"] else V.VP_FP32
    plan = dict(kernel=V.VP_KERNEL_AUTO, tile_x=0, tile_p=0)
    if case.get("tuned"):
        wl = I.Workload("case", grid, push, basis, prec, case["steps"], "", projection=proj)
        t = V.autotune([wl], precision=prec, projection=proj)[0]   # kept for the process
        plan = {k: t[k] for k in plan}
    st["sim"] = V.Sim(grid, basis, push, precision=prec, projection=proj, **plan)
    st["f"] = f.cpu().numpy() if case["run"] == "host" else f
    st["out"] = torch.empty_like(f)
    return st


# ------------------------------------------------------------------ the passes
def _kept(case, values):
    """Diagnostics and histories as numbers of the run's own precision."""
    return torch.tensor(values, dtype=torch.float64 if case.get("fp64") else torch.float32)


def run(state):
    case = state["case"]
    if case["run"] == "serve":
        srv, reqs = state["server"], state["requests"]
        for k, (grid, push, steps, f) in enumerate(reqs):
            srv.submit(k, grid, CUBIC, push, f, steps, keep_f=True)
        while sum(srv.run(16)) > 0:
            pass
        done = sorted(srv.poll(), key=lambda r: r["id"])
        weights = [srv.take_f(k, f.shape, np.float32) for k, (*_, f) in enumerate(reqs)]
        return dict(weights=weights, moments=_kept(case, [list(r["moments"].values()) for r in done]))
    if case["run"] == "batch":
        for s, f in zip(state["sims"], state["f"]):
            s.set_f(f)
        state["batch"].step(case["steps"])
        for s, o in zip(state["sims"], state["out"]):
            s.get_f_device(o)
        torch.cuda.current_stream().wait_stream(state["stream"])
        return state["out"]
    sim = state["sim"]
    sim.set_f(state["f"])
    if case["run"] == "host":
        sim.step(case["steps"])
        return sim.get_f(np.float64 if case["fp64"] else np.float32)
    if case["run"] == "watch":
        seen = []
        for _ in range(case["looks"]):
            sim.step(case["steps"])
            seen.append(list(sim.moments().values()))
        return dict(moments=_kept(case, seen), weights=sim.get_f_device(state["out"]))
    sim.step(case["steps"])
    out = dict(weights=sim.get_f_device(state["out"]))
    if case["moments"]:
        out["moments"] = _kept(case, list(sim.moments().values()))
    if case["physics"] in ("fel", "fel_rk4"):
        out["field"] = _kept(case, sim.field_history(case["steps"]).tolist())
    return out


def work(case):
    """Weights read and written once per step, and once each for the initial and the final ones; the
    diagnostics read them once more. Operations per node and step: the taps of the deposit, their weights, the
    push and, for the Galerkin projection, the two solves."""
    if case["run"] in ("batch", "serve"):
        members = [(n * n, steps, 4, ph) for ph, n, steps in _members(case)]
        looks, taps, solve = 0, 16, 20
    else:
        looks = case.get("looks", 1 if case.get("moments") else 0)
        n = case["nx"] * case["np"]
        members = [(n, case["steps"] * max(1, case.get("looks", 1)), 8 if case["fp64"] else 4, case["physics"])]
        taps = 4 if case["basis"] == "tent" else 16
        solve = 20 if taps == 16 and not case["lumped"] else 0
    nbytes = flops = 0.0
    for n, steps, sz, ph in members:
        nbytes += n * sz * (2.0 * steps + 4.0 + looks)
        push = 160 if ph == "fel_rk4" else 16   # RK4: four stages of phases and bunching
        flops += n * (steps * (2.0 * taps + 2.0 * math.sqrt(taps) * 5 + push + solve) + 25.0 * looks)
    return dict(bytes=nbytes, flops=flops)


# ------------------------------------------------------------------ the same in 64 bits, in plain torch
def _taps(t, cubic):
    if not cubic:
        return [1 - t, t]
    s = 1 - t
    return [s ** 3 / 6, 2 / 3 - t ** 2 + t ** 3 / 2, 2 / 3 - s ** 2 + s ** 3 / 2, t ** 3 / 6]


class _Exact:
    def __init__(self, physics, grid, push, f, cubic, galerkin):
        self.physics, self.grid, self.push, self.cubic, self.galerkin = physics, grid, push, cubic, galerkin
        self.w = f.double()
        self.x, self.p = _nodes(grid)
        self.hx, self.hp = (grid.x1 - grid.x0) / grid.nx, (grid.p1 - grid.p0) / (grid.np - 1)
        self.lost, self.n, self.history = 0.0, 0, []
        self.A = complex(push.a0_re, push.a0_im) if physics.startswith("fel") else 0j
        if physics == "fel":
            self.Ah = self.A + 0.5 * push.dt * self.bunching(self.x[None, :])
        if galerkin:
            k = torch.arange(grid.nx // 2 + 1, dtype=torch.float64, device="cuda")
            self.lx = 2 / 3 + torch.cos(2 * PI * k / grid.nx) / 3
            if grid.np <= 4096:
                m = torch.zeros(grid.np, grid.np, dtype=torch.float64, device="cuda")
                m.diagonal().fill_(2 / 3)
                m.diagonal(1).fill_(1 / 6)
                m.diagonal(-1).fill_(1 / 6)
                self.lp = torch.linalg.inv(m)
            else:
                self.lp = None

    def bunching(self, theta):
        c, s = (self.w * torch.cos(theta)).sum(), (self.w * torch.sin(theta)).sum()
        return complex((c / self.w.sum()).item(), (-s / self.w.sum()).item())

    def solve(self, r):
        r = torch.fft.irfft(torch.fft.rfft(r, dim=1) / self.lx, n=self.grid.nx, dim=1)
        if self.lp is not None:
            return self.lp @ r
        c, cp = 0.0, []   # elimination of tridiag(1/6, 2/3, 1/6), row by row
        for j in range(self.grid.np):
            d = 2 / 3 - c / 6
            if j:
                r[j].sub_(r[j - 1], alpha=1 / 6)
            r[j].div_(d)
            c = 1 / (6 * d)
            cp.append(c)
        for j in range(self.grid.np - 2, -1, -1):
            r[j].sub_(r[j + 1], alpha=cp[j])
        return r

    def displacement(self):
        x, p, h = self.x[None, :], self.p[:, None], self.push.dt
        if self.physics == "pendulum":
            ph = p - 0.5 * h * torch.sin(x)
            dx = h * ph
            return dx, (ph - 0.5 * h * torch.sin(x + dx)) - p
        if self.physics == "rotation":
            c, s = math.cos(h), math.sin(h)
            return x * (c - 1) + p * s, p * (c - 1) - x * s
        if self.physics == "fel":
            a = x + 0.5 * h * p
            dp = -2 * h * (self.Ah.real * torch.cos(a) - self.Ah.imag * torch.sin(a))
            return h * p + 0.5 * h * dp, dp
        th, eta, b, K = x, p, [], []
        vel, acc = [], []
        for s in range(4):
            c = (0.0, 0.5 * h, 0.5 * h, h)[s]
            if s:
                th, eta = x + c * vel[-1], p + c * acc[-1]
            b.append(self.bunching(th))
            K.append(self.A + (c * b[s - 1] if s else 0))
            vel.append(eta)
            acc.append(-2 * (K[s].real * torch.cos(th) - K[s].imag * torch.sin(th)))
        self.A = self.A + h / 6 * (b[0] + 2 * b[1] + 2 * b[2] + b[3])
        return (h / 6 * (vel[0] + 2 * vel[1] + 2 * vel[2] + vel[3]), h / 6 * (acc[0] + 2 * acc[1] + 2 * acc[2] + acc[3]))

    def step(self):
        g = self.grid
        dx, dp = self.displacement()
        out = torch.zeros(g.np * g.nx + 1, dtype=torch.float64, device="cuda")   # the last cell: weight lost
        rows = max(1, (1 << 24) // g.nx)   # in bands of rows, for the memory
        for j0 in range(0, g.np, rows):
            j1 = min(g.np, j0 + rows)
            w = self.w[j0:j1]
            u = (dx[j0:j1] if dx.shape[0] > 1 else dx) / self.hx
            v = (dp[j0:j1] if dp.shape[0] > 1 else dp) / self.hp
            u, v = u.expand_as(w), v.expand_as(w)
            fu, fv = torch.floor(u), torch.floor(v)
            wx, wy = _taps(u - fu, self.cubic), _taps(v - fv, self.cubic)
            lo = -1 if self.cubic else 0
            i0 = fu.long() + torch.arange(g.nx, device="cuda")[None, :] + lo
            k0 = fv.long() + torch.arange(j0, j1, device="cuda")[:, None] + lo
            for b in range(len(wy)):
                k = k0 + b
                wb = w * wy[b]
                inside = (k >= 0) & (k < g.np)
                for a in range(len(wx)):
                    cell = torch.where(inside, k * g.nx + torch.remainder(i0 + a, g.nx), g.np * g.nx)
                    out.index_add_(0, cell.reshape(-1), (wb * wx[a]).reshape(-1))
        self.lost += float(out[-1])
        self.w = out[:-1].view(g.np, g.nx)
        if self.galerkin:
            self.w = self.solve(self.w)
        self.n += 1
        if self.physics == "fel":
            b = self.bunching(self.x[None, :])
            self.A = self.Ah + 0.5 * self.push.dt * b
            self.Ah = self.A + 0.5 * self.push.dt * b
        self.history.append([self.A.real, self.A.imag])

    def moments(self):
        """In the order of vp_moments_t."""
        w, x, p = self.w, self.x[None, :], self.p[:, None]
        S, hh = w.sum(), self.hx * self.hp
        mean = lambda q: float((w * q).sum() / S)   # noqa: E731
        mx, mp = mean(x), mean(p)
        v = -torch.cos(x) if self.physics == "pendulum" else 0.0 * x
        H = 0.5 * p * p + v
        pos = torch.where(w > 0, w, torch.ones_like(w))
        trapped = float((w * (H < 1.0)).sum()) * hh if self.physics == "pendulum" else 0.0
        energy = mp + abs(self.A) ** 2 if self.physics == "fel" else mean(H)
        return [float(S), float(S) * hh, mx, mp, mean(x * x) - mx * mx, mean(p * p) - mp * mp, mean(x * p) - mx * mp,
                energy, trapped, float(-(pos * torch.log(pos)).sum()) * hh, float(w[w < 0].sum()) * hh,
                mean(torch.cos(x)), -mean(torch.sin(x)), float(w.abs().max()), self.lost * hh, self.A.real,
                self.A.imag, self.n * self.push.dt, float(self.n)]


def exact(case, seed):
    ends = []
    for ph, grid, push, steps, f in _inputs(case, seed):
        cubic = case.get("basis", "cubic") == "cubic"
        e = _Exact(ph, grid, push, f, cubic, cubic and not case.get("lumped", False))
        del f
        seen = []
        for _ in range(case.get("looks", 1)):
            for _ in range(steps):
                e.step()
            if case["run"] in ("watch", "serve") or case.get("moments"):
                seen.append(e.moments())
        ends.append((e.w, seen, e.history))
    wide = lambda v: torch.tensor(v, dtype=torch.float64)   # noqa: E731
    if case["run"] == "serve":
        return dict(weights=[w for w, _, _ in ends], moments=wide([m[0] for _, m, _ in ends]))
    if case["run"] == "batch":
        return [w for w, _, _ in ends]
    w, seen, history = ends[0]
    if case["run"] == "host":
        return w
    if case["run"] == "watch":
        return dict(moments=wide(seen), weights=w)
    out = dict(weights=w)
    if case["moments"]:
        out["moments"] = wide(seen[0])
    if case["physics"] in ("fel", "fel_rk4"):
        out["field"] = wide(history)
    return out
