"""Workloads of libaf that stand for what its users run, each through the public
entry points, with a plain float64 torch restatement of the scheme as the exact value.

Nine kinds of work, over the range of grids of the repository's tests and benchmark:
  step      a 2D run advanced by a few SSP-RK3 steps (af_step), the main path; with
            `monitor` also the divergence measures and the run diagnostics of the result;
  host      members of a host-resident study, one step each (af_step_host);
  ensemble  uneven runs advanced as one batch with a captured step cycle (af_batch_step);
  adjoint   a differentiable solve and its gradient (af_steps): the smooth branch
            (kappa = 0) or the recorded branch of a limited run (kappa > 0);
  step1d    a 1D run (af1d_step).

The inputs are the repository's test problems with seeded amplitudes, centres and a
small smooth perturbation, so that no symmetry line is left where the sensor of Sec. 3.4
divides rounding noise by rounding noise.
"""
import math
import random

import torch

import paper_2506_04857_gb300 as af
from paper_2506_04857_gb300.adjoint import af_steps

PERIODIC, OUTFLOW = 0, 1
DEV = "cuda"


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest run in use: the 64x64 vortex of the accuracy tests, a short time loop
        # (launches and latency count)
        {"name": "vortex-64", "what": "step", "flow": "vortex", "nx": 64, "ny": 64, "kappa": 0.0, "steps": 10,
         "monitor": False},
        # a run at the paper's size with odd extents, outflow sides and its run monitoring
        {"name": "cloud-399x401", "what": "step", "flow": "cloud", "nx": 399, "ny": 401, "kappa": 1.0, "steps": 3,
         "monitor": True},
        # the benchmark's second configuration: Orszag-Tang 512x512, periodic, sensor on
        {"name": "orszag-512", "what": "step", "flow": "orszag_tang", "nx": 512, "ny": 512, "kappa": 1.0, "steps": 3,
         "monitor": False},
        # the benchmark's default: the 2048x2048 low-beta blast, outflow, mostly quiet gas
        {"name": "blast-2048", "what": "step", "flow": "blast", "nx": 2048, "ny": 2048, "kappa": 1.0, "steps": 2,
         "monitor": False},
        # every positivity limiter and the Newton solve at work in each stage
        {"name": "lattice-1021x767", "what": "step", "flow": "lattice", "nx": 1021, "ny": 767, "kappa": 1.0,
         "steps": 1, "monitor": False},
        # the MHD jets at the paper's size: reflective and inflow sides
        {"name": "jets-200x600", "what": "step", "flow": "jets", "nx": 200, "ny": 600, "kappa": 2.0, "steps": 3,
         "monitor": False},
        # a host-resident study: members of 512x512 in pinned memory, one step each
        {"name": "host-512", "what": "host", "flow": "orszag_tang", "nx": 512, "ny": 512, "kappa": 1.0, "steps": 4},
        # a sweep of uneven Orszag-Tang runs as one batch
        {"name": "ensemble-32", "what": "ensemble", "flow": "orszag_tang", "nx": 256, "ny": 256, "kappa": 1.0,
         "steps": 3, "runs": 32},
        # gradient of a smooth solve (kappa = 0), the benchmark's adjoint workload
        {"name": "adjoint-256", "what": "adjoint", "flow": "vortex", "nx": 256, "ny": 256, "kappa": 0.0, "steps": 6,
         "every": 3},
        # gradient of a limited solve along its recorded branch
        {"name": "adjoint-limited-160x128", "what": "adjoint", "flow": "blast", "nx": 160, "ny": 128, "kappa": 1.0,
         "steps": 4, "every": 4},
        # a 1D Riemann problem at the paper's size, a short time loop
        {"name": "riemann1d-800", "what": "step1d", "flow": "riemann", "nx": 800, "kappa": 10.0, "steps": 20},
        # the 1D strong blast on a long grid
        {"name": "blast1d-4m", "what": "step1d", "flow": "blast1d", "nx": 4194304, "kappa": 1.0, "steps": 2},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above (about half of the draws are plain 2D runs)."""
    what = rng.choice(["step", "step", "step", "step", "host", "ensemble", "adjoint", "adjoint", "step1d"])
    if what == "step1d":
        n = _log_int(rng, 100, 4000000)
        return {"what": what, "flow": rng.choice(["riemann", "blast1d"]), "nx": n,
                "kappa": rng.choice([0.0, 1.0, 10.0]), "steps": 20 if n < 20000 else 2}
    if what == "ensemble":
        return {"what": what, "flow": "orszag_tang", "nx": _log_int(rng, 32, 256), "ny": _log_int(rng, 32, 256),
                "kappa": rng.choice([0.0, 1.0]), "steps": rng.choice([1, 3, 4]), "runs": rng.randint(2, 32)}
    if what == "adjoint":
        flow = rng.choice(["vortex", "blast"])
        return {"what": what, "flow": flow, "nx": _log_int(rng, 24, 256), "ny": _log_int(rng, 24, 256),
                "kappa": 0.0 if flow == "vortex" else 1.0, "steps": rng.randint(2, 5), "every": rng.randint(1, 5)}
    if what == "host":
        return {"what": what, "flow": rng.choice(["orszag_tang", "vortex"]), "nx": _log_int(rng, 48, 600),
                "ny": _log_int(rng, 48, 600), "kappa": rng.choice([0.0, 1.0]), "steps": rng.randint(2, 5)}
    flow = rng.choice(["vortex", "orszag_tang", "cloud", "blast", "lattice", "jets"])
    hi = 2000 if flow in ("blast", "vortex", "orszag_tang") else 900
    nx, ny = _log_int(rng, 24, hi), _log_int(rng, 24, hi)
    if flow == "jets":   # half as wide as it is high or less
        ny = max(ny, 2 * nx)
    return {"what": "step", "flow": flow, "nx": nx, "ny": ny,
            "kappa": 0.0 if flow == "vortex" else rng.choice([1.0, 2.0]),
            "steps": 10 if nx * ny < 20000 else (3 if nx * ny < 500000 else 1),
            "monitor": rng.random() < 0.25}


# ---------------------------------------------------------------------------
# initial states: class 0 cell averages, 1 x-faces, 2 y-faces, 3 corners, [8][ny_c][nx_c]
# ---------------------------------------------------------------------------
class Flow:
    """Grid, boundary, gas and initial primitive fields of one 2D problem."""

    def __init__(self, case, seed, member=0):
        r = random.Random("%d/%d" % (seed, member))
        self.kind = case["flow"]
        self.nx, self.ny = case["nx"], case["ny"]
        if case["what"] == "ensemble":   # uneven runs: sizes of the sweep around the case's
            s = random.Random(member)    # the sizes are the sweep's own, the same for every seed
            self.nx = max(16, int(self.nx * s.choice([0.25, 0.5, 0.75, 1.0])) + s.randint(0, 3))
            self.ny = max(16, int(self.ny * s.choice([0.25, 0.5, 0.75, 1.0])) + s.randint(0, 3))
        self.kappa, self.cfl = case["kappa"], 0.2
        self.gamma, self.bc = 5.0 / 3.0, PERIODIC
        self.x0, self.x1, self.y0, self.y1 = 0.0, 1.0, 0.0, 1.0
        self.sides, self.inflow = (0, 0, 0, 0), None
        self.modes = [[(r.randint(-3, 3), r.randint(1, 3), r.uniform(0.5, 1.0), r.uniform(0, 2 * math.pi))
                       for _ in range(3)] for _ in range(6)]
        self.c = (r.uniform(-0.05, 0.05), r.uniform(-0.05, 0.05))
        self.a = (r.uniform(0.8, 1.2), r.uniform(0.8, 1.2), r.uniform(0, 2 * math.pi), r.uniform(0, 2 * math.pi))
        if self.kind == "vortex":
            self.x0, self.x1, self.y0, self.y1 = -5.0, 5.0, -5.0, 5.0
        elif self.kind == "orszag_tang":
            self.x1 = self.y1 = 2.0 * math.pi
        elif self.kind == "blast":
            self.gamma, self.bc = 1.4, OUTFLOW
            self.x0, self.x1, self.y0, self.y1 = -0.5, 0.5, -0.5, 0.5
        elif self.kind == "cloud":
            self.bc = OUTFLOW
        elif self.kind == "lattice":
            self.gamma = 1.4
        else:   # jets: the left half, reflective at its right side, the jet entering at the bottom
            self.gamma, self.bc = 1.4, OUTFLOW
            self.x0, self.x1, self.y1 = -0.5, 0.0, 1.5
            self.sides = (0, 1, 2, 0)
            self.ba = math.sqrt(20000.0) * self.a[0]
            one = torch.ones(1, 1, dtype=torch.float64)
            u = conserved((self.gamma * one, 0 * one, 800.0 * one, 0 * one, 0 * one, self.ba * one, 0 * one, one),
                          self.gamma)
            self.inflow = (-0.05, 0.05, [float(v) for v in u[:, 0, 0]])

    @property
    def dx(self):
        return (self.x1 - self.x0) / self.nx

    @property
    def dy(self):
        return (self.y1 - self.y0) / self.ny

    def noise(self, k, x, y):
        s, t = (x - self.x0) / (self.x1 - self.x0), (y - self.y0) / (self.y1 - self.y0)
        return sum(a * torch.cos(2 * math.pi * (p * s + q * t) + ph) for p, q, a, ph in self.modes[k])

    def prim(self, x, y):
        """(rho, v1, v2, v3, B1, B2, B3, p) at x [1, n], y [m, 1]."""
        z = torch.zeros_like(x + y)
        n = [self.noise(k, x, y) for k in range(6)]
        av, ab, px, py = self.a
        if self.kind == "vortex":
            xs, ys = x - self.c[0], y - self.c[1]
            r2 = xs * xs + ys * ys
            e = torch.exp(0.5 * (1.0 - r2)) / (2.0 * math.pi)
            p = 1.0 - r2 * torch.exp(1.0 - r2) / (8.0 * math.pi ** 2)
            return (1.0 + 1e-2 * n[0], 1.0 - e * ys + 1e-2 * n[1], 1.0 + e * xs + 1e-2 * n[2], 1e-2 * n[3],
                    -e * ys + 1e-2 * n[4], e * xs + 1e-2 * n[5], 1e-2 * n[0], p + z)
        if self.kind == "orszag_tang":
            xp, yp = x + px, y + py
            return (self.gamma ** 2 + 1e-2 * n[0], -av * torch.sin(yp) + 1e-2 * n[1], av * torch.sin(xp) + 1e-2 * n[2],
                    1e-2 * n[3], -ab * torch.sin(yp) + 1e-2 * n[4], ab * torch.sin(2.0 * xp) + 1e-2 * n[5], z,
                    self.gamma + z)
        if self.kind == "blast":   # gas at rest away from the blast
            b = 100.0 / math.sqrt(8.0 * math.pi)
            xs, ys = x - self.c[0], y - self.c[1]
            r2 = xs * xs + ys * ys
            w = 0.05 * torch.clamp(1.0 - r2 / 0.05, min=0.0) ** 3
            return (1.0 + w * n[0], w * n[1], w * n[2], w * n[3], b + w * n[4], b + w * n[5], w * n[0],
                    torch.where(r2 < 0.01, z + 1000.0 * av, z + 0.1))
        if self.kind == "cloud":
            left = (x < 0.6) & (z == 0)
            cloud = (x - 0.8 - self.c[0]) ** 2 + (y - 0.5 - self.c[1]) ** 2 < 0.15 ** 2
            rho = torch.where(left, z + 3.86859, torch.where(cloud, z + 10.0, z + 1.0))
            return (rho, torch.where(left, z, z - 11.2536) + 1e-2 * n[1], 1e-2 * n[2], 1e-2 * n[3], 1e-3 * n[4],
                    torch.where(left, z + 2.1826182, z + 0.56418958), torch.where(left, z - 2.1826182, z + 0.56418958),
                    torch.where(left, z + 167.345, z + 1.0))
        if self.kind == "lattice":   # cells of 32 grid points: rarefactions towards vacuum, colliding streams
            m1, m2 = max(1, self.nx // 32), max(1, self.ny // 32)
            v1 = torch.where(torch.sin(2.0 * math.pi * m1 * x + px) < 0, z - 6.0, z + 6.0)
            v2 = torch.where(torch.sin(2.0 * math.pi * m2 * y + py) < 0, z - 6.0, z + 6.0)
            return (1.0 + 1e-2 * n[0], v1 * av + 0.1 * n[1], v2 * av + 0.1 * n[2], 0.1 * n[3], 1e-2 * n[4],
                    0.5 + 1e-2 * n[5], 1e-2 * n[0], z + 0.4)
        return (0.1 * self.gamma * (1.0 + 1e-2 * n[0]), 0.1 * n[1], 0.1 * n[2], 0.1 * n[3], 0.1 * n[4],
                self.ba + 0.1 * n[5], z, z + 1.0)

    def state(self):
        """Point values exactly; cell averages by Simpson's rule on the cell's nodes."""
        nx, ny, o = self.nx, self.ny, 1
        ar = lambda n, s: torch.arange(n, dtype=torch.float64, device=DEV) + s  # noqa: E731
        xc, xf = self.x0 + ar(nx, 0.5) * self.dx, self.x0 + ar(nx + o, 0.0) * self.dx
        yc, yf = self.y0 + ar(ny, 0.5) * self.dy, self.y0 + ar(ny + o, 0.0) * self.dy
        at = lambda xs, ys: conserved(self.prim(xs[None, :], ys[:, None]), self.gamma)  # noqa: E731
        Z, X, Y, C = at(xc, yc), at(xf, yc), at(xc, yf), at(xf, yf)
        if self.bc == PERIODIC:   # the last point is the first one
            X[:, :, nx], Y[:, ny, :] = X[:, :, 0], Y[:, 0, :]
            C[:, :, nx] = C[:, :, 0]
            C[:, ny, :] = C[:, 0, :]
        A = (16.0 * Z + 4.0 * (X[:, :, :-1] + X[:, :, 1:] + Y[:, :-1] + Y[:, 1:])
             + (C[:, :-1, :-1] + C[:, :-1, 1:] + C[:, 1:, :-1] + C[:, 1:, 1:])) / 36.0
        if self.bc == PERIODIC:
            X, Y, C = X[:, :, :nx], Y[:, :ny], C[:, :ny, :nx]
        return [t.contiguous() for t in (A, X, Y, C)]

    def solver(self, stream=None):
        return af.Solver(self.nx, self.ny, self.gamma, self.bc, domain=(self.x0, self.x1, self.y0, self.y1),
                         cfl=self.cfl, kappa=self.kappa, stream=stream, sides=self.sides, inflow=self.inflow)


class Flow1D:
    def __init__(self, case, seed):
        r = random.Random(seed)
        self.n, self.kappa, self.cfl = case["nx"], case["kappa"], 0.2
        self.riemann = case["flow"] == "riemann"
        self.gamma = 2.0 if self.riemann else 1.4
        self.x0, self.x1 = (0.0, 1.0) if self.riemann else (-0.5, 0.5)
        self.dx = (self.x1 - self.x0) / self.n
        self.a = [r.uniform(0.8, 1.2) for _ in range(4)]
        self.ph = [r.uniform(0, 2 * math.pi) for _ in range(4)]

    def prim(self, x):
        z = torch.zeros_like(x)
        w = [1e-2 * torch.sin(2 * math.pi * x + p) for p in self.ph]
        if self.riemann:
            left = x < 0.5
            pick = lambda a, b: torch.where(left, z + a, z + b)  # noqa: E731
            return (pick(1.0, 0.125 * self.a[0]), w[0], w[1], w[2], z + 0.75, pick(1.0, -self.a[1]), w[3],
                    pick(1.0, 0.1))
        b = 100.0 / math.sqrt(8.0 * math.pi)
        w = [v * torch.clamp(1.0 - (x / 0.2) ** 2, min=0.0) ** 3 for v in w]
        return (1.0 + w[0], w[1], w[2], z, z + b, b + w[3], z,
                torch.where(x.abs() < 0.1, z + 1000.0 * self.a[0], z + 0.1))

    def state(self):
        f = self.x0 + torch.arange(self.n + 1, dtype=torch.float64, device=DEV) * self.dx
        P = conserved(self.prim(f), self.gamma)
        Z = conserved(self.prim(f[:-1] + 0.5 * self.dx), self.gamma)
        return [((4.0 * Z + P[:, :-1] + P[:, 1:]) / 6.0).contiguous(), P.contiguous()]

    def solver(self):
        return af.Solver1D(self.n, self.gamma, OUTFLOW, domain=(self.x0, self.x1), cfl=self.cfl, kappa=self.kappa)


def conserved(w, gamma):
    rho, v1, v2, v3, b1, b2, b3, p = torch.broadcast_tensors(*w)
    return torch.stack([rho, rho * v1, rho * v2, rho * v3, b1, b2, b3,
                        p / (gamma - 1.0) + 0.5 * rho * (v1 * v1 + v2 * v2 + v3 * v3)
                        + 0.5 * (b1 * b1 + b2 * b2 + b3 * b3)])


# ---------------------------------------------------------------------------
# what a user's program has in hand, and one pass
# ---------------------------------------------------------------------------
def _cotangents(shapes, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed + 7)
    return [torch.randn(s, generator=g, dtype=torch.float64, device=DEV) for s in shapes]


def prepare(case, seed):
    what = case["what"]
    if what == "step1d":
        f = Flow1D(case, seed)
        U = f.state()
        return {"case": case, "solver": f.solver(), "U": U, "out": [torch.empty_like(u) for u in U]}
    if what == "ensemble":
        flows = [Flow(case, seed, m) for m in range(case["runs"])]
        stream = torch.cuda.Stream()
        b = af.af_batch_create([f.nx for f in flows], [f.ny for f in flows], [f.gamma for f in flows],
                               [f.bc for f in flows])
        af.af_batch_set_stream(b, stream)
        for m, f in enumerate(flows):
            af.af_batch_set_domain(b, m, f.x0, f.x1, f.y0, f.y1)
            af.af_batch_set_params(b, m, cfl=f.cfl, kappa=f.kappa)
        U = [f.state() for f in flows]
        flat = [torch.empty(sum(u.numel() for u in s), dtype=torch.float64, device=DEV) for s in U]
        out = []
        for s, t in zip(U, flat):
            parts = torch.split(t, [u.numel() for u in s])
            out.append([p.view(u.shape) for p, u in zip(parts, s)])
        torch.cuda.synchronize()
        af.af_batch_graph(b, True)
        return {"case": case, "batch": Batch(b), "stream": stream, "U": U, "flat": flat, "out": out}
    if what == "host":
        flows = [Flow(case, seed, m) for m in range(case["steps"])]
        U = [[torch.empty(u.shape, dtype=u.dtype, pin_memory=True).copy_(u) for u in f.state()] for f in flows]
        out = [[torch.empty(u.shape, dtype=u.dtype, pin_memory=True) for u in s] for s in U]
        return {"case": case, "solver": flows[0].solver(), "U": U, "out": out}
    f = Flow(case, seed)
    U = f.state()
    if what == "adjoint":
        return {"case": case, "solver": f.solver(), "U": [u.requires_grad_(True) for u in U],
                "lam": _cotangents([u.shape for u in U], seed)}
    s = {"case": case, "solver": f.solver(), "U": U, "out": [torch.empty_like(u) for u in U]}
    if case["monitor"]:
        s["divb"] = torch.empty(2, dtype=torch.float64, device=DEV)
        s["diag"] = torch.empty(9, dtype=torch.float64, device=DEV)
    return s


class Batch:
    """Owns a batch handle."""

    def __init__(self, handle):
        self.handle = handle

    def __del__(self):
        af.af_batch_destroy(self.handle)


def run(state):
    case, what = state["case"], state["case"]["what"]
    if what == "ensemble":
        b, stream = state["batch"].handle, state["stream"]
        stream.wait_stream(torch.cuda.current_stream())
        for m, U in enumerate(state["U"]):
            af.af_batch_set_state(b, m, U)
        af.af_batch_step(b, case["steps"])
        for m, out in enumerate(state["out"]):
            af.af_batch_get_state(b, m, out)
        torch.cuda.current_stream().wait_stream(stream)
        return state["flat"]
    s = state["solver"]
    if what == "host":
        for U, out in zip(state["U"], state["out"]):
            s.step_host(U, out)
        s.sync()   # the results are read on the host
        return state["out"]
    if what == "adjoint":
        out = af_steps(s, state["U"], case["steps"], checkpoint_every=case["every"])
        grads = torch.autograd.grad(out, state["U"], grad_outputs=state["lam"])
        return {"state": [o.detach() for o in out], "gradient": list(grads)}
    s.set_state(state["U"])
    for _ in range(case["steps"]):
        s.step(False)
    s.get_state(state["out"])
    if what == "step" and case["monitor"]:
        s.divb(state["divb"])
        s.diagnostics(state["diag"])
        return {"state": state["out"], "divb": state["divb"], "diagnostics": state["diag"]}
    return state["out"]


# ---------------------------------------------------------------------------
# work: the scheme's own traffic and arithmetic (unlimited operators, literal count)
# ---------------------------------------------------------------------------
def work(case):
    what = case["what"]
    # bytes per cell and step: each stage reads U^(s) (and U^n in stages 2 and 3) and writes its result
    if what == "step1d":
        n = case["nx"] * case["steps"]
        return {"bytes": 8 * 128.0 * n, "flops": 3 * 970.0 * n}
    if what == "ensemble":
        cells = sum(f.nx * f.ny for f in (Flow(case, 0, m) for m in range(case["runs"])))
    else:
        cells = case["nx"] * case["ny"]
    n = cells * case["steps"]
    by, fl = 8 * 256.0 * n, 3 * (2900.0 if case["kappa"] else 2700.0) * n
    if what == "host":
        by += 2 * 256.0 * n          # the copies in and out
    if what == "adjoint":            # forward, recomputation and three transposed stages of about twice the work
        by, fl = 4 * by, 4 * fl
    if case.get("monitor"):
        by, fl = by + 2 * 256.0 * cells, fl + 500.0 * cells
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------------------
# exact: the scheme in plain float64 torch
# ---------------------------------------------------------------------------
FLIP_X, FLIP_Y = (1, 4), (2, 5)   # momentum and field components normal to a reflective side


def _safe_sqrt(x):
    """sqrt with derivative 0 at 0."""
    pos = x > 0
    return torch.where(pos, torch.sqrt(torch.where(pos, x, torch.ones_like(x))), torch.zeros_like(x))


def _pressure(U, gm1):
    return gm1 * (U[7] - 0.5 * (U[1] ** 2 + U[2] ** 2 + U[3] ** 2) / U[0] - 0.5 * (U[4] ** 2 + U[5] ** 2 + U[6] ** 2))


class Data:
    """Pointwise quantities of an array of states."""

    def __init__(self, U, gamma):
        self.U = U
        rho = U[0]
        v = self.v = U[1:4] / rho
        B = self.B = U[4:7]
        BB = (B * B).sum(0)
        p = (gamma - 1.0) * (U[7] - 0.5 * (U[1:4] * v).sum(0) - 0.5 * BB)
        self.pt = p + 0.5 * BB
        self.vB = (v * B).sum(0)
        self.F = []
        for l in range(2):
            m = U[1 + l]
            f = [m] + [m * v[k] - B[l] * B[k] + (self.pt if k == l else 0.0) for k in range(3)]
            f += [v[l] * B[k] - B[l] * v[k] for k in range(3)]
            f.append((U[7] + self.pt) * v[l] - B[l] * self.vB)
            self.F.append(torch.stack(f))
        c2 = gamma * p / rho
        a = c2 + BB / rho
        self.cf = [_safe_sqrt(0.5 * (a + _safe_sqrt(a * a - 4.0 * c2 * B[l] ** 2 / rho))) for l in range(2)]
        self.sr = [v[l].abs() + self.cf[l] for l in range(2)]
        self.srho = torch.sqrt(rho)
        self.psi = torch.cat([torch.zeros_like(U[:1]), B, v, self.vB[None]])

    def part(self, ys, xs):
        """The same quantities on a window."""
        d = object.__new__(Data)
        for k in ("U", "v", "B", "psi"):
            setattr(d, k, getattr(self, k)[:, ys, xs])
        for k in ("pt", "vB", "srho"):
            setattr(d, k, getattr(self, k)[ys, xs])
        d.F = [f[:, ys, xs] for f in self.F]
        d.cf = [f[ys, xs] for f in self.cf]
        d.sr = [f[ys, xs] for f in self.sr]
        return d


def _llf(a, b, l):
    """LLF flux of eq. (2d_llf_flux) with alpha of Lemma 3.1, and alpha."""
    nB = _safe_sqrt(((a.B - b.B) ** 2).sum(0))
    al = torch.maximum(a.v[l].abs(), b.v[l].abs()) + torch.maximum(a.cf[l], b.cf[l]) + nB / (a.srho + b.srho)
    return 0.5 * (a.F[l] + b.F[l] - al * (b.U - a.U))


def _scaling(UH, UL, gm1):
    """Sec. 3.3 scaling limiter and the round-off shrink of Remark 4.1 (coefficients held fixed under autograd)."""
    with torch.no_grad():
        rL, pL = UL[0], _pressure(UL, gm1)
        er, ep = rL.clamp(max=1e-13), pL.clamp(max=1e-13)
        t1 = torch.where(UH[0] < er, (rL - er) / (rL - UH[0]), torch.ones_like(rL))
        Us = torch.cat([(t1 * UH[0] + (1 - t1) * rL)[None], UH[1:]])
        ps = _pressure(Us, gm1)
        t2 = torch.where(ps < ep, (pL - ep) / (pL - ps), torch.ones_like(rL))
        t0 = t2.clone()
        for m in range(11):
            out = t2 * Us + (1 - t2) * UL
            bad = ~((out[0] > 0) & (_pressure(out, gm1) > 0))
            if not bool(bad.any()):
                break
            t2 = torch.where(bad, (t0 - 1e-8 * 2 ** m).clamp(min=0.0) if m < 10 else torch.zeros_like(t2), t2)
    high = torch.cat([(t1 * UH[0] + (1 - t1) * UL[0])[None], UH[1:]])
    return torch.where((t1 < 1) | (t2 < 1), t2 * high + (1 - t2) * UL, UH)


class Scheme:
    """One stage of the limited scheme on one grid (ny = 1 rows of cells are not special)."""

    def __init__(self, f):
        self.f, self.g, self.gm1 = f, f.gamma, f.gamma - 1.0
        self.nx, self.ny, self.dx, self.dy = f.nx, f.ny, f.dx, f.dy

    def index(self, cls, axis):
        """Interior index of each extended index -2 .. n + 1 (+ 1 for points), and the ghost masks."""
        n = self.nx if axis == 0 else self.ny
        face = cls in ((1, 3) if axis == 0 else (2, 3))
        i = torch.arange(-2, n + 2 + int(face), device=DEV)
        lo, hi = i < 0, i >= n + int(face)
        if self.f.bc == PERIODIC:
            return i % n, torch.zeros_like(lo), torch.zeros_like(hi)
        if face:
            return torch.where(lo, -i, torch.where(hi, 2 * n - i, i)), lo, hi
        return torch.where(lo, -1 - i, torch.where(hi, 2 * n - 1 - i, i)), lo, hi

    def extend(self, U, cls):
        f = self.f
        ix, xl, xh = self.index(cls, 0)
        iy, yl, yh = self.index(cls, 1)
        E = U[:, iy][:, :, ix]
        if any(f.sides):
            for side, m, comps, ax in ((0, xl, FLIP_X, 0), (1, xh, FLIP_X, 0), (2, yl, FLIP_Y, 1), (3, yh, FLIP_Y, 1)):
                if f.sides[side] == 1:
                    sg = torch.where(m, -1.0, 1.0).to(E.dtype)
                    s8 = torch.ones(8, 1, 1, dtype=E.dtype, device=E.device)
                    w = (sg[None, :] if ax == 0 else sg[:, None])
                    E = torch.stack([E[k] * w if k in comps else E[k] for k in range(8)]) * s8
                elif f.sides[side] == 2:
                    lo, hi, u = f.inflow
                    x = f.x0 + (ix.double() + (0.0 if cls in (1, 3) else 0.5)) * f.dx
                    w = m[:, None] & ((x > lo) & (x < hi))[None, :]
                    E = torch.where(w, torch.tensor(u, dtype=E.dtype, device=E.device)[:, None, None], E)
        return E

    @staticmethod
    def win(D, i0, j0, nx, ny):
        """Window of extended data starting at interior index (i0, j0)."""
        return D.part(slice(2 + j0, 2 + j0 + ny), slice(2 + i0, 2 + i0 + nx))

    def fvs(self, P, l, h):
        """(D+ F+ + D- F-) and the central derivative of B_l along the 5-point line P (Sec. 2.3)."""
        al = P[0].sr[l]
        for q in P[1:]:
            al = torch.maximum(al, q.sr[l])
        plus = [0.5 * (q.F[l] + al * q.U) for q in P[:3]]
        minus = [0.5 * (q.F[l] - al * q.U) for q in P[2:]]
        dF = (plus[0] - 4 * plus[1] + 3 * plus[2]) / h + (-3 * minus[0] + 4 * minus[1] - minus[2]) / h
        dB = (P[0].B[l] - 4 * P[1].B[l] + 4 * P[3].B[l] - P[4].B[l]) / (2 * h)
        return dF, dB

    def centre(self, U):
        X, Y, C = [self.extend(U[c], c) for c in (1, 2, 3)]
        nx, ny = self.nx, self.ny
        w = lambda E, i, j: E[:, 2 + j:2 + j + ny, 2 + i:2 + i + nx]  # noqa: E731
        Z = 2.25 * U[0] - 0.25 * (w(X, 0, 0) + w(X, 1, 0) + w(Y, 0, 0) + w(Y, 0, 1)) \
            - (w(C, 0, 0) + w(C, 1, 0) + w(C, 0, 1) + w(C, 1, 1)) / 16.0
        return _scaling(Z, U[0], self.gm1)

    def dt(self, U):
        D = [Data(u, self.g) for u in U]
        m = [max(float(d.sr[l].max()) for d in D) for l in range(2)]
        return self.f.cfl / (m[0] / self.dx + m[1] / self.dy)

    def phi(self, A):
        """Sensor values of Sec. 3.4 on the cells -1 .. n."""
        s = lambda q, i, j: q[..., 1 + j:q.shape[-2] - 1 + j, 1 + i:q.shape[-1] - 1 + i]  # noqa: E731
        p, v, B = A.pt, A.v, A.B
        out = []
        for i, j in ((1, 0), (0, 1)):
            a, b = s(p, i, j), s(p, -i, -j)
            out.append((a - 2 * s(p, 0, 0) + b).abs() / (a + 2 * s(p, 0, 0) + b).abs())
        div = (s(v[0], 1, 0) - s(v[0], -1, 0)) / (2 * self.dx) + (s(v[1], 0, 1) - s(v[1], 0, -1)) / (2 * self.dy)
        curl = (s(v[1], 1, 0) - s(v[1], -1, 0)) / (2 * self.dx) - (s(v[0], 0, 1) - s(v[0], 0, -1)) / (2 * self.dy)
        out.append((-div / torch.sqrt(div ** 2 + curl ** 2 + 1e-40)).clamp(min=0.0))
        dB = s(B[0], 1, 0) - s(B[0], -1, 0) + s(B[1], 0, 1) - s(B[1], 0, -1)
        out.append(dB.abs() / ((s(B[0], 0, 0) + s(B[1], 0, 0)).abs() + 1e-40))
        return out

    def stage(self, Un, Us, dt, a, b):
        """a U^n + b FE(U^s)."""
        f, g, gm1, nx, ny, dx, dy = self.f, self.g, self.gm1, self.nx, self.ny, self.dx, self.dy
        Z = self.centre(Us)
        D = [Data(self.extend(u, c), g) for c, u in enumerate(Us)] + [Data(self.extend(Z, 4), g)]
        fx, fy = (nx, ny) if f.bc == PERIODIC else (nx + 1, ny + 1)
        w = self.win
        out = [None] * 4
        for cls, mx, my in ((1, fx, ny), (2, nx, fy), (3, fx, fy)):
            at = lambda c, i, j: w(D[c], i, j, mx, my)  # noqa: E731
            me = at(cls, 0, 0)
            if cls == 2:
                lo, hi = at(3, 0, 0), at(3, 1, 0)
                Lx, Bx = (hi.F[0] - lo.F[0]) / dx, (hi.B[0] - lo.B[0]) / dx
            else:
                mid = 2 if cls == 3 else 4
                Lx, Bx = self.fvs([at(cls, -1, 0), at(mid, -1, 0), me, at(mid, 0, 0), at(cls, 1, 0)], 0, dx)
            if cls == 1:
                lo, hi = at(3, 0, 0), at(3, 0, 1)
                Ly, By = (hi.F[1] - lo.F[1]) / dy, (hi.B[1] - lo.B[1]) / dy
            else:
                mid = 1 if cls == 3 else 4
                Ly, By = self.fvs([at(cls, 0, -1), at(mid, 0, -1), me, at(mid, 0, 0), at(cls, 0, 1)], 1, dy)
            UH = me.U - dt * (Lx + Ly + (Bx + By) * me.psi)
            if cls == 2:
                n = [at(3, 0, 0), at(3, 1, 0)]
            else:
                n = [at(cls, -1, 0), at(cls, 1, 0)]
            n += [at(3, 0, 0), at(3, 0, 1)] if cls == 1 else [at(cls, 0, -1), at(cls, 0, 1)]
            div = (n[1].B[0] - n[0].B[0]) / (2 * dx) + (n[3].B[1] - n[2].B[1]) / (2 * dy)
            UL = me.U - dt * ((_llf(me, n[1], 0) - _llf(n[0], me, 0)) / dx + (_llf(me, n[3], 1) - _llf(n[2], me, 1)) / dy
                              + div * me.psi)
            out[cls] = _scaling(UH, UL, gm1)
        # faces 0 .. n in each direction: sensor, Simpson flux, LLF flux
        if f.kappa:
            with torch.no_grad():
                ph = self.phi(w(D[0], -2, -2, nx + 4, ny + 4))
                tx = [torch.maximum(q[1:-1, :-1], q[1:-1, 1:]) for q in ph]
                ty = [torch.maximum(q[:-1, 1:-1], q[1:, 1:-1]) for q in ph]
                ts = [torch.exp(-f.kappa * (tx[0] * tx[2] + tx[3])), torch.exp(-f.kappa * (ty[1] * ty[2] + ty[3]))]
        else:
            one = torch.ones(1, dtype=Z.dtype, device=Z.device)
            ts = [one.expand(ny, nx + 1), one.expand(ny + 1, nx)]
        LLF = [_llf(w(D[0], -1, 0, nx + 1, ny), w(D[0], 0, 0, nx + 1, ny), 0),
               _llf(w(D[0], 0, -1, nx, ny + 1), w(D[0], 0, 0, nx, ny + 1), 1)]
        HO = [(w(D[3], 0, 0, nx + 1, ny).F[0] + 4 * w(D[1], 0, 0, nx + 1, ny).F[0] + w(D[3], 0, 1, nx + 1, ny).F[0]) / 6,
              (w(D[3], 0, 0, nx, ny + 1).F[1] + 4 * w(D[2], 0, 0, nx, ny + 1).F[1] + w(D[3], 1, 0, nx, ny + 1).F[1]) / 6]
        G = [ts[l] * (HO[l] - LLF[l]) for l in range(2)]
        # cell sources on the 3x3 Simpson nodes, eq. (semi_av_src)
        nd = [[w(D[c], i, j, nx, ny) for i, c in ((0, c0), (0, c1), (1, c0))]
              for j, c0, c1 in ((0, 3, 2), (0, 1, 4), (1, 3, 2))]
        wt, d1 = (1 / 6, 2 / 3, 1 / 6), ((-3, 4, -1), (-1, 0, 1), (1, -4, 3))
        S = 0.0
        for m in range(3):
            for l in range(3):
                div = sum(d1[l][t] * nd[m][t].B[0] for t in range(3)) / dx \
                    + sum(d1[m][t] * nd[t][l].B[1] for t in range(3)) / dy
                S = S + wt[l] * wt[m] * div * nd[m][l].psi
        me = w(D[0], 0, 0, nx, ny)
        divc = (w(D[0], 1, 0, nx, ny).B[0] - w(D[0], -1, 0, nx, ny).B[0]) / (2 * dx) \
            + (w(D[0], 0, 1, nx, ny).B[1] - w(D[0], 0, -1, nx, ny).B[1]) / (2 * dy)
        SL = divc * me.psi
        cx, cy = dt / dx, dt / dy
        Ullf = me.U - cx * (LLF[0][:, :, 1:] - LLF[0][:, :, :-1]) - cy * (LLF[1][:, 1:] - LLF[1][:, :-1]) - dt * SL
        H = [cx * G[0][:, :, :-1], -cx * G[0][:, :, 1:], cy * G[1][:, :-1], -cy * G[1][:, 1:]]
        tsc = torch.minimum(torch.minimum(ts[0][:, :-1], ts[0][:, 1:]), torch.minimum(ts[1][:-1], ts[1][1:]))
        dU = -dt * tsc * (S - SL)
        with torch.no_grad():
            ep, er = _pressure(Ullf, gm1).clamp(max=1e-13), Ullf[0].clamp(max=1e-13)
            pl, psrc = _pressure(Ullf, gm1), _pressure(Ullf + dU, gm1)
            th = torch.where(psrc < ep, ((pl - ep) / (pl - psrc)).clamp(max=1.0), torch.ones_like(pl))
        L1 = Ullf + th * dU
        with torch.no_grad():
            Lam = flux_box(L1, H, er, ep, gm1)
            tL, tR, tD, tU = face_theta(Lam, f.bc)
        fe = L1 + tL * H[0] + tR * H[1] + tD * H[2] + tU * H[3]
        out[0] = fe
        return [b * o if a == 0.0 else a * u + b * o for u, o in zip(Un, out)]

    def step(self, U):
        with torch.no_grad():
            dt = self.dt(U)
        U1 = self.stage(U, U, dt, 0.0, 1.0)
        U2 = self.stage(U, U1, dt, 0.75, 0.25)
        return self.stage(U, U2, dt, 1 / 3, 2 / 3)

    def divb(self, U):
        Z = self.centre(U)
        E = [self.extend(u, c) for c, u in enumerate(list(U) + [Z])]
        nx, ny, dx, dy = self.nx, self.ny, self.dx, self.dy
        at = lambda c, i, j, k: E[c][k, 2 + j:2 + j + ny, 2 + i:2 + i + nx]  # noqa: E731
        lay = [((0, 3), (0, 2), (1, 3)), ((0, 1), (0, 4), (1, 1)), ((0, 3), (0, 2), (1, 3))]
        B = [[[at(c, i, j, 4 + l) for i, c in row] for j, row in zip((0, 0, 1), lay)] for l in range(2)]
        wt, d1 = (1 / 6, 2 / 3, 1 / 6), ((-3, 4, -1), (-1, 0, 1), (1, -4, 3))
        s1 = 0.0
        for m in range(3):
            for l in range(3):
                div = sum(d1[l][t] * B[0][m][t] for t in range(3)) / dx + sum(d1[m][t] * B[1][t][l] for t in range(3)) / dy
                s1 = s1 + (wt[l] * wt[m] * dx * dy * div.abs()).sum()
        edge = lambda a, b, c: a + 4 * b + c  # noqa: E731
        s2 = (dy / 6 * (edge(*[B[0][m][2] for m in range(3)]) - edge(*[B[0][m][0] for m in range(3)]))
              + dx / 6 * (edge(*B[1][2]) - edge(*B[1][0]))).abs().sum()
        return torch.stack([s1, s2])

    def diagnostics(self, U):
        return torch.stack([u[0].min() for u in U] + [_pressure(u, self.gm1).min() for u in U]
                           + [self.dx * self.dy * U[0][0].sum()])


def flux_box(L1, H, er, ep, gm1):
    """Lambda_I of Sec. 3.2 step (2): the density rectangle, then the vertices below the pressure floor."""
    neg = sum(h[0].clamp(max=0.0) for h in H)
    one = torch.ones_like(er)
    LR = [torch.where(h[0] < 0, ((L1[0] - er) / (1e-12 - neg)).clamp(max=1.0), one) for h in H]
    Lam = [q.clone() for q in LR]
    for k in range(1, 2 ** len(H)):
        ks = [I for I in range(len(H)) if (k >> I) & 1]
        V = L1 + sum(LR[I] * H[I] for I in ks)
        bad = _pressure(V, gm1) < ep
        if not bool(bad.any()):
            continue
        L, D, e = L1[:, bad], (V - L1)[:, bad], ep[bad]
        c = e / gm1
        lo, hi = torch.zeros_like(e), torch.ones_like(e)
        for _ in range(54):
            r = 0.5 * (lo + hi)
            W = L + r * D
            q = W[0] * W[7] - 0.5 * (W[1:4] ** 2).sum(0) - W[0] * (0.5 * (W[4:7] ** 2).sum(0) + c)
            lo, hi = torch.where(q >= 0, r, lo), torch.where(q >= 0, hi, r)
        r = 0.5 * (lo + hi)
        for I in ks:
            Lam[I][bad] = torch.minimum(Lam[I][bad], r * LR[I][bad])
    return Lam


def face_theta(Lam, bc):
    """The face coefficients min(Lambda_R, Lambda_L) seen from each cell."""
    L, R, Dn, Up = Lam
    left, right = torch.roll(R, 1, 1), torch.roll(L, -1, 1)
    down, up = torch.roll(Up, 1, 0), torch.roll(Dn, -1, 0)
    if bc == OUTFLOW:
        left[:, 0], right[:, -1], down[0], up[-1] = L[:, 0], R[:, -1], Dn[0], Up[-1]
    return torch.minimum(L, left), torch.minimum(R, right), torch.minimum(Dn, down), torch.minimum(Up, up)


class Scheme1D:
    """The scheme on one row: averages [8, n] and points [8, n + 1], outflow, no source."""

    def __init__(self, f):
        self.f, self.g, self.gm1, self.n, self.dx = f, f.gamma, f.gamma - 1.0, f.n, f.dx

    def extend(self, U, face):
        i = torch.arange(-2, self.n + 2 + int(face), device=DEV)
        n = self.n
        i = torch.where(i < 0, -i - int(not face), torch.where(i >= n + int(face), 2 * n - int(not face) - i, i))
        return Data(U[:, None, i], self.g)

    def stage(self, Un, Us, dt, a, b):
        n, gm1, f = self.n, self.gm1, self.f
        A, P = Us
        Z = _scaling((6 * A - P[:, :-1] - P[:, 1:])[:, None] / 4, A[:, None], gm1)[:, 0]
        DA, DP, DZ = self.extend(A, False), self.extend(P, True), self.extend(Z, False)
        w = lambda D, i, m: D.part(slice(None), slice(2 + i, 2 + i + m))  # noqa: E731
        pts = [w(DP, -1, n + 1), w(DZ, -1, n + 1), w(DP, 0, n + 1), w(DZ, 0, n + 1), w(DP, 1, n + 1)]
        UH = pts[2].U - dt * Scheme.fvs(None, pts, 0, self.dx)[0]
        UL = pts[2].U - dt / self.dx * (_llf(pts[2], pts[4], 0) - _llf(pts[0], pts[2], 0))
        oP = _scaling(UH, UL, gm1)[:, 0]
        q = lambda v, i: v[0, 1 + i:v.shape[1] - 1 + i]  # noqa: E731
        ts = torch.ones(n + 1, dtype=A.dtype, device=A.device)
        if f.kappa:
            p, v, B = DA.pt, DA.v, DA.B
            p1 = (q(p, 1) - 2 * q(p, 0) + q(p, -1)).abs() / (q(p, 1) + 2 * q(p, 0) + q(p, -1)).abs()
            div, curl = [(q(v[k:k + 1, 0], 1) - q(v[k:k + 1, 0], -1)) / (2 * self.dx) for k in range(2)]
            p2 = (-div / torch.sqrt(div ** 2 + curl ** 2 + 1e-40)).clamp(min=0.0)
            b1, b2 = B[0:1, 0], B[1:2, 0]
            p3 = (q(b1, 1) - q(b1, -1)).abs() / ((q(b1, 0) + q(b2, 0)).abs() + 1e-40)
            m = [torch.maximum(t[:-1], t[1:]) for t in (p1, p2, p3)]
            ts = torch.exp(-f.kappa * (m[0] * m[1] + m[2]))
        F = _llf(w(DA, -1, n + 1), w(DA, 0, n + 1), 0)
        G = ts * (pts[2].F[0] - F)
        c = dt / self.dx
        Ul = A[:, None] - c * (F[:, :, 1:] - F[:, :, :-1])
        H = [c * G[:, :, :-1], -c * G[:, :, 1:]]
        L, R = flux_box(Ul, H, Ul[0].clamp(max=1e-13), _pressure(Ul, gm1).clamp(max=1e-13), gm1)
        left, right = torch.roll(R, 1, 1), torch.roll(L, -1, 1)
        left[:, 0], right[:, -1] = L[:, 0], R[:, -1]
        oA = (Ul + torch.minimum(L, left) * H[0] + torch.minimum(R, right) * H[1])[:, 0]
        return [b * o if a == 0.0 else a * u + b * o for u, o in zip(Un, (oA, oP))]

    def step(self, U):
        dt = self.f.cfl * self.dx / max(float(Data(u[:, None], self.g).sr[0].max()) for u in U)
        U1 = self.stage(U, U, dt, 0.0, 1.0)
        U2 = self.stage(U, U1, dt, 0.75, 0.25)
        return self.stage(U, U2, dt, 1 / 3, 2 / 3)


def _advance(scheme, U, steps):
    for _ in range(steps):
        U = scheme.step(U)
    return U


def exact(case, seed):
    what, steps = case["what"], case["steps"]
    if what == "adjoint":
        f = Flow(case, seed)
        U0 = [u.requires_grad_(True) for u in f.state()]
        out = _advance(Scheme(f), U0, steps)
        grads = torch.autograd.grad(out, U0, grad_outputs=_cotangents([u.shape for u in U0], seed))
        return {"state": [o.detach() for o in out], "gradient": list(grads)}
    with torch.no_grad():
        if what == "step1d":
            f = Flow1D(case, seed)
            return _advance(Scheme1D(f), f.state(), steps)
        if what == "ensemble":
            out = []
            for m in range(case["runs"]):
                f = Flow(case, seed, m)
                out.append(torch.cat([u.reshape(-1) for u in _advance(Scheme(f), f.state(), steps)]))
            return out
        if what == "host":
            return [_advance(Scheme(f), f.state(), 1) for f in (Flow(case, seed, m) for m in range(steps))]
        f = Flow(case, seed)
        s = Scheme(f)
        U = _advance(s, f.state(), steps)
        if case["monitor"]:
            return {"state": U, "divb": s.divb(U), "diagnostics": s.diagnostics(U)}
        return U
