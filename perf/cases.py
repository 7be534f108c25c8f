"""The work that users of this framework have it do, as cases for timing.

A case is one call as a user's program makes it through the public API: a solve (fields in, n
steps, fields out), a boundary study (a solve that samples the errors against a reference and the
conserved totals on the way), or a batch of uneven instances advanced together. The state holds
what such a program keeps between calls (the contexts and its initial fields on the device);
every pass initializes from those fields again, so that all passes do the same work.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2504_20169_gb300 import Solver
from paper_2504_20169_gb300.serving import Batch

GAMMA = 2.0                                    # (D + 2) / D in two dimensions
ORDER = {9: 2, 17: 3, 37: 4}                   # Hermite order of the equilibrium
REACH = {9: 1, 17: 3, 37: 3}                   # largest displacement: boundary layers outside F
DEGREE = {9: 5, 17: 7, 37: 9}
SHELLS = {9: ((0, 0), (1, 0), (1, 1)),
          17: ((0, 0), (1, 0), (1, 1), (2, 2), (3, 0)),
          37: ((0, 0), (1, 0), (1, 1), (2, 0), (2, 1), (2, 2), (3, 0), (3, 1))}
# floating-point operations of one node update (moments, equilibrium, relaxation)
FLOPS = {9: 120, 17: 260, 37: 628}


def solve(name, nx, ny, widths, steps, ic, bc="nrbc", edges="0100", tau=0.8, sigma=0.1, power=3,
          q=37, precision="fp32dev", grad="central", split=False, py=False, mach=0.2, samples=0):
    """One solve; samples > 0: a study that takes errors and totals that many times."""
    ww, we, ws, wn = widths
    return dict(name=name, kind="solve", nx=nx, ny=ny, ww=ww, we=we, ws=ws, wn=wn, steps=steps,
                ic=ic, bc=bc, edges=edges, tau=tau, sigma=sigma, power=power, q=q,
                precision=precision, grad=grad, split=split, py=py, mach=mach, samples=samples)


def batch(name, members, nmin, nmax, wmin, wmax, steps, pick, precision="fp32dev", grad="link"):
    """A batch; `pick` seeds the members' sizes, PML widths and boundary kinds."""
    return dict(name=name, kind="batch", members=members, nmin=nmin, nmax=nmax, wmin=wmin,
                wmax=wmax, steps=steps, pick=pick, precision=precision, grad=grad, q=37)


def listed():
    return [
        # the smallest solve (a pulse leaving a 64^2 box in a slow flow): launches and latency
        solve("pulse64_fp64", 64, 64, (8,) * 4, 100, "pulse", bc="zg", precision="fp64", mach=0.1),
        # the density-step study: 200 x 20, periodic upper and lower boundary, errors every 20 steps
        solve("step200x20_q17_fp64", 200, 20, (20, 20, 0, 0), 200, "step", edges="0000", sigma=0.08,
              power=2, q=17, precision="fp64", py=True, mach=0.05, samples=10),
        # the thermal-vortex study: 300^2, every edge open, CBC outlet, errors every 50 steps
        solve("vortex300_q17_fp64", 300, 300, (20,) * 4, 100, "vortex", sigma=0.002, power=2, q=17,
              precision="fp64", mach=0.1, samples=2),
        # the quick start's size and boundary, single precision
        solve("vortex512_fp32", 512, 512, (32,) * 4, 100, "vortex", tau=0.55, mach=0.3),
        # the benchmark's grid and parameters
        solve("vortex2048_fp32", 2048, 2048, (32,) * 4, 60, "vortex", tau=0.55, mach=0.3),
        # long runs take the stable link gradient and PNR-LODI on every edge
        solve("vortex1024_link_fp32", 1024, 1024, (32,) * 4, 60, "vortex", edges="0000", tau=0.55,
              grad="link", mach=0.3),
        # reference accuracy at a production size
        solve("vortex1024_fp64", 1024, 1024, (32,) * 4, 20, "vortex", tau=0.55, precision="fp64",
              mach=0.3),
        # the largest single grid: four pulses on 8192^2 with a 64-node PML
        solve("stress8192_fp32", 8192, 8192, (64,) * 4, 16, "pulses", tau=0.52, mach=0.2),
        # odd sizes, a PML that differs per edge, the split sigma form, zero-gradient edges
        solve("ragged_split_fp32", 1001, 613, (8, 33, 0, 17), 60, "smooth", bc="zg", sigma=0.08,
              power=2, split=True, mach=0.15),
        # a long channel: periodic y, PML and LODI on x, the 17-velocity lattice
        solve("channel_q17_fp32", 3000, 515, (24, 40, 0, 0), 60, "step", edges="0000", power=2,
              q=17, py=True, mach=0.1),
        # the 9-velocity lattice on a large box without a PML
        solve("box1500_q9_fp32", 1500, 1500, (0,) * 4, 60, "pulses", bc="zg", q=9, mach=0.05),
        # serving: uneven instances stepped together (sizes and widths of the batched sweep)
        batch("sweep16_link_fp32", 16, 128, 1024, 4, 64, 40, pick=3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another call of the same ranges: sizes over their logarithm, every lattice, precision,
    boundary, gradient and PML form."""
    if rng.random() < 0.15:
        c = batch("", rng.randint(2, 16), 64, rng.choice((256, 512, 1024)), 4, 64,
                  rng.randint(10, 40), rng.randint(10, 10 ** 6), rng.choice(("fp32dev",) * 3 + ("fp64",)),
                  rng.choice(("link", "central")))
        if c["precision"] == "fp64":
            c["nmax"] = min(c["nmax"], 512)
        del c["name"]
        return c
    q = rng.choice((37, 37, 37, 17, 9))
    fp64 = rng.random() < 0.35
    n = _log_int(rng, 64, 1200 if fp64 else 5000)
    aspect = math.exp(rng.uniform(-math.log(2.5), math.log(2.5)))
    nx, ny = max(40, int(n * math.sqrt(aspect))), max(16, int(n / math.sqrt(aspect)))
    py = rng.random() < 0.25
    bc = rng.choice(("nrbc", "nrbc", "zg"))
    form = rng.random()
    if form < 0.15:
        w = (0, 0, 0, 0)
    elif form < 0.6:
        w = (rng.randint(4, 64),) * 4
    else:
        w = tuple(rng.choice((0, rng.randint(2, 16), rng.randint(8, 64))) for _ in range(4))
    if py:
        w = (w[0], w[1], 0, 0)
    grad = rng.choice(("central", "central", "link"))
    split = grad == "central" and rng.random() < 0.3
    work_left = 6e9 if not fp64 else 1.2e8     # bytes / nodes of all steps together
    unit = nx * ny * (1 if fp64 else 2 * q * 4)
    steps = max(4, min(rng.randint(20, 100), int(work_left * 4 / unit)))
    samples = rng.choice((0, 0, 2)) if fp64 and steps >= 10 else 0   # studies run in 64 bits
    c = solve("", nx, ny, w, steps - steps % max(samples, 1),
              rng.choice(("vortex", "pulses", "smooth", "step")), bc=bc,
              edges=rng.choice(("0100", "0000")), tau=round(rng.uniform(0.55, 0.9), 3),
              sigma=round(math.exp(rng.uniform(math.log(0.01), math.log(0.1))), 4),
              power=rng.choice((2, 3)), q=q, precision="fp64" if fp64 else "fp32dev", grad=grad,
              split=split, py=py, mach=round(rng.uniform(0.05, 0.3), 3), samples=samples)
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------ inputs
def _coords(c, dev):
    y = torch.arange(c["ny"] + c["ws"] + c["wn"], dtype=torch.float64, device=dev) - c["ws"]
    x = torch.arange(c["nx"] + c["ww"] + c["we"], dtype=torch.float64, device=dev) - c["ww"]
    return x[None, :], y[:, None]


def _mean(c, rng):
    """Uniform flow of the case's Mach number, a few degrees off the x axis."""
    a = math.radians(rng.uniform(8.0, 25.0))
    return (1.0, c["mach"] * math.cos(a), c["mach"] * math.sin(a), 1.0)


def _pulse(p, x, y, cx, cy, amp, half):
    return p + amp * torch.exp(-math.log(2.0) * ((x - cx) ** 2 + (y - cy) ** 2) / half ** 2)


def _fields(c, rng, dev):
    """(mean state, four initial fields over F) of a case; centres and amplitudes from rng."""
    mean = _mean(c, rng)
    x, y = _coords(c, dev)
    nx, ny = c["nx"], c["ny"]
    one = torch.ones((y.shape[0], x.shape[1]), dtype=torch.float64, device=dev)
    ux, uy = one * mean[1], one * mean[2]
    size = min(nx, ny)

    def centre():
        return rng.uniform(0.3, 0.7) * (nx - 1), rng.uniform(0.3, 0.7) * (ny - 1)

    if c["ic"] == "vortex":                    # isentropic Gaussian vortex in the mean flow
        R, Mv = size * rng.uniform(1 / 20, 1 / 10), rng.uniform(0.03, 0.06)
        cx, cy = centre()
        e = torch.exp(1.0 - ((x - cx) ** 2 + (y - cy) ** 2) / R ** 2)
        a = Mv / R * torch.sqrt(e)
        T = 1.0 - 0.25 * Mv * Mv * e
        return mean, (T ** (1.0 / (GAMMA - 1.0)), ux - a * (y - cy), uy + a * (x - cx), T)
    if c["ic"] in ("pulse", "pulses"):         # isentropic pressure pulses
        p = one
        for _ in range(1 if c["ic"] == "pulse" else 4):
            p = _pulse(p, x, y, *centre(), rng.uniform(1e-3, 1e-2), max(3.0, size / 64.0) *
                       rng.uniform(1.0, 1.6))
        rho = p ** (1.0 / GAMMA)
        return mean, (rho, ux, uy, p / rho)
    if c["ic"] == "step":                      # tanh density plateau, its fronts wavy along y
        ph, wave = rng.uniform(0, 2 * math.pi), rng.uniform(0.01, 0.02) * nx
        shift = wave * torch.sin(2 * math.pi * y / y.shape[0] + ph)
        amp, s = rng.uniform(0.03, 0.06), 0.5
        rho = 1.0 + 0.5 * amp * (torch.tanh(s * (x - 0.25 * nx - shift)) -
                                 torch.tanh(s * (x - 0.75 * nx - shift)))
        return mean, (rho, ux, uy, one.clone())
    out = []                                   # smooth random state: a few low Fourier modes
    for amp, base in ((0.02, 1.0), (0.05, mean[1]), (0.05, mean[2]), (0.02, 1.0)):
        f = one * base
        for _ in range(4):
            kx, ky = rng.randint(1, 3), rng.randint(1, 3)
            f = f + amp / 4 * rng.uniform(-1, 1) * (
                torch.sin(2 * math.pi * kx * x / x.shape[1] + rng.uniform(0, 6.28)) *
                torch.cos(2 * math.pi * ky * y / y.shape[0] + rng.uniform(0, 6.28)))
        out.append(f)
    return mean, tuple(out)


def _references(c, rng, dev):
    """Reference fields over the bulk that a study compares with, one set per sample."""
    inner = dict(c, ww=0, we=0, ws=0, wn=0, ic="smooth")
    return [_fields(inner, rng, dev)[1] for _ in range(c["samples"])]


def _members(c):
    """The instances of a batch: sizes, PML widths, sigma and boundary kinds of the sweep."""
    rng = random.Random(c["pick"])
    out = []
    for _ in range(c["members"]):
        n, w = rng.randint(c["nmin"], c["nmax"]), rng.randint(c["wmin"], c["wmax"])
        bc = rng.choice(("zg", "nrbc"))
        vortex = rng.random() < 0.5
        out.append(solve("", n, n, (w,) * 4, c["steps"], "vortex" if vortex else "pulse", bc=bc,
                         edges="0000", sigma=math.exp(rng.uniform(math.log(0.01), math.log(0.1))),
                         precision=c["precision"], grad=c["grad"],
                         mach=rng.uniform(0.1, 0.3) if vortex else 0.1))
    return out


def _solver(c, mean):
    return Solver(c["nx"], c["ny"], 0, c["tau"], c["sigma"], c["power"], c["bc"], c["q"],
                  tuple(int(k) for k in c["edges"]), c["mach"], mean, precision=c["precision"],
                  pml_widths=(c["ww"], c["we"], c["ws"], c["wn"]), periodic_y=c["py"],
                  sigma_split=c["split"], pml_grad=c["grad"])


def _inputs(c, seed, dev):
    """(parameters, mean state, initial fields, references) of every solve in a case."""
    rng = random.Random(seed)
    out = []
    for m in (_members(c) if c["kind"] == "batch" else [c]):
        mean, fields = _fields(m, rng, dev)
        out.append((m, mean, fields, _references(m, rng, dev)))
    return out


def prepare(case, seed):
    parts = _inputs(case, seed, "cuda")
    state = {"case": case, "fields": [f for _, _, f, _ in parts], "refs": parts[0][3],
             "solvers": [_solver(m, mean) for m, mean, _, _ in parts]}
    if case["kind"] == "batch":
        for s, f in zip(state["solvers"], state["fields"]):
            s.init(*f)
        state["batch"] = Batch()
        state["batch"].set(state["solvers"])
    return state


def _result(s):
    """The fields over the bulk, in the precision of the run."""
    out = s.moments(region="bulk", device=True)
    return [t.float() for t in out] if s.precision == "fp32dev" else list(out)


def run(state):
    c = state["case"]
    for s, f in zip(state["solvers"], state["fields"]):
        s.init(*f)
    if c["kind"] == "batch":
        state["batch"].step(c["steps"])
        return [_result(s) for s in state["solvers"]]
    s = state["solvers"][0]
    if not c["samples"]:
        s.step(c["steps"])
        return _result(s)
    sampled = []
    for ref in state["refs"]:
        s.step(c["steps"] // c["samples"])
        sampled.append([s.error_sums(ref), s.reduce()])
    return [sampled, _result(s)]


def work(case):
    """Per step: every node's populations read and written once, in the PML the accumulator too,
    the boundary layers written once; per pass the fields read and written once."""
    total_b = total_f = 0.0
    for c in (_members(case) if case["kind"] == "batch" else [case]):
        q, M, b = c["q"], REACH[c["q"]], 4 if c["precision"] == "fp32dev" else 8
        Lx, Ly = c["nx"] + c["ww"] + c["we"], c["ny"] + c["ws"] + c["wn"]
        pml = Lx * Ly - c["nx"] * c["ny"]
        outside = 2 * M * (Lx + 2 * M) + 2 * M * Ly
        per_step = q * b * (2 * Lx * Ly + 2 * pml + outside)
        per_sample = 8 * 4 * c["nx"] * c["ny"] + 2 * q * b * Lx * Ly
        total_b += (c["steps"] * per_step + c["samples"] * per_sample +
                    8 * 4 * (Lx * Ly + c["nx"] * c["ny"]))
        total_f += c["steps"] * FLOPS[q] * (Lx * Ly + pml)
    return {"bytes": total_b, "flops": total_f}


# ------------------------------------------------------------------------ the same in 64 bits
def _lattice(q):
    """(velocities, weights, scale): one weight per shell and the scale r, by Newton's method on
    the Gauss-Hermite conditions of the lattice's degree."""
    e, shell = [], []
    for k, (a, b) in enumerate(SHELLS[q]):
        for v in sorted({(s * p, t * o) for p, o in ((a, b), (b, a)) for s in (1, -1)
                         for t in (1, -1)}):
            e.append(v)
            shell.append(k)
    e, shell = np.array(e), np.array(shell)
    conds = [(a, s - a) for s in range(0, DEGREE[q], 2) for a in range(s, -1, -1)
             if a % 2 == 0 and a >= s - a]

    def dfact(n):
        return float(np.prod(np.arange(n - 1, 0, -2))) if n > 1 else 1.0

    m = np.array([[np.sum(e[shell == k, 0] ** a * e[shell == k, 1] ** b)
                   for k in range(len(SHELLS[q]))] for a, b in conds], dtype=np.longdouble)
    rhs = np.array([dfact(a) * dfact(b) for a, b in conds], dtype=np.longdouble)
    deg = np.array([a + b for a, b in conds], dtype=np.longdouble)
    r = np.longdouble({9: 1.73, 17: 1.64, 37: 1.2}[q])
    w = np.linalg.lstsq((m * r ** deg[:, None]).astype(float), rhs.astype(float), rcond=None)[0]
    w = w.astype(np.longdouble)
    for _ in range(60):
        A = m * r ** deg[:, None]
        res = A @ w - rhs
        J = np.column_stack([A, deg * (A @ w) / r])
        d = np.linalg.solve(J.astype(float), res.astype(float))
        w, r = w - d[:-1], r - d[-1]
    return e, np.array(w, dtype=float)[shell], float(r)


class _Plain:
    """The scheme written out with plain tensors in 64 bits."""

    def __init__(self, c, mean, dev):
        self.c, self.M, self.order = c, REACH[c["q"]], ORDER[c["q"]]
        self.e, w, self.r = _lattice(c["q"])
        t = lambda a: torch.tensor(a, dtype=torch.float64, device=dev)  # noqa: E731
        self.ex, self.ey, self.w = t(self.e[:, 0]), t(self.e[:, 1]), t(w)
        self.Lx, self.Ly = c["nx"] + c["ww"] + c["we"], c["ny"] + c["ws"] + c["wn"]
        self.gx = torch.arange(self.Lx + 2 * self.M, device=dev) - self.M
        self.gy = torch.arange(self.Ly + 2 * self.M, device=dev) - self.M
        self.wrap_y = self.gy % self.Ly + self.M
        self.pml = c["ww"] + c["we"] + c["ws"] + c["wn"] > 0
        self.bar = self.feq(*[t(v) for v in mean])[:, None, None]

        def fraction(L, lo, hi):
            z, f = np.arange(L), np.zeros(L)
            if lo:
                f = np.maximum(f, (lo - z) / lo)
            if hi:
                f = np.maximum(f, (z - (L - 1 - hi)) / hi)
            return f

        fx = np.broadcast_to(fraction(self.Lx, c["ww"], c["we"])[None, :], (self.Ly, self.Lx))
        fy = np.broadcast_to(fraction(self.Ly, c["ws"], c["wn"])[:, None], (self.Ly, self.Lx))
        if not c["split"]:
            fx = fy = np.maximum(fx, fy)
        self.sx, self.sy = (t(np.where(f > 0, c["sigma"] * f ** c["power"], 0.0)) for f in (fx, fy))

    def feq(self, rho, ux, uy, T):
        sh = (-1,) + (1,) * rho.dim()
        ex, ey, w = self.ex.reshape(sh), self.ey.reshape(sh), self.w.reshape(sh)
        s = self.r * (ex * ux + ey * uy)
        u2, th, c2 = ux * ux + uy * uy, T - 1.0, self.r ** 2 * (ex * ex + ey * ey)
        p = 1.0 + s + 0.5 * (s * s - u2 + th * (c2 - 2.0))
        if self.order >= 3:
            p = p + s / 6.0 * (s * s - 3.0 * u2 + 3.0 * th * (c2 - 4.0))
        if self.order >= 4:
            p = p + (s ** 4 - 6.0 * s * s * u2 + 3.0 * u2 * u2 +
                     6.0 * th * (s * s * (c2 - 6.0) + u2 * (4.0 - c2)) +
                     3.0 * th * th * (c2 * c2 - 8.0 * c2 + 8.0)) / 24.0
        return w * rho * p

    def moments(self, f):
        sh = (-1,) + (1,) * (f.dim() - 1)
        ex, ey = self.ex.reshape(sh), self.ey.reshape(sh)
        rho = f.sum(0)
        ux, uy = self.r * (f * ex).sum(0) / rho, self.r * (f * ey).sum(0) / rho
        e2 = self.r ** 2 * (f * (ex * ex + ey * ey)).sum(0)
        return rho, ux, uy, 0.5 * (e2 / rho - ux * ux - uy * uy)

    def inner(self, a):
        return a[..., self.M:self.M + self.Ly, self.M:self.M + self.Lx]

    def fill(self, f):
        """The layers outside F of post-stream populations."""
        M, Lx, Ly = self.M, self.Lx, self.Ly
        f = f[:, self.gy.clamp(0, Ly - 1) + M][:, :, self.gx.clamp(0, Lx - 1) + M].clone()
        if self.c["bc"] == "nrbc":
            for k in range(2 if self.c["py"] else 4):
                line = self.line(f, k, 0)
                neq = line - self.feq(*self.moments(line))
                for j in range(1, M + 1):
                    V = self.V[k][j - 1]
                    u = (V[:, 1], V[:, 2]) if k < 2 else (V[:, 2], V[:, 1])
                    self.line(f, k, -j).copy_(self.feq(V[:, 0], *u, V[:, 3]) + neq)
        return f[:, self.wrap_y] if self.c["py"] else f

    def line(self, a, k, depth):
        """Nodes at `depth` inside edge k (W E S N; negative: outside), along the edge."""
        M, Lx, Ly = self.M, self.Lx, self.Ly
        if k == 0:
            return a[..., M:M + Ly, M + depth]
        if k == 1:
            return a[..., M:M + Ly, M + Lx - 1 - depth]
        if k == 2:
            return a[..., M + depth, M:M + Lx]
        return a[..., M + Ly - 1 - depth, M:M + Lx]

    def prim(self, U, k, depth):
        """(rho, normal velocity, tangential velocity, T) along an edge."""
        rho, ux, uy, T = (self.line(a, k, depth) for a in U)
        return torch.stack([rho, ux, uy, T] if k < 2 else [rho, uy, ux, T], -1)

    def rate(self, V, f0, f1, k):
        """Time derivative of the boundary states V [layer, node, 4] of edge k."""
        out = -1.0 if k in (0, 2) else 1.0
        full = torch.cat([f1[None], f0[None], V])
        dn = out * 0.5 * (3.0 * full[2:] - 4.0 * full[1:-1] + full[:-2]) / self.r
        rho, un, ut, T = V.unbind(-1)
        c = torch.sqrt(GAMMA * T)

        def waves(d):
            dP = T * d[..., 0] + rho * d[..., 3]
            return torch.stack([dP - rho * c * d[..., 1], T * d[..., 0] - rho * d[..., 3],
                                d[..., 2], dP + rho * c * d[..., 1]], -1)

        lam = torch.stack([un - c, un, un, un + c], -1)
        L, incoming = lam * waves(dn), lam * out < 0.0
        if self.c["edges"][k] == "0":
            w = torch.where(incoming, torch.zeros_like(L), L)
        else:
            dt = 0.5 * (torch.roll(V, -1, 1) - torch.roll(V, 1, 1))
            if not (self.c["py"] and k < 2):
                dt[:, 0] = -0.5 * (3.0 * V[:, 0] - 4.0 * V[:, 1] + V[:, 2])
                dt[:, -1] = 0.5 * (3.0 * V[:, -1] - 4.0 * V[:, -2] + V[:, -3])
            dt = dt / self.r
            B = torch.stack([ut * dt[..., 0] + rho * dt[..., 2], ut * dt[..., 1],
                             T / rho * dt[..., 0] + ut * dt[..., 2] + dt[..., 3],
                             T * dt[..., 2] + ut * dt[..., 3]], -1)
            tc = waves(B)
            w = torch.where(incoming, -(1.0 - self.c["mach"]) * tc, L) + tc
        dP = 0.5 * (w[..., 0] + w[..., 3])
        drho = (dP + w[..., 1]) / (c * c)
        return -torch.stack([drho, (w[..., 3] - w[..., 0]) / (2.0 * rho * c), w[..., 2],
                             (dP - T * drho) / rho], -1)

    def init(self, fields):
        M = self.M
        if self.c["bc"] == "nrbc":
            U = [torch.nn.functional.pad(f[None], (M,) * 4, mode="replicate")[0] for f in fields]
            self.V = [torch.stack([self.prim(U, k, 0)] * M) for k in range(4)]
        f = torch.zeros((len(self.e), self.Ly + 2 * M, self.Lx + 2 * M), dtype=torch.float64,
                        device=fields[0].device)
        self.inner(f).copy_(self.feq(*fields))
        self.f, self.Q, self.hat = self.fill(f), None, None

    def step(self):
        M, Lx, Ly, f = self.M, self.Lx, self.Ly, self.f
        U = self.moments(f)
        fe = self.feq(*U)
        star = f - (f - fe) / self.c["tau"]
        if self.pml:
            hat = fe - self.bar
            Q = torch.zeros_like(hat) if self.Q is None else self.Q + 0.5 * (self.hat + hat)
            self.Q, self.hat = Q, hat
            h, q = self.inner(hat), self.inner(Q)
            omega = (self.sx + self.sy) * h + self.sx * self.sy * q
            if self.c["grad"] == "link":
                for i, (a, b) in enumerate(self.e):
                    omega[i] += self.sx * (Q[i, M + b:M + b + Ly, M + a:M + a + Lx] - q[i])
            else:
                gx, gy = torch.empty_like(q), torch.empty_like(q)
                for g, a in ((gx, q), (gy.transpose(1, 2), q.transpose(1, 2))):
                    g[:, :, 1:-1] = 0.5 * (a[:, :, 2:] - a[:, :, :-2])
                    g[:, :, -1] = 0.5 * (3.0 * a[:, :, -1] - 4.0 * a[:, :, -2] + a[:, :, -3])
                    g[:, :, 0] = -0.5 * (3.0 * a[:, :, 0] - 4.0 * a[:, :, 1] + a[:, :, 2])
                if self.c["py"]:
                    gy = 0.5 * (torch.roll(q, -1, 1) - torch.roll(q, 1, 1))
                omega += (self.sy * self.ex[:, None, None] * gx +
                          self.sx * self.ey[:, None, None] * gy)
            self.inner(star).sub_(torch.where((self.sx + self.sy) > 0, omega,
                                              torch.zeros_like(omega)))
        if self.c["py"]:
            star = star[:, self.wrap_y]
        new = torch.empty_like(f)
        for i, (a, b) in enumerate(self.e):
            self.inner(new)[i] = star[i, M - b:M - b + Ly, M - a:M - a + Lx]
        if self.c["bc"] == "nrbc":
            for k in range(2 if self.c["py"] else 4):
                V, u0, u1 = self.V[k], self.prim(U, k, 0), self.prim(U, k, 1)
                k1 = self.rate(V, u0, u1, k)
                k2 = self.rate(V + 0.5 * k1, u0, u1, k)
                k3 = self.rate(V + 0.5 * k2, u0, u1, k)
                k4 = self.rate(V + k3, u0, u1, k)
                self.V[k] = V + (k1 + 2.0 * k2 + 2.0 * k3 + k4) / 6.0
        self.f = self.fill(new)

    def fields(self, region="bulk"):
        out = self.moments(self.inner(self.f))
        if region == "F":
            return list(out)
        c = self.c
        return [a[c["ws"]:c["ws"] + c["ny"], c["ww"]:c["ww"] + c["nx"]].contiguous() for a in out]


def exact(case, seed):
    parts = _inputs(case, seed, "cuda")
    if any(f[0].numel() * m["q"] > 2e8 for m, _, f, _ in parts):
        return None                            # minutes in this form
    got = []
    for m, mean, fields, refs in parts:
        p = _Plain(m, mean, "cuda")
        p.init(fields)
        sampled = []
        for n in range(m["steps"]):
            p.step()
            if m["samples"] and (n + 1) % (m["steps"] // m["samples"]) == 0:
                ref = refs[len(sampled)]
                sums = []
                for z, zr in zip(p.fields(), ref):
                    sums += [((z - zr) ** 2).sum(), (zr * zr).sum(), (((z - zr) / zr) ** 2).sum()]
                rho, ux, uy, T = p.fields("F")
                tot = [rho.sum(), (rho * ux).sum(), (rho * uy).sum(),
                       (0.5 * rho * (ux * ux + uy * uy + 2.0 * T)).sum(), rho.min(), T.min(),
                       torch.zeros((), dtype=torch.float64, device=rho.device)]
                sampled.append([torch.stack(sums), torch.stack(tot)])
        got.append([sampled, p.fields()] if m["samples"] else p.fields())
        del p
    return got if case["kind"] == "batch" else got[0]
