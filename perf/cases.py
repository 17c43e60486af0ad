"""Performance cases of the cRKDG library: what its users run, at the sizes they run it.

A case is a dict of plain values; `prepare` makes a user's inputs and handles on the GPU, `run` is one pass through
the public entry points (`binding.Solver`, `binding.Batch`, `binding.MLP`), `work` the bytes and operations the pass
cannot do without, and `exact` the same pass in 64 bits with plain torch (the method written out for whole meshes:
nothing of the library's arithmetic is used).  `draw` makes further cases of the listed ones' ranges.

Solvers run on two torch tensors of their caller (`state_buffers`), the way a program that keeps its fields in torch
uses the library; the outputs are those tensors.  A state's later passes continue its run.
"""
import math

import numpy as np
import torch

from paper_2307_06471_gb300 import binding as B
from paper_2307_06471_gb300 import tableaux as T
from paper_2307_06471_gb300 import workcount

GAMMA = 1.4
T_END = 1.0e6          # device-driven runs never reach it
DMR_M, PP_EPS = 50.0, 1e-10
PREC = {"f32": B.F32, "f64": B.F64, "f32d": B.F32D}
CFL = {("dmr", 2): 0.16, ("dmr", 1): 0.3, ("vortex", 2): 0.1, ("ensemble", 2): 0.16}


# ---- the cases ------------------------------------------------------------------------------------------------
def listed():
    return [
        # the double Mach reflection at the paper's finest mesh: device-driven steps with the limiters (the bench's workload)
        {"name": "dmr_1920x480_p2_f32", "kind": "dmr", "nx": 1920, "ny": 480, "k": 2, "precision": "f32", "call": "advance", "steps": 4},
        # the same flow on the paper's coarse P1 mesh with a host-driven loop (dt read back before every step): the
        # smallest call, all launches and latency
        {"name": "dmr_480x120_p1_f32_host", "kind": "dmr", "nx": 480, "ny": 120, "k": 1, "precision": "f32", "call": "host", "steps": 1},
        # the FP64 arm of the shock workload
        {"name": "dmr_640x160_p2_f64", "kind": "dmr", "nx": 640, "ny": 160, "k": 2, "precision": "f64", "call": "advance", "steps": 2},
        # convergence studies on small meshes: the vortex in FP64, graph-replayed steps
        {"name": "vortex_80_f64", "kind": "vortex", "nx": 80, "ny": 80, "precision": "f64", "call": "graph", "steps": 10},
        # FP32 at FP64 accuracy (the deviation form) on the studies' finest vortex mesh
        {"name": "vortex_320_f32d", "kind": "vortex", "nx": 320, "ny": 320, "precision": "f32d", "call": "graph", "steps": 20},
        # a smooth FP32 run that fills the GPU, on a mesh with odd sizes and cells that are not square
        {"name": "vortex_1001x613_f32", "kind": "vortex", "nx": 1001, "ny": 613, "precision": "f32", "call": "advance", "steps": 4},
        # linear advection, the largest state: one step reads and writes 1.2 GB
        {"name": "advection_4096_q2_f32", "kind": "advection", "nx": 4096, "ny": 4096, "k": 2, "basis": "Q", "precision": "f32", "steps": 1},
        # the boundary-order study: Q3, RK4, FP64, time-dependent inflow data at the stage times, one step at a time
        {"name": "inflow_80_q3_f64", "kind": "inflow", "nx": 80, "ny": 80, "k": 3, "steps": 8},
        # the 1D study: a fixed-dt run on 160 cells
        {"name": "line_160_p2_f64", "kind": "line", "physics": "advection", "nx": 160, "k": 2, "precision": "f64", "steps": 160},
        # an ensemble of uneven problems advanced together to a snapshot, then read back
        {"name": "ensemble_12_f32", "kind": "ensemble", "problems": 12, "largest": 256, "precision": "f32", "steps": 40},
        # one epoch of the learned indicator's training (minibatches of 1024, the last one ragged)
        {"name": "train_8000", "kind": "train", "samples": 8000, "batch": 1024},
        # evaluating the indicator on a state: features and labels of every cell, then the network's logits
        {"name": "indicator_1024x512_f32", "kind": "indicator", "nx": 1024, "ny": 512, "precision": "f32"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ones' ranges (no drawn case is larger than the largest listed one)."""
    kind = rng.choice(["dmr", "dmr", "vortex", "vortex", "advection", "inflow", "line", "ensemble", "train", "indicator"])
    if kind == "dmr":
        precision = rng.choice(["f32", "f32", "f64"])
        ny = _log_int(rng, 24, 480 if precision == "f32" else 160)
        call = rng.choice(["advance", "host"])
        return {"kind": kind, "nx": 4 * ny + rng.randint(-3, 3), "ny": ny, "k": rng.choice([1, 2]), "precision": precision,
                "call": call, "steps": rng.randint(1, 4) if precision == "f32" else rng.randint(1, 2)}
    if kind == "vortex":
        precision = rng.choice(["f32", "f32d", "f64"])
        hi = {"f32": 1000, "f32d": 640, "f64": 320}[precision]
        nx = _log_int(rng, 40, hi)
        ny = nx if rng.random() < 0.5 else max(24, int(nx * rng.uniform(0.5, 1.0)))
        return {"kind": kind, "nx": nx, "ny": ny, "precision": precision, "call": rng.choice(["advance", "graph"]),
                "steps": rng.randint(1, 6)}
    if kind == "advection":
        nx = _log_int(rng, 64, 4096)
        return {"kind": kind, "nx": nx, "ny": max(32, int(nx * rng.uniform(0.4, 1.0))), "k": rng.choice([1, 2, 3]),
                "basis": rng.choice(["P", "Q"]) if nx < 3000 else "P", "precision": rng.choice(["f32", "f64"]) if nx < 2000 else "f32",
                "steps": rng.randint(1, 3)}
    if kind == "inflow":
        return {"kind": kind, "nx": _log_int(rng, 10, 160), "ny": _log_int(rng, 10, 100), "k": rng.choice([2, 3]), "steps": rng.randint(1, 8)}
    if kind == "line":
        return {"kind": kind, "physics": rng.choice(["advection", "euler"]), "nx": _log_int(rng, 20, 960), "k": rng.choice([1, 2, 3]),
                "precision": "f64", "steps": rng.randint(10, 200)}
    if kind == "ensemble":
        return {"kind": kind, "problems": rng.randint(2, 12), "largest": _log_int(rng, 64, 256), "precision": "f32", "steps": rng.randint(4, 40)}
    if kind == "train":
        return {"kind": kind, "samples": _log_int(rng, 300, 9000), "batch": rng.choice([256, 1024, 4096])}
    nx = _log_int(rng, 60, 1500)
    return {"kind": kind, "nx": nx, "ny": max(30, int(nx * rng.uniform(0.3, 0.7))), "precision": rng.choice(["f32", "f64"])}


# ---- the method in 64 bits (plain torch, whole meshes) -----------------------------------------------------------
def _legendre(n, x):
    c = np.zeros(n + 1)
    c[n] = 1.0
    return np.polynomial.legendre.legval(x, c)


def _dlegendre(n, x):
    c = np.zeros(n + 1)
    c[n] = 1.0
    return np.polynomial.legendre.legval(x, np.polynomial.legendre.legder(c)) if n else 0.0 * x


def _degrees(k, basis):
    top = k if basis == "P" else 2 * k
    return [(i, d - i) for d in range(top + 1) for i in range(d, -1, -1) if i <= k and d - i <= k]


class Method:
    """cRKDG on one mesh, states u[v, m, y, x] in FP64.  `sides`: W, E, S, N boundary conditions, "periodic",
    "outflow" or a function (interior state [v, ...], x, y, t) -> exterior state."""

    def __init__(self, nx, ny, box, k, modes, physics, sides, tableau, beta=(0.0, 0.0), gamma=GAMMA):
        self.nx, self.ny, self.k, self.modes = nx, ny, k, modes
        self.x0, self.x1, self.y0, self.y1 = box
        self.dx, self.dy = (box[1] - box[0]) / nx, (box[3] - box[2]) / ny
        self.physics, self.sides, self.tableau, self.beta, self.gamma = physics, sides, tableau, beta, gamma
        g, w = np.polynomial.legendre.leggauss(k + 1)
        self.g, self.w = g, w
        dev = lambda a: torch.tensor(np.array(a), dtype=torch.float64, device="cuda")  # noqa: E731
        one = np.ones(1)
        P = [_legendre(i, g) for i in range(k + 1)]
        D = [_dlegendre(i, g) for i in range(k + 1)]
        ends = {s: [_legendre(i, s * one)[0] for i in range(k + 1)] for s in (1.0, -1.0)}
        outer = lambda a, b: np.outer(a, b).reshape(-1)  # noqa: E731
        W = outer(w, w)
        self.phi = dev([outer(P[i], P[j]) for i, j in modes]).T.contiguous()                      # [q, m]
        self.vx = dev([W * outer(D[i], P[j]) / (2 * self.dx) for i, j in modes])                  # [m, q]
        self.vy = dev([W * outer(P[i], D[j]) / (2 * self.dy) for i, j in modes])
        self.cm = dev([(2 * i + 1) * (2 * j + 1) for i, j in modes])
        self.project = dev([(2 * i + 1) * (2 * j + 1) * 0.25 * W * outer(P[i], P[j]) for i, j in modes])
        self.trace = {"E": dev([ends[1.0][i] * P[j] for i, j in modes]).T, "W": dev([ends[-1.0][i] * P[j] for i, j in modes]).T,
                      "N": dev([ends[1.0][j] * P[i] for i, j in modes]).T, "S": dev([ends[-1.0][j] * P[i] for i, j in modes]).T}
        ww = dev(0.5 * w)
        self.lift = {s: (t * ww[:, None]).T / (self.dx if s in "EW" else self.dy) for s, t in self.trace.items()}   # [m, p]

    def points(self, gx, gy):
        """Coordinates [.., y, x] of the points at reference positions gx, gy of every cell."""
        d = dict(dtype=torch.float64, device="cuda")
        xc = self.x0 + (torch.arange(self.nx, **d) + 0.5) * self.dx
        yc = self.y0 + (torch.arange(self.ny, **d) + 0.5) * self.dy
        gx, gy = (torch.as_tensor(np.array(v), **d).reshape(-1, 1, 1) for v in (gx, gy))
        X = xc[None, None, :] + 0.5 * self.dx * gx
        Y = yc[None, :, None] + 0.5 * self.dy * gy
        return torch.broadcast_tensors(X, Y)

    def projection(self, fn):
        """Modes [v, m, y, x] of fn(X, Y) -> [v, ...] by the volume Gauss rule."""
        gx, gy = np.repeat(self.g, self.k + 1), np.tile(self.g, self.k + 1)
        return torch.einsum("mq,vqyx->vmyx", self.project, fn(*self.points(gx, gy)))

    def flux(self, u, axis):
        """Flux along an axis and the wave speed at states u[v, ...]."""
        if self.physics == "advection":
            b = self.beta[axis]
            return b * u, torch.full_like(u[0], abs(b))
        vel = u[1 + axis] / u[0]
        p = (self.gamma - 1) * (u[3] - 0.5 * (u[1] ** 2 + u[2] ** 2) / u[0])
        f = u * vel
        f[1 + axis] += p
        f[3] += p * vel
        return f, vel.abs() + torch.sqrt(torch.clamp(self.gamma * p / u[0], min=0.0))

    def faces(self, u, axis, t):
        """Lax--Friedrichs fluxes [v, p, y, x] on the low and the high face of every cell along an axis."""
        dim = 3 - axis
        lo, hi = ("W", "E") if axis == 0 else ("S", "N")
        n = self.nx if axis == 0 else self.ny
        tl = torch.einsum("pm,vmyx->vpyx", self.trace[lo], u)
        th = torch.einsum("pm,vmyx->vpyx", self.trace[hi], u)
        below, above = th.narrow(dim, n - 1, 1), tl.narrow(dim, 0, 1)      # periodic neighbours of the first and last cell
        if self.sides[2 * axis] != "periodic":
            one = np.ones(self.k + 1)
            at = lambda s: self.points(s * one, self.g) if axis == 0 else self.points(self.g, s * one)  # noqa: E731
            for end in (0, 1):
                side, inner = self.sides[2 * axis + end], (tl.narrow(dim, 0, 1), th.narrow(dim, n - 1, 1))[end]
                ext = inner
                if side != "outflow":
                    X, Y = (c.narrow(dim - 1, (0, n - 1)[end], 1) for c in at((-1.0, 1.0)[end]))
                    ext = side(inner, X, Y, t)
                below, above = (ext, above) if end == 0 else (below, ext)
        left, right = torch.cat([below, th], dim), torch.cat([tl, above], dim)
        (fl, sl), (fr, sr) = self.flux(left, axis), self.flux(right, axis)
        F = 0.5 * (fl + fr - torch.maximum(sl, sr) * (right - left))
        return F.narrow(dim, 0, n), F.narrow(dim, 1, n)

    def volume(self, u):
        q = torch.einsum("qm,vmyx->vqyx", self.phi, u)
        return torch.einsum("mq,vqyx->vmyx", self.vx, self.flux(q, 0)[0]) + torch.einsum("mq,vqyx->vmyx", self.vy, self.flux(q, 1)[0])

    def lifted(self, low, high, axis):
        lo, hi = ("W", "E") if axis == 0 else ("S", "N")
        return torch.einsum("mp,vpyx->vmyx", self.lift[hi], high) - torch.einsum("mp,vpyx->vmyx", self.lift[lo], low)

    def local(self, u, vol):
        out = -vol
        for axis, (lo, hi) in enumerate((("W", "E"), ("S", "N"))):
            own = [self.flux(torch.einsum("pm,vmyx->vpyx", self.trace[s], u), axis)[0] for s in (lo, hi)]
            out += self.lifted(own[0], own[1], axis)
        return out * self.cm[:, None, None]

    def step(self, u, t, dt):
        A, b = self.tableau
        ops, out = [], u.clone()
        for i in range(len(b)):
            w = u.clone()
            for j in range(i):
                if A[i][j]:
                    w -= dt * A[i][j] * ops[j]
            vol = self.volume(w)
            ops.append(self.local(w, vol) if i + 1 < len(b) else None)
            if b[i]:
                ti = t + sum(A[i][:i]) * dt
                L = -vol
                for axis in (0, 1):
                    L += self.lifted(*self.faces(w, axis, ti), axis)
                out -= dt * b[i] * L * self.cm[:, None, None]
        return out

    def speed(self, u):
        a = u[:, 0]
        return float((self.flux(a, 0)[1] / self.dx + self.flux(a, 1)[1] / self.dy).max())

    def neighbours(self, a, t):
        """Cell averages of the W, E, S, N neighbours (ghost averages at the ghost cells' centres)."""
        out = []
        for s, (axis, shift) in enumerate(((0, 1), (0, -1), (1, 1), (1, -1))):
            dim = 2 - axis
            nb = torch.roll(a, shift, dim)
            if self.sides[s] != "periodic":
                n, at = a.shape[dim], 0 if shift == 1 else a.shape[dim] - 1
                own = a.narrow(dim, at, 1)
                if self.sides[s] != "outflow":
                    X, Y = (c[0] for c in self.points([2.0 * (-shift)] if axis == 0 else [0.0], [2.0 * (-shift)] if axis == 1 else [0.0]))
                    own = self.sides[s](own, X.narrow(dim - 1, at, 1), Y.narrow(dim - 1, at, 1), t)
                nb = torch.cat([own, nb.narrow(dim, 1, n - 1)], dim) if at == 0 else torch.cat([nb.narrow(dim, 0, n - 1), own], dim)
            out.append(nb)
        return out

    def tvb(self, u, M, t):
        """TVB-minmod limiter in characteristic fields (Euler): the limited state and the troubled cells."""
        a, g1 = u[:, 0], self.gamma - 1
        W, E, S, N = self.neighbours(a, t)
        rho, vel = a[0], [a[1] / a[0], a[2] / a[0]]
        q2 = vel[0] ** 2 + vel[1] ** 2
        p = g1 * (a[3] - 0.5 * rho * q2)
        c, H = torch.sqrt(self.gamma * p / rho), (a[3] + p) / rho
        new, flag = [], torch.zeros_like(rho, dtype=torch.bool)
        for axis, (lo, hi, h) in enumerate(((W, E, self.dx), (S, N, self.dy))):
            n, tt = 1 + axis, 2 - axis
            vn, vt = vel[axis], vel[1 - axis]
            b1, b2 = g1 / c ** 2, 0.5 * g1 * q2 / c ** 2

            def left(d):
                k = b1 * (vn * d[n] + vt * d[tt] - d[3])
                return torch.stack([0.5 * (b2 * d[0] - k + (vn * d[0] - d[n]) / c), (1 - b2) * d[0] + k, d[tt] - vt * d[0],
                                    0.5 * (b2 * d[0] - k - (vn * d[0] - d[n]) / c)])
            s1, s2, s3 = left(u[:, 1 + axis]), left(hi - a), left(a - lo)
            m = torch.minimum(torch.minimum(s1.abs(), s2.abs()), s3.abs())
            same = ((s1 > 0) & (s2 > 0) & (s3 > 0)) | ((s1 < 0) & (s2 < 0) & (s3 < 0))
            mt = torch.where(s1.abs() <= M * h * h, s1, torch.where(same, torch.sign(s1) * m, torch.zeros_like(m)))
            flag |= (mt != s1).any(0)
            r = [None] * 4
            r[0] = mt[0] + mt[1] + mt[3]
            r[n] = vn * r[0] + c * (mt[3] - mt[0])
            r[tt] = vt * r[0] + mt[2]
            r[3] = H * (mt[0] + mt[3]) + vn * c * (mt[3] - mt[0]) + 0.5 * q2 * mt[1] + vt * mt[2]
            new.append(torch.stack(r))
        out = u.clone()
        out[:, 1:] = torch.where(flag, torch.zeros_like(out[:, 1:]), out[:, 1:])
        for axis in (0, 1):
            out[:, 1 + axis] = torch.where(flag, new[axis], u[:, 1 + axis])
        return out, flag

    def positive(self, u, eps):
        """Positivity-preserving scaling of density, then pressure (Zhang and Shu, J. Comput. Phys. 229, 2010)."""
        pts = torch.cat([self.phi] + [self.trace[s] for s in "EWNS"], 0)
        u = u.clone()
        rmin = torch.einsum("qm,myx->qyx", pts, u[0]).amin(0)
        th = torch.where(rmin < eps, ((u[0, 0] - eps) / (u[0, 0] - rmin).clamp(min=1e-300)).clamp(0.0, 1.0), torch.ones_like(rmin))
        u[0, 1:] *= th
        avg = u[:, :1].transpose(0, 1)[0]
        th2, kk = torch.ones_like(rmin), eps / (self.gamma - 1)
        for q in range(pts.shape[0]):
            d = torch.einsum("m,vmyx->vyx", pts[q, 1:], u[:, 1:])
            a = d[0] * d[3] - 0.5 * (d[1] ** 2 + d[2] ** 2)
            b = avg[0] * d[3] + avg[3] * d[0] - avg[1] * d[1] - avg[2] * d[2] - kk * d[0]
            c = avg[0] * avg[3] - 0.5 * (avg[1] ** 2 + avg[2] ** 2) - kk * avg[0]
            root = torch.sqrt((b * b - 4 * a * c).clamp(min=0.0))
            z = -0.5 * (b + torch.where(b >= 0, root, -root))
            far = torch.full_like(a, 2.0)
            r1, r2 = (torch.where((r > 0) & (r <= 1), r, far) for r in (c / z, z / a))
            r = torch.minimum(r1, r2)
            th2 = torch.minimum(th2, torch.where(a + b + c < 0, torch.where(r > 1, torch.zeros_like(r), r), torch.ones_like(r)))
        u[:, 1:] *= th2
        return u


# ---- problems ---------------------------------------------------------------------------------------------------
def _conserved(rho, w, v, p):
    rho, w, v, p = torch.broadcast_tensors(*(torch.as_tensor(a, dtype=torch.float64, device="cuda") for a in (rho, w, v, p)))
    return torch.stack([rho, rho * w, rho * v, p / (GAMMA - 1) + 0.5 * rho * (w * w + v * v)])


def _waves(rng, amp, box):
    """A smooth random field of the given amplitude: a few sine waves over the box."""
    terms = [(rng.uniform(0.2, 1.0), 2 * math.pi * rng.integers(1, 4) / (box[1] - box[0]), 2 * math.pi * rng.integers(1, 4) / (box[3] - box[2]),
              rng.uniform(0, 2 * math.pi)) for _ in range(4)]
    norm = amp / sum(t[0] for t in terms)
    return lambda X, Y: norm * sum(a * torch.sin(kx * X + ky * Y + ph) for a, kx, ky, ph in terms)


def _dmr_numbers():
    """Mach 10 shock at 60 degrees into rho = 1.4, p = 1 at rest (Rankine--Hugoniot)."""
    rho2, p2 = 1.4 * 2.4 * 100 / (0.4 * 100 + 2), 1 + 2 * 1.4 / 2.4 * 99
    u2 = 10.0 * (1 - 1.4 / rho2)
    post = (rho2, u2 * math.cos(math.pi / 6), -u2 * math.sin(math.pi / 6), p2)
    cons = lambda r, w, v, p: [r, r * w, r * v, p / (GAMMA - 1) + 0.5 * r * (w * w + v * v)]  # noqa: E731
    return post, cons(*post), cons(1.4, 0.0, 0.0, 1.0), 1.0 / 6.0, 1.0 / math.sqrt(3.0), 10.0 / math.cos(math.pi / 6)


def _dmr(case, seed):
    nx, ny, k, box = case["nx"], case["ny"], case["k"], (0.0, 4.0, 0.0, 1.0)
    prim, post, pre, x0, slope, speed = _dmr_numbers()
    const = lambda st, like: torch.tensor(st, dtype=torch.float64, device="cuda").reshape(4, *([1] * (like.dim() - 1))).expand_as(like)  # noqa: E731

    def bottom(u, X, Y, t):
        wall = u.clone()
        wall[2] = -wall[2]
        return torch.where(X < x0, const(post, u), wall)

    def top(u, X, Y, t):
        return torch.where(X < x0 + slope * Y + speed * t, const(post, u), const(pre, u))
    sides = [lambda u, X, Y, t: const(post, u), "outflow", bottom, top]
    m = Method(nx, ny, box, k, _degrees(k, "P"), "euler", sides, T.SSPRK3)
    bump = _waves(np.random.default_rng(seed), 0.02, box)

    def ic(X, Y):
        behind = X < x0 + slope * Y
        pick = lambda a, b: torch.where(behind, torch.full_like(X, a), torch.full_like(X, b))  # noqa: E731
        return _conserved(pick(prim[0], 1.4) * (1 + bump(X, Y)), pick(prim[1], 0.0), pick(prim[2], 0.0), pick(prim[3], 1.0))
    mesh = B.make_mesh(2, nx, ny, box, [B.BC_DIRICHLET, B.BC_OUTFLOW, B.BC_DIRICHLET, B.BC_DIRICHLET],
                       [B.FN_CONST, 0, B.FN_DMR_BOTTOM, B.FN_DMR_TOP], [post, None, post + [x0], post + pre + [x0, slope, speed]])
    return m, mesh, ic, dict(k=k, basis=B.BASIS_P, tableau=T.SSPRK3, physics=B.EULER)


def _vortex(case, seed):
    nx, ny, box = case["nx"], case["ny"], (0.0, 10.0, 0.0, 10.0)
    rng = np.random.default_rng(seed)
    cx, cy, eps = rng.uniform(3, 7), rng.uniform(3, 7), rng.uniform(4.0, 5.0)

    def ic(X, Y):
        xb, yb = X - cx, Y - cy
        xb, yb = xb - 10 * torch.round(xb / 10), yb - 10 * torch.round(yb / 10)
        r2 = xb * xb + yb * yb
        a = eps / (2 * math.pi) * torch.exp(0.5 * (1 - r2))
        rho = (1 - (GAMMA - 1) * eps ** 2 / (8 * GAMMA * math.pi ** 2) * torch.exp(1 - r2)) ** (1 / (GAMMA - 1))
        return _conserved(rho, 1 - a * yb, 1 + a * xb, rho ** GAMMA)
    m = Method(nx, ny, box, 2, _degrees(2, "Q"), "euler", ["periodic"] * 4, T.RK4)
    mesh = B.make_mesh(2, nx, ny, box, [B.BC_PERIODIC] * 4)
    return m, mesh, ic, dict(k=2, basis=B.BASIS_Q, tableau=T.RK4, physics=B.EULER)


def _advection(case, seed):
    nx, ny, k, box, beta = case["nx"], case["ny"], case["k"], (0.0, 1.0, 0.0, 1.0), (1.0, 0.5)
    field = _waves(np.random.default_rng(seed), 1.0, box)
    m = Method(nx, ny, box, k, _degrees(k, case["basis"]), "advection", ["periodic"] * 4, T.SSPRK3, beta)
    mesh = B.make_mesh(2, nx, ny, box, [B.BC_PERIODIC] * 4)
    return m, mesh, lambda X, Y: field(X, Y)[None], dict(k=k, basis=B.BASIS_P if case["basis"] == "P" else B.BASIS_Q, tableau=T.SSPRK3,
                                                         physics=B.ADVECTION, beta=beta)


def _inflow(case, seed):
    nx, ny, k, box = case["nx"], case["ny"], case["k"], (-1.0, 1.0, -1.0, 1.0)
    rng = np.random.default_rng(seed)
    pp = [float(rng.uniform(0.5, 1.5)), math.pi, 1.0, math.pi, 1.0]
    data = lambda X, Y, t: pp[0] * torch.sin(math.pi * (X - t)) * torch.sin(math.pi * (Y - t))  # noqa: E731
    inflow = lambda u, X, Y, t: data(X, Y, t)[None].expand_as(u)  # noqa: E731
    m = Method(nx, ny, box, k, _degrees(k, "Q"), "advection", [inflow, "outflow", inflow, "outflow"], T.RK4, (1.0, 1.0))
    mesh = B.make_mesh(2, nx, ny, box, [B.BC_DIRICHLET, B.BC_OUTFLOW, B.BC_DIRICHLET, B.BC_OUTFLOW],
                       [B.FN_SINE_PROD, 0, B.FN_SINE_PROD, 0], [pp, None, pp, None])
    return m, mesh, lambda X, Y: data(X, Y, 0.0)[None], dict(k=k, basis=B.BASIS_Q, tableau=T.RK4, physics=B.ADVECTION, beta=(1.0, 1.0))


def _line(case, seed):
    """1D runs; in 64 bits as a 2D mesh of one periodic row with the modes (i, 0)."""
    nx, k = case["nx"], case["k"]
    rng = np.random.default_rng(seed)
    ph = rng.uniform(0, 2 * math.pi)
    euler = case["physics"] == "euler"
    m = Method(nx, 1, (0.0, 2 * math.pi, 0.0, 1.0), k, [(i, 0) for i in range(k + 1)], case["physics"], ["periodic"] * 4, T.SSPRK3, (1.0, 0.0))
    mesh = B.make_mesh(1, nx, 1, (0.0, 2 * math.pi, 0.0, 1.0), [B.BC_PERIODIC] * 4)

    def ic(X, Y):
        if not euler:
            return torch.sin(X + ph)[None]
        return _conserved(1 + 0.2 * torch.sin(X + ph), 0.7 + 0 * X, 0 * X, 1 + 0.1 * torch.cos(X))
    return m, mesh, ic, dict(k=k, basis=B.BASIS_P, tableau=T.SSPRK3, physics=B.EULER if euler else B.ADVECTION, beta=(1.0, 0.0))


def _indicator(case, seed):
    """A shock and a vortex on [0, 2] x [0, 1] with small waves everywhere."""
    nx, ny, box = case["nx"], case["ny"], (0.0, 2.0, 0.0, 1.0)
    bump = _waves(np.random.default_rng(seed), 0.02, box)
    c1 = math.sqrt(GAMMA)
    up = [1.0, 1.1 * c1, 0.0, 1 / (GAMMA - 1) + 0.5 * (1.1 * c1) ** 2]
    m = Method(nx, ny, box, 2, _degrees(2, "P"), "euler",
               [lambda u, X, Y, t: torch.tensor(up, dtype=torch.float64, device="cuda").reshape(4, *([1] * (u.dim() - 1))).expand_as(u)] + ["outflow"] * 3, T.SSPRK3)

    def ic(X, Y):
        xb, yb = (X - 0.25) / 0.05, (Y - 0.5) / 0.05
        r2 = xb * xb + yb * yb
        a = 0.3 / (2 * math.pi) * torch.exp(0.5 * (1 - r2))
        ahead = X < 0.5
        rho2, p2 = 2.4 * 1.21 / (0.4 * 1.21 + 2), 1 + 2 * 1.4 / 2.4 * 0.21
        rho = torch.where(ahead, 1 + 0 * X, rho2 + 0 * X) * (1 + bump(X, Y))
        w = torch.where(ahead, 1.1 * c1 - a * yb, 1.1 * c1 / rho2 + 0 * X) + 0.3 * bump(Y, X)
        return _conserved(rho, w, torch.where(ahead, a * xb, 0 * X) + 0.2 * bump(X, 1 - Y), torch.where(ahead, 1 + 0 * X, p2 + 0 * X) * (1 - bump(X, Y)))
    mesh = B.make_mesh(2, nx, ny, box, [B.BC_DIRICHLET, B.BC_OUTFLOW, B.BC_OUTFLOW, B.BC_OUTFLOW], [B.FN_CONST, 0, 0, 0], [up, None, None, None])
    return m, mesh, ic, dict(k=2, basis=B.BASIS_P, tableau=T.SSPRK3, physics=B.EULER)


PROBLEMS = {"dmr": _dmr, "vortex": _vortex, "advection": _advection, "inflow": _inflow, "line": _line, "indicator": _indicator}


def _initial(case, seed):
    """The method, the mesh, the solver's arguments and the initial state as the solver stores it."""
    m, mesh, ic, scheme = PROBLEMS[case["kind"]](case, seed)
    u = m.projection(ic)
    if case["kind"] == "line" and case["physics"] == "euler":
        u = u[[0, 1, 3]]
    precision = case.get("precision", "f64")
    if precision == "f32d":
        hi = u.float()
        u = torch.stack([hi, (u - hi.double()).float()])
    else:
        u = u.to(torch.float32 if precision == "f32" else torch.float64)
    return m, mesh, scheme, u.contiguous()


def _sizes(case, rng):
    """Uneven problem sizes of an ensemble, odd ones among them."""
    lo = min(48, case["largest"])
    out = [int(round(math.exp(rng.uniform(math.log(lo), math.log(case["largest"] + 0.4))))) for _ in range(case["problems"])]
    return [case["largest"]] + out[1:]


def _ensemble(case, seed):
    """Four smoothly joined quadrant states per problem; sizes depend on the case alone."""
    sizes = _sizes(case, np.random.default_rng(case["problems"] * 1000 + case["largest"]))
    rng = np.random.default_rng(seed)
    out = []
    for n in sizes:
        m = Method(n, n, (0.0, 1.0, 0.0, 1.0), 2, _degrees(2, "P"), "euler", ["outflow"] * 4, T.SSPRK3)
        q = [[rng.uniform(0.5, 1.5), rng.uniform(-0.5, 0.5), rng.uniform(-0.5, 0.5), rng.uniform(0.5, 1.5)] for _ in range(4)]

        def ic(X, Y, q=q):
            a, b = (0.5 * (1 + torch.tanh((c - 0.5) / 0.08)) for c in (X, Y))
            return _conserved(*(q[0][i] * a * b + q[1][i] * (1 - a) * b + q[2][i] * (1 - a) * (1 - b) + q[3][i] * a * (1 - b) for i in range(4)))
        out.append((m, m.projection(ic)))
    return sizes, out


def _samples(case, seed):
    """Feature vectors as the indicator's: 36 values in [-1, 1], four log scales; about one label in six positive."""
    n = case["samples"]
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    X = torch.randn(n, 40, generator=g, device="cuda")
    X[:, :36] /= X[:, :36].reshape(n, 4, 9).abs().amax(2).repeat_interleave(9, 1)
    X[:, 36:] = (X[:, 36:] * 1.5).clamp(-8, 8)
    y = ((X[:, 36] + X[:, 0] * X[:, 4] + 0.5 * X[:, 9]) > 1.5).float()
    return X, y


# ---- a pass -------------------------------------------------------------------------------------------------------
_stream = None


def _compute_stream():
    """The program's one compute stream (not the default stream: graphs are captured on it)."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


def prepare(case, seed):
    kind = case["kind"]
    stream = _compute_stream()
    s = {"case": case, "stream": stream}
    if kind == "train":
        s["X"], s["y"] = _samples(case, seed)
        torch.cuda.current_stream().synchronize()
        s["net"] = B.MLP(seed=seed, stream=stream.cuda_stream)
        s["params"] = s["net"].get_params()
        return s
    if kind == "ensemble":
        sizes, problems = _ensemble(case, seed)
        b = B.Batch([(n, n, (0.0, 1.0, 0.0, 1.0)) for n in sizes], 2, B.BASIS_P, T.SSPRK3, PREC[case["precision"]], stream=stream.cuda_stream)
        for p, (_, u) in enumerate(problems):
            b.set_state(p, u.cpu().numpy())
        b.limit(DMR_M)
        b.positivity(PP_EPS)
        s["batch"] = b
        return s
    m, mesh, scheme, u = _initial(case, seed)
    s["a"], s["b"] = u, torch.zeros_like(u)
    torch.cuda.current_stream().synchronize()
    sol = B.Solver(mesh, scheme["k"], scheme["basis"], scheme["tableau"], scheme["physics"], PREC[case.get("precision", "f64")], gamma=GAMMA,
                   beta=scheme.get("beta", (1.0, 0.0)), stream=stream.cuda_stream, state_buffers=(s["a"].data_ptr(), s["b"].data_ptr()))
    s["solver"] = sol
    if kind == "dmr":
        sol.limit(DMR_M)
        sol.positivity(PP_EPS)
    if kind == "indicator":
        n = case["nx"] * case["ny"]
        s["net"] = B.MLP(seed=11, stream=stream.cuda_stream)
        s["X"], s["y"], s["z"] = (torch.empty(n, d, device="cuda").squeeze(1) for d in (40, 1, 1))
    s["dt"] = _fixed_dt(case, m)
    return s


def _fixed_dt(case, m):
    if case["kind"] == "advection":
        return 0.1 / (1.0 / m.dx + 0.5 / m.dy)
    if case["kind"] == "inflow":
        return min(m.dx, m.dy) / 30
    return 0.05 * m.dx if case["kind"] == "line" else None


def run(s):
    case = s["case"]
    kind, n = case["kind"], case.get("steps", 0)
    if kind == "train":
        net = s["net"]
        net.set_params(s["params"])
        loss = net.train(s["X"].data_ptr(), s["y"].data_ptr(), case["samples"], 1, case["batch"], 1e-3, pos_weight=0.25, seed=7)
        return [net.get_params(), loss]
    if kind == "ensemble":
        s["batch"].run(CFL["ensemble", 2], T_END, steps_per_graph=n, max_graphs=1)
        return [s["batch"].get_state(p) for p in range(case["problems"])]
    sol = s["solver"]
    if kind == "indicator":
        cells = case["nx"] * case["ny"]
        sol.features(s["X"].data_ptr(), s["y"].data_ptr(), DMR_M)
        s["net"].predict(s["X"].data_ptr(), cells, s["z"].data_ptr())
        return [s["X"], s["y"], s["z"]]
    if kind == "line":
        sol.run_fixed(n, s["dt"])
    elif kind in ("advection", "inflow"):
        for _ in range(n):
            sol.step(s["dt"])
    elif case["call"] == "host":
        for _ in range(n):
            sol.step(sol.cfl_dt(CFL[kind, case.get("k", 2)]))
    else:
        sol.advance(n, CFL[kind, case.get("k", 2)], T_END, capture=case["call"] == "graph")
    return s["b"] if sol.current_state()[0] else s["a"]


# ---- what a pass cannot do without ---------------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind == "train":
        n, params = case["samples"], 11009
        return {"bytes": 4.0 * (41 * n + 2 * params), "flops": 6.0 * params * n}
    if kind == "indicator":
        n, e = case["nx"] * case["ny"], 4 if case["precision"] == "f32" else 8
        return {"bytes": float(n * (24 * e + 4 * 42)), "flops": float(n * (2 * 11009 + 300))}
    if kind == "ensemble":
        cells = sum(n * n for n in _sizes(case, np.random.default_rng(case["problems"] * 1000 + case["largest"])))
        return {"bytes": cells * 24 * (4.0 + 8.0), "flops": case["steps"] * cells * float(workcount.step_flops_per_cell(2, "P", "euler", *T.SSPRK3))}
    cells, e = case["nx"] * case.get("ny", 1), {"f32": 4, "f32d": 8, "f64": 8}[case.get("precision", "f64")]
    if kind == "line":
        nv, nm = 3 if case["physics"] == "euler" else 1, case["k"] + 1
        # per stage: point values, their fluxes and projections on k + 1 points, two traces and a face flux
        return {"bytes": 2.0 * cells * nv * nm * e, "flops": case["steps"] * cells * 3.0 * nv * (4 * nm * nm + 8 * nm + 20)}
    if kind == "advection":
        modes = _degrees(case["k"], case["basis"])
        # the linear flux as fixed maps of the modes: s applications of the derivative, two inflow-face lifts, the sums
        nnz = sum((i + 1) // 2 + (j + 1) // 2 for i, j in modes)
        return {"bytes": 2.0 * cells * len(modes) * e, "flops": case["steps"] * cells * (3 * 2.0 * nnz + 10.0 * len(modes))}
    k, basis, tab = {"dmr": (case.get("k"), "P", T.SSPRK3), "vortex": (2, "Q", T.RK4), "inflow": (case.get("k"), "Q", T.RK4)}[kind]
    physics = "advection" if kind == "inflow" else "euler"
    dof = len(_degrees(k, basis)) * (1 if kind == "inflow" else 4)
    return {"bytes": 2.0 * cells * dof * e, "flops": case["steps"] * cells * float(workcount.step_flops_per_cell(k, basis, physics, *tab))}


# ---- the same pass in 64 bits ----------------------------------------------------------------------------------------
def _advance(m, u, steps, cfl=None, dt=None, limited=False):
    t = 0.0
    for _ in range(steps):
        if limited:
            u = m.positive(m.tvb(u, DMR_M, t)[0], PP_EPS)
        d = cfl / m.speed(u) if cfl else dt
        u = m.step(u, t, d)
        t += d
    return u, t


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "ensemble":
        out = []
        for m, u in _ensemble(case, seed)[1]:
            u = u.float().double() if case["precision"] == "f32" else u
            u, t = _advance(m, u, case["steps"], cfl=CFL["ensemble", 2], limited=True)
            out.append(m.positive(m.tvb(u, DMR_M, t)[0], PP_EPS).cpu())      # read back limited
        return out
    m, _, _, u = _initial(case, seed)
    if kind == "indicator":
        return _exact_indicator(m, u.double())
    u = u.double()
    if case.get("precision") == "f32d":
        u = u[0] + u[1]
    thin = kind == "line" and case["physics"] == "euler"
    if thin:
        u = torch.stack([u[0], u[1], torch.zeros_like(u[0]), u[2]])
    cfl = CFL.get((kind, case.get("k", 2)))
    u, _ = _advance(m, u, case["steps"], cfl=cfl, dt=_fixed_dt(case, m), limited=kind == "dmr")
    if thin:
        u = u[[0, 1, 3]]
    if case.get("precision") == "f32d":      # the nearest pair of 32-bit planes
        hi = u.float().double()
        u = torch.stack([hi, u - hi])
    return u


def _layers(p):
    out, o = [], 0
    for nout, nin in ((64, 40), (64, 64), (64, 64), (1, 64)):
        out += [p[o:o + nout * nin].reshape(nout, nin), p[o + nout * nin:o + nout * nin + nout]]
        o += nout * nin + nout
    return out


def _logits(layers, X):
    for W, b in (layers[0:2], layers[2:4], layers[4:6]):
        X = torch.relu(X @ W.T + b)
    return (X @ layers[6].T + layers[7])[:, 0]


def _exact_indicator(m, u):
    a = u[:, 0]
    W, E, S, N = m.neighbours(a, 0.0)
    d = torch.stack([E - a, W - a, N - a, S - a] + [u[:, i] for i in range(1, 6)], 1)         # [q, 9, y, x]
    s = d.abs().amax(1).clamp(min=1e-30)
    scale = torch.log10(s / (DMR_M * max(m.dx, m.dy) ** 2)).clamp(-8, 8)
    X = torch.cat([(d / s[:, None]).reshape(36, -1), scale.reshape(4, -1)], 0).T
    net = B.MLP(seed=11)
    p = torch.tensor(net.get_params(), dtype=torch.float64, device="cuda")
    return [X, m.tvb(u, DMR_M, 0.0)[1].double().reshape(-1), _logits(_layers(p), X)]


def _exact_train(case, seed):
    """Adam over the library's seeded shuffle (SplitMix64, Fisher--Yates), in 64 bits."""
    X, y = _samples(case, seed)
    X, y = X.double(), y.double()
    net = B.MLP(seed=seed)
    p = torch.tensor(net.get_params(), dtype=torch.float64, device="cuda")
    n, state, mask = case["samples"], 7, (1 << 64) - 1
    order = list(range(n))
    for i in range(n - 1, 0, -1):
        state = (state + 0x9E3779B97F4A7C15) & mask
        z = state
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        j = (z ^ (z >> 31)) % (i + 1)
        order[i], order[j] = order[j], order[i]
    order = torch.tensor(order, device="cuda")
    m1, m2, losses = torch.zeros_like(p), torch.zeros_like(p), []
    for t, at in enumerate(range(0, n, case["batch"]), 1):
        rows = order[at:at + case["batch"]]
        q = p.detach().requires_grad_(True)
        z = _logits(_layers(q), X[rows])
        loss = torch.nn.functional.binary_cross_entropy_with_logits(z, y[rows], pos_weight=torch.tensor(0.25, dtype=torch.float64, device="cuda"))
        g, = torch.autograd.grad(loss, q)
        m1, m2 = 0.9 * m1 + 0.1 * g, 0.999 * m2 + 0.001 * g * g
        p = p - 1e-3 * (m1 / (1 - 0.9 ** t)) / (torch.sqrt(m2 / (1 - 0.999 ** t)) + 1e-8)
        losses.append(float(loss))
    return [p, sum(losses) / len(losses)]
