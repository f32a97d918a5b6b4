"""What is timed: the public calls of the solver library over the sizes they are used at.

listed() are the cases, draw() more of the same ranges. prepare() makes what a caller holds before
the call (a domain and its vectors), run() is one call, work() the bytes and operations it cannot do
without, exact() the same results in 64 bits from the 1-D matrices of the separable operator
(curved elements: from the metric at the nodes), in plain numpy and torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2111_06767_gb300 as dgg

DEV = "cuda"
TOL = 1e-10  # relative residual of every solve


def _case(kind, n, N, **more):
    c = {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "N": N, "precision": "fp64", "hx": 1.0, "hy": 1.0,
         "hz": 1.0, "neumann": 0}
    c.update(more)
    return c


def listed():
    return [
        # one operator call on the smallest documented problem: a launch and its latency
        _case("apply", (2, 2, 2), 6, name="apply_fp64_2x2x2_N6"),
        # the outer FP64 operator of the binary-puncture workload, called once per Krylov iteration
        _case("apply", (16, 16, 16), 6, name="apply_fp64_16x16x16_N6"),
        # the FP64 operator at the size of the operator sweep, odd order and odd counts
        _case("apply", (43, 43, 43), 9, name="apply_fp64_43x43x43_N9"),
        # the FP32 operator of the preconditioner: the headline sweep size at low and at high order
        _case("apply", (96, 96, 96), 4, precision="fp32", name="apply_fp32_96x96x96_N4"),
        _case("apply", (48, 48, 48), 8, precision="fp32", name="apply_fp32_48x48x48_N8"),
        # ragged counts, unequal element widths, Neumann on -x and +z
        _case("apply", (37, 41, 29), 7, precision="fp32", hx=0.9, hy=1.0, hz=1.3, neumann=33,
              name="apply_fp32_37x41x29_N7_neumann"),
        # a curved mesh with a variable coefficient, FP64 operator
        _case("curved", (8, 8, 8), 8, name="curved_fp64_8x8x8_N8"),
        # the Schwarz smoother of a plain FP64 domain at the Gaussian workload's grid
        _case("smooth", (8, 8, 8), 8, name="smooth_fp64_8x8x8_N8"),
        # the FP64 multigrid preconditioner on an uneven grid of the batched stream
        _case("vcycle", (6, 8, 4), 5, name="vcycle_fp64_6x8x4_N5"),
        # the headline solve: 16 Gaussians, mixed precision, 3 levels
        _case("solve", (8, 8, 8), 8, precision="mixed", levels=3, name="solve_mixed_8x8x8_N8"),
        # Newton-Krylov on the binary-puncture workload
        _case("puncture", (16, 16, 16), 6, precision="mixed", name="puncture_mixed_16x16x16_N6"),
        # uneven solves captured as one graph, as in the batched stream
        _case("batch", (2, 2, 2), 4, precision="mixed", count=20, shapes=4, name="batch_mixed_20_uneven"),
    ]


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "curved", "smooth", "vcycle", "solve", "puncture", "batch"])
    if kind == "apply":
        N = rng.randint(4, 9)
        dof = math.exp(rng.uniform(math.log(2e3), math.log(4e7)))
        edge = (dof / N**3) ** (1.0 / 3.0)
        n = tuple(max(1, round(edge * math.exp(rng.uniform(-0.3, 0.3)))) for _ in range(3))
        return _case("apply", n, N, precision=rng.choice(["fp64", "fp32"]), hx=rng.choice([1.0, 0.8, 1.25]),
                     hz=rng.choice([1.0, 1.5]), neumann=rng.choice([0, 0, 0, 1, 12, 34]))
    if kind == "curved":
        return _case("curved", tuple(rng.randint(2, 8) for _ in range(3)), rng.randint(4, 8))
    if kind == "smooth":
        return _case("smooth", tuple(rng.randint(2, 8) for _ in range(3)), rng.randint(4, 8),
                     neumann=rng.choice([0, 0, 1, 36]))
    if kind == "vcycle":
        return _case("vcycle", tuple(rng.randint(2, 8) for _ in range(3)), rng.randint(4, 8),
                     hy=rng.choice([1.0, 1.2]))
    if kind == "solve":
        return _case("solve", (rng.randint(2, 12),) * 3, rng.randint(4, 8), precision="mixed", levels=0)
    if kind == "puncture":
        N = rng.randint(4, 6)
        return _case("puncture", (rng.randint(4, 16),) * 3, N, precision="mixed")
    return _case("batch", (2, 2, 2), 4, precision="mixed", count=rng.randint(4, 20), shapes=rng.randint(1, 1000))


# ---------------------------------------------------------------------------- inputs


def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + salt)
    return g


def _random(n, seed, salt, dtype=torch.float64):
    """U[-1, 1) values, as Krylov vectors are: rough on the scale of the grid."""
    u = torch.empty(n, dtype=dtype, device=DEV)
    return u.uniform_(-1.0, 1.0, generator=_gen(seed, salt))


def _box(c):
    """Box with the element widths hx : hy : hz, [-1, 1]^3 for equal widths on a cube."""
    n = (c["nx"], c["ny"], c["nz"])
    w = [n[i] * c["h" + "xyz"[i]] for i in range(3)]
    s = 1.0 / max(w)
    return tuple(-s * a for a in w), tuple(s * a for a in w), n


def _faces(c):
    return tuple(f for f in range(6) if c["neumann"] >> f & 1)


def _gaussians(seed, salt):
    """16 Gaussians: amplitudes U[-1, 1], centres U[-0.8, 0.8]^3, widths U[0.1, 0.4]."""
    r = np.random.RandomState((7919 * int(seed) + 31 * salt + 2) % 2**31)
    return r.uniform(-1, 1, 16), r.uniform(-0.8, 0.8, (16, 3)), r.uniform(0.1, 0.4, 16)


def _source(seed, salt, x, y, z):
    amp, cen, wid = _gaussians(seed, salt)
    f = torch.zeros_like(x)
    for a, c, s in zip(amp, cen, wid):
        f += a * torch.exp(-((x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2) / (s * s))
    return f


class _Puncture:
    def __init__(self, position, mass, momentum):
        self.position, self.mass, self.momentum = position, mass, momentum


def _punctures(seed):
    """Two punctures near (+-3, 0, 0) with bare masses near 0.5 and momenta near +-(0, 0.1, 0)."""
    r = np.random.RandomState((104729 * int(seed) + 3) % 2**31)
    d, m, p = 3.0 + r.uniform(-0.2, 0.2), 0.5 + r.uniform(-0.03, 0.03), 0.1 + r.uniform(-0.01, 0.01)
    return (_Puncture((d, 0.0, 0.0), m, (0.0, p, 0.0)), _Puncture((-d, 0.0, 0.0), m, (0.0, -p, 0.0)))


def _batch_shapes(c):
    r = np.random.RandomState(c["shapes"])
    return [(tuple(int(v) for v in r.randint(2, 9, 3)), int(r.randint(4, 10))) for _ in range(c["count"])]


def _warp(x, y, z):
    """Smooth map of [-1, 1]^3 onto itself that keeps the six faces planar."""
    b = 0.08 * np.sin(np.pi * x) * np.sin(np.pi * y) * np.sin(np.pi * z)
    return x + b, y - 0.75 * b, z + 0.5 * b


def _coefficient(seed, x, y, z):
    r = np.random.RandomState((15485863 * int(seed) + 5) % 2**31)
    k = r.uniform(0.5, 1.5, 3)
    return 1.0 + 0.3 * np.sin(k[0] * x + 1.0) * np.cos(k[1] * y) + 0.1 * np.sin(k[2] * z)


def prepare(case, seed):
    c = case
    kind = c["kind"]
    lower, upper, n = _box(c)
    N = c["N"]
    if kind == "apply":
        dom = dgg.Domain(lower, upper, n, N, precision="mixed" if c["precision"] == "fp32" else "fp64",
                         neumann=_faces(c))
        u = _random(dom.n_dof, seed, 1, torch.float32 if c["precision"] == "fp32" else torch.float64)
        return {"kind": kind, "fp32": c["precision"] == "fp32", "dom": dom, "u": u, "out": torch.empty_like(u)}
    if kind == "curved":
        xyz, K = _curved_nodes(c, seed)
        dom = dgg.Domain(lower, upper, n, N, node_xyz=xyz, coef=K)
        u = _random(dom.n_dof, seed, 1)
        return {"kind": "apply", "fp32": False, "dom": dom, "u": u, "out": torch.empty_like(u)}
    if kind in ("smooth", "vcycle"):
        dom = dgg.Domain(lower, upper, n, N, precision=c["precision"], neumann=_faces(c))
        b = dom.rhs(_source(seed, 1, *dom.coordinates()))
        u0 = 0.01 * _random(dom.n_dof, seed, 2)
        return {"kind": kind, "dom": dom, "b": b, "u0": u0, "u": torch.empty_like(u0)}
    if kind == "solve":
        dom = dgg.Domain(lower, upper, n, N, precision=c["precision"], mg_levels=c["levels"])
        b = dom.rhs(_source(seed, 1, *dom.coordinates()))
        return {"kind": kind, "dom": dom, "b": b, "u": torch.empty_like(b)}
    if kind == "puncture":
        dom = dgg.Domain((-20.0,) * 3, (20.0,) * 3, n, N, precision=c["precision"], problem="puncture",
                         punctures=_punctures(seed))
        return {"kind": kind, "dom": dom, "b": None, "u": torch.empty(dom.n_dof, dtype=torch.float64, device=DEV)}
    doms, bs, us = [], [], []
    for i, (m, order) in enumerate(_batch_shapes(c)):
        doms.append(dgg.Domain(n=m, N=order, precision=c["precision"]))
        bs.append(doms[-1].rhs(_source(seed, i, *doms[-1].coordinates())))
        us.append(torch.zeros_like(bs[-1]))
    return {"kind": kind, "batch": dgg.Batch(doms, bs, us, tol=TOL), "us": us}


def run(state):
    kind = state["kind"]
    if kind == "apply":
        return (state["dom"].apply_f32(state["u"], out=state["out"]) if state["fp32"]
                else state["dom"].apply(state["u"], out=state["out"]))
    if kind == "smooth":  # three smoothing steps from the guess at hand
        state["u"].copy_(state["u0"])
        return state["dom"].schwarz_smooth(0, state["b"], state["u"], 3)
    if kind == "vcycle":
        return state["dom"].vcycle(state["b"], out=state["u"])
    if kind in ("solve", "puncture"):
        state["u"].zero_()
        state["dom"].solve(state["b"], state["u"], tol=TOL)
        return state["u"]
    torch._foreach_zero_(state["us"])
    state["batch"].run()
    return state["us"]


# ---------------------------------------------------------------------------- what a call cannot do without


def _apply_work(n_el, N, size):
    """Read u, write A u; per direction two contractions in even and odd halves, and the faces."""
    dof = n_el * N**3
    return 2.0 * size * dof, (6.0 * N + 12.0) * dof


def _levels(n, most):
    out = [tuple(n)]
    while (most == 0 or len(out) < most) and any(m % 2 == 0 for m in out[-1]):
        out.append(tuple(m // 2 if m % 2 == 0 else m for m in out[-1]))
    return out


def _step_work(n, N, size):
    """One Schwarz step: the operator, every distinct subdomain inverse once, the subdomain products."""
    n_el = n[0] * n[1] * n[2]
    by, fl = _apply_work(n_el, N, size)
    codes = [{(min(i, 2), min(m - 1 - i, 2)) for i in range(m)} for m in n]
    classes = {tuple(sorted(tuple(sorted(v)) for v in (a, b, c))) for a in codes[0] for b in codes[1] for c in codes[2]}
    inv = mac = 0.0
    for k in classes:  # rows of the slots that are present
        inv += (N**3 + 2 * N * N * sum((v[0] > 0) + (v[1] > 0) for v in k)) ** 2
    nbr = [(2.0 * m - 2.0) / m for m in n]
    mac = n_el * (N**3 + 2 * N * N * sum(nbr)) ** 2
    return by + size * inv, fl + 2.0 * mac


def _vcycle_work(n, N, size, most=0):
    by = fl = 0.0
    for m in _levels(n, most):
        b, f = _step_work(m, N, size)
        by, fl = by + b, fl + 6.0 * f  # six steps a level; an inverse that stays on the chip is read once
    return by, fl


def _solve_work(n, N, iterations, most=0):
    dof = n[0] * n[1] * n[2] * N**3
    b, f = _vcycle_work(n, N, 4.0, most)
    a = _apply_work(n[0] * n[1] * n[2], N, 8.0)
    return (iterations * (b + a[0] + 8.0 * dof * 2.0 * iterations), iterations * (f + a[1] + 4.0 * dof * iterations))


def work(case):
    c = case
    n, N = (c["nx"], c["ny"], c["nz"]), c["N"]
    n_el = n[0] * n[1] * n[2]
    kind = c["kind"]
    if kind == "apply":
        b, f = _apply_work(n_el, N, 4 if c["precision"] == "fp32" else 8)
    elif kind == "curved":  # also the nodal metric (J, G) and K, and the chain rule at the nodes
        b, f = _apply_work(n_el, N, 8)
        b, f = b + 11.0 * 8.0 * n_el * N**3, f + 40.0 * n_el * N**3
    elif kind == "smooth":
        b, f = _step_work(n, N, 8.0)
        f *= 3.0
    elif kind == "vcycle":
        b, f = _vcycle_work(n, N, 8.0)
    elif kind == "solve":
        b, f = _solve_work(n, N, 10, c["levels"])
    elif kind == "puncture":
        b, f = _solve_work(n, N, 12)
    else:
        parts = [_solve_work(m, order, 10) for m, order in _batch_shapes(c)]
        b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------- the same in 64 bits


def _lgl(N):
    """Legendre-Gauss-Lobatto points, weights and derivative matrix."""
    P = np.polynomial.legendre.Legendre.basis(N - 1)
    x = np.concatenate([[-1.0], np.sort(P.deriv().roots().real), [1.0]])
    for _ in range(3):  # polish the roots of P'
        x[1:-1] -= P.deriv()(x[1:-1]) / P.deriv(2)(x[1:-1])
    x = 0.5 * (x - x[::-1])
    w = 2.0 / (N * (N - 1) * P(x) ** 2)
    return x, w, _lagrange_deriv(x)


def _lagrange_deriv(x):
    N = len(x)
    c = np.array([np.prod([x[j] - x[k] for k in range(N) if k != j]) for j in range(N)])
    D = np.zeros((N, N))
    for i in range(N):
        for j in range(N):
            if i != j:
                D[i, j] = c[i] / (c[j] * (x[i] - x[j]))
        D[i, i] = -D[i].sum()
    return D


def _interp(x, t):
    """Lagrange interpolation from the points x to t."""
    return np.array([[np.prod([(s - x[k]) / (x[j] - x[k]) for k in range(len(x)) if k != j]) for j in range(len(x))]
                     for s in t])


def _matrix_1d(n, N, h, neumann, C=1.5):
    """1-D operator of n elements of width h (unit transverse weights) and its mass diagonal.

    The 3-D operator on a box is A_x M_y M_z + M_x A_y M_z + M_x M_y A_z.
    """
    _, w, D = _lgl(N)
    A = np.zeros((n * N, n * N))
    lift, sigma = 2.0 / (h * w[0]), C * N * N / h
    g = np.zeros((n, N, n * N))
    for e in range(n):
        g[e][:, e * N:(e + 1) * N] = (2.0 / h) * D
    for e in range(n):
        v, flux = g[e].copy(), np.zeros((N, n * N))
        for side, s in ((0, -1.0), (1, 1.0)):
            p, o = (0, N - 1) if side == 0 else (N - 1, 0)
            q = e + (1 if side else -1)
            ui = np.zeros(n * N)
            ui[e * N + p] = 1.0
            if 0 <= q < n:
                ue = np.zeros(n * N)
                ue[q * N + o] = 1.0
                ge = g[q][o]
            elif neumann[side]:
                ue, ge = ui, -g[e][p]
            else:
                ue, ge = -ui, g[e][p]
            flux[p] += 0.5 * s * (ge - g[e][p]) + (sigma - 0.5 * lift) * (ue - ui)
            v[p] += s * 0.5 * lift * (ue - ui)
        A[e * N:(e + 1) * N] = -(0.5 * h * w)[:, None] * (2.0 / h) * (D @ v) - flux
    return A, np.tile(0.5 * h * w, n)


class _Grid:
    """The separable operator of one box: 1-D matrices, global tensors [z, y, x]."""

    def __init__(self, lower, upper, n, N, neumann=0):
        self.n, self.N, self.box = n, N, (lower, upper, neumann)
        pairs = [_matrix_1d(n[d], N, (upper[d] - lower[d]) / n[d], (neumann >> 2 * d & 1, neumann >> 2 * d + 1 & 1))
                 for d in range(3)]
        self.A = [torch.from_numpy(p[0]).to(DEV) for p in pairs]
        self.m = [torch.from_numpy(p[1]).to(DEV) for p in pairs]
        self.eig = None

    def tensor(self, v):
        """Element-major vector -> [z, y, x]."""
        nx, ny, nz = self.n
        N = self.N
        return (v.to(torch.float64).reshape(nz, ny, nx, N, N, N).permute(0, 3, 1, 4, 2, 5)
                .reshape(nz * N, ny * N, nx * N))

    def vector(self, t):
        nx, ny, nz = self.n
        N = self.N
        return t.reshape(nz, N, ny, N, nx, N).permute(0, 2, 4, 1, 3, 5).reshape(-1)

    def mass(self):
        return self.m[2][:, None, None] * self.m[1][:, None] * self.m[0]

    @staticmethod
    def along(Mx, My, Mz, t):
        t = t @ Mx.T
        t = torch.matmul(My, t)
        return torch.tensordot(Mz, t, dims=1)

    def apply(self, t):
        out = (t @ self.A[0].T) * (self.m[2][:, None, None] * self.m[1][:, None])
        out += torch.matmul(self.A[1], t) * (self.m[2][:, None, None] * self.m[0])
        out += torch.tensordot(self.A[2], t, dims=1) * (self.m[1][:, None] * self.m[0])
        return out

    def solve(self, b):
        """A^-1 b by the 1-D eigenvectors (A_d q = lambda M_d q)."""
        if self.eig is None:
            self.eig = []
            for d in range(3):
                s = self.m[d].rsqrt()
                lam, Q = torch.linalg.eigh((s[:, None] * self.A[d] * s + (s[:, None] * self.A[d] * s).T) * 0.5)
                self.eig.append((lam, s[:, None] * Q))
        (lx, X), (ly, Y), (lz, Z) = self.eig
        t = self.along(X.T, Y.T, Z.T, b) / (lz[:, None, None] + ly[:, None] + lx)
        return self.along(X, Y, Z, t)

    def refined_solve(self, b):
        u = self.solve(b)
        return u + self.solve(b - self.apply(u))

    def coordinates(self):
        lower, upper, _ = self.box
        x = _lgl(self.N)[0]
        axes = []
        for d in range(3):
            h = (upper[d] - lower[d]) / self.n[d]
            axes.append(torch.from_numpy((lower[d] + h * (np.arange(self.n[d])[:, None] + 0.5 * (x + 1.0))).ravel())
                        .to(DEV))
        z, y, x = torch.meshgrid(axes[2], axes[1], axes[0], indexing="ij")
        return x, y, z


class _Schwarz:
    """Additive Schwarz on one grid: each element's points and `ov` layers of its face neighbours."""

    def __init__(self, g, ov=2):
        self.g = g
        n, N = g.n, g.N
        x = _lgl(N)[0]
        delta = 1.0 + x[ov]

        def phi(v):
            v = np.asarray(v)
            return np.where(np.abs(v) <= 1, (15 * v - 10 * v**3 + 3 * v**5) / 8, np.sign(v))

        def w1(v):
            return 0.5 * (phi((v + 1) / delta) - phi((v - 1) / delta))

        self.groups = {}
        code = lambda d, c: (min(c, 2), min(n[d] - 1 - c, 2))  # noqa: E731
        for ez in range(n[2]):
            for ey in range(n[1]):
                for ex in range(n[0]):
                    self.groups.setdefault((code(0, ex), code(1, ey), code(2, ez)), []).append((ex, ey, ez))
        # 1-D factors of the weights at every global point: own, and towards the lower / upper neighbour
        self.f = []
        for d in range(3):
            a, lo, hi = [], [], []
            for e in range(n[d]):
                has = (e > 0, e + 1 < n[d])
                a.append(0.5 * ((phi((x + 1) / delta) if has[0] else 1.0) - (phi((x - 1) / delta) if has[1] else -1.0))
                         * np.ones(N))
                lo.append(w1(x + 2) if has[0] else np.zeros(N))
                hi.append(w1(x - 2) if has[1] else np.zeros(N))
            self.f.append(tuple(torch.from_numpy(np.concatenate(v)).to(DEV) for v in (a, lo, hi)))
        self.ov, self.built = ov, {}

    def points(self, e):
        """Global (x, y, z) indices of the points of element e's subdomain and their weights."""
        n, N, ov = self.g.n, self.g.N, self.ov
        r = np.arange(N)
        k, j, i = (v.ravel() for v in np.meshgrid(r, r, r, indexing="ij"))
        base = np.stack([i, j, k])
        origin = np.array(e)[:, None] * N
        parts, slots = [origin + base], [np.zeros(N**3, int)]
        for f in range(6):
            d, side = divmod(f, 2)
            c = e[d] + (1 if side else -1)
            if not 0 <= c < n[d]:
                continue
            keep = base[:, (base[d] if side else N - 1 - base[d]) < ov]
            at = np.array(e)
            at[d] = c
            parts.append(at[:, None] * N + keep)
            slots.append(np.full(keep.shape[1], 1 + 2 * d + (1 - side)))  # the neighbour sees e across that face
        p = torch.from_numpy(np.concatenate(parts, axis=1)).to(DEV)
        s = torch.from_numpy(np.concatenate(slots)).to(DEV)
        (ax, lx, hx), (ay, ly, hy), (az, lz, hz) = self.f
        a = [ax[p[0]], ay[p[1]], az[p[2]]]
        B = [(lx + hx)[p[0]], (ly + hy)[p[1]], (lz + hz)[p[2]]]
        one = [[lx[p[0]], hx[p[0]]], [ly[p[1]], hy[p[1]]], [lz[p[2]], hz[p[2]]]]
        w = torch.where(s == 0, a[0] * a[1] * a[2], 0.0)
        for d in range(3):
            q, t = (d + 1) % 3, (d + 2) % 3
            rest = a[q] * a[t] + (B[q] * a[t] + a[q] * B[t]) / 2 + B[q] * B[t] / 3
            for side in range(2):
                w = w + torch.where(s == 1 + 2 * d + side, one[d][side] * rest, 0.0)
        return p, w

    def _group(self, key):
        if key not in self.built:
            A, m = self.g.A, self.g.m
            members = self.groups[key]
            p, w = self.points(members[0])
            same = [p[d][:, None] == p[d][None, :] for d in range(3)]
            S = torch.zeros(p.shape[1], p.shape[1], dtype=torch.float64, device=DEV)
            for d in range(3):
                q, t = (d + 1) % 3, (d + 2) % 3
                S += A[d][p[d][:, None], p[d][None, :]] * same[q] * same[t] * (m[q][p[q]] * m[t][p[t]])
            shift = torch.tensor(members, device=DEV).T[:, :, None] - torch.tensor(members[0], device=DEV)[:, None, None]
            at = p[:, None, :] + self.g.N * shift  # [3, members, points]
            nx, ny = self.g.n[0] * self.g.N, self.g.n[1] * self.g.N
            self.built[key] = (torch.linalg.cholesky(0.5 * (S + S.T)), at[0] + nx * (at[1] + ny * at[2]), w)
        return self.built[key]

    def smooth(self, b, u, steps):
        for _ in range(steps):
            r = (b - self.g.apply(u)).reshape(-1)
            du = torch.zeros_like(r)
            for key in self.groups:
                L, at, w = self._group(key)
                du.index_add_(0, at.reshape(-1), (w * torch.cholesky_solve(r[at].T, L).T).reshape(-1))
            u = u + du.reshape(u.shape)
        return u


def _transfer(nf, nc, N):
    """1-D prolongation matrix from nc to nf elements."""
    x = _lgl(N)[0]
    if nf == nc:
        return torch.eye(nf * N, dtype=torch.float64, device=DEV)
    halves = [_interp(x, 0.5 * (x - 1.0)), _interp(x, 0.5 * (x + 1.0))]
    P = np.zeros((nf * N, nc * N))
    for e in range(nf):
        P[e * N:(e + 1) * N, (e // 2) * N:(e // 2 + 1) * N] = halves[e % 2]
    return torch.from_numpy(P).to(DEV)


def _vcycle(c, b):
    lower, upper, n = _box(c)
    grids = [_Grid(lower, upper, m, c["N"], c["neumann"]) for m in _levels(n, 0)]
    smoothers = [_Schwarz(g) for g in grids]
    P = [[_transfer(grids[i].n[d], grids[i + 1].n[d], c["N"]) for d in range(3)] for i in range(len(grids) - 1)]
    bs, us = [b], []
    for i, g in enumerate(grids):
        last = i == len(grids) - 1
        us.append(smoothers[i].smooth(bs[i], torch.zeros_like(bs[i]), 6 if last else 3))
        if not last:
            bs.append(g.along(*(p.T for p in P[i]), bs[i] - g.apply(us[i])))
    for i in range(len(grids) - 2, -1, -1):
        us[i] = smoothers[i].smooth(bs[i], us[i] + grids[i].along(*P[i], us[i + 1]), 3)
    return us[0]


def _puncture(c, seed):
    """Newton's method with conjugate gradients preconditioned by the separable Laplacian's inverse."""
    g = _Grid((-20.0,) * 3, (20.0,) * 3, (c["nx"], c["ny"], c["nz"]), c["N"])
    X = g.coordinates()
    inv_alpha, Abar = 0.0, [[0.0] * 3 for _ in range(3)]
    for q in _punctures(seed):
        d = [X[i] - q.position[i] for i in range(3)]
        r = torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
        ell = [v / r for v in d]
        Pl = sum(q.momentum[i] * ell[i] for i in range(3))
        inv_alpha = inv_alpha + q.mass / (2.0 * r)
        for i in range(3):
            for j in range(3):
                Abar[i][j] = Abar[i][j] + 1.5 / r**2 * (q.momentum[i] * ell[j] + q.momentum[j] * ell[i]
                                                      - (float(i == j) - ell[i] * ell[j]) * Pl)
    alpha = 1.0 / inv_alpha
    beta = alpha**7 * sum(Abar[i][j] ** 2 for i in range(3) for j in range(3)) / 8.0
    M, u = g.mass(), torch.zeros_like(alpha)
    for _ in range(12):
        res = M * beta * (1.0 + alpha * (1.0 + u)) ** -7 - g.apply(u)
        diag = M * 7.0 * alpha * beta * (1.0 + alpha * (1.0 + u)) ** -8
        du, r = torch.zeros_like(u), res
        z = g.solve(r)
        p, rz = z, torch.sum(r * z)
        for _ in range(60):
            q = g.apply(p) + diag * p
            a = rz / torch.sum(p * q)
            du, r = du + a * p, r - a * q
            z = g.solve(r)
            new = torch.sum(r * z)
            if float(new) < 1e-30 * float(torch.sum(res * g.solve(res))):
                break
            p, rz = z + new / rz * p, new
        u = u + du
        if float(du.norm()) < 1e-14 * float(u.norm()):
            break
    return g.vector(u)


def _curved_nodes(c, seed):
    desc = dgg.make_desc(*_box(c), c["N"])
    xyz = _warp(*dgg.host_coordinates(desc))
    return xyz, _coefficient(seed, *xyz)


def _curved_apply(c, seed, u):
    """Strong-form operator on mapped elements with the metric at the nodes."""
    lower, upper, n = _box(c)
    N = c["N"]
    _, w, D = _lgl(N)
    D, w = torch.from_numpy(D).to(DEV), torch.from_numpy(w).to(DEV)
    g = _Grid(lower, upper, n, N)
    xyz = [torch.from_numpy(v).to(DEV) for v in _warp(*(g.vector(t).cpu().numpy() for t in g.coordinates()))]
    K = torch.from_numpy(_coefficient(seed, *(v.cpu().numpy() for v in xyz))).to(DEV)
    shape = (n[2], n[1], n[0], N, N, N)
    node = (5, 4, 3)  # axis of the nodes along x, y, z
    elem = (2, 1, 0)

    def deriv(f, d):
        return torch.movedim(torch.movedim(f, node[d], -1) @ D.T, -1, node[d])

    def face(f, d, side):
        return f.select(node[d], N - 1 if side else 0)

    u, K = u.reshape(shape), K.reshape(shape)
    X = [v.reshape(shape) for v in xyz]
    jac = torch.stack([torch.stack([deriv(X[i], j) for j in range(3)], -1) for i in range(3)], -2)
    J, G = torch.linalg.det(jac), torch.linalg.inv(jac)  # G[..., j, i] = d xi_j / d x_i
    M = J * w[:, None, None] * w[:, None] * w
    B = w[:, None] * w
    du = [deriv(u, j) for j in range(3)]
    grad = [sum(G[..., j, i] * du[j] for j in range(3)) for i in range(3)]
    v = [t.clone() for t in grad]
    faces = []
    for d in range(3):
        for side, s in ((0, -1.0), (1, 1.0)):
            ax = elem[d]
            Gd = [face(G[..., d, i], d, side) for i in range(3)]
            norm = torch.sqrt(sum(t * t for t in Gd))
            nrm = [s * t / norm for t in Gd]
            bf = face(J, d, side) * norm * B
            h = 2.0 / norm

            def outer(f, mine):
                """The neighbour's trace; on the box's boundary `mine`."""
                t = torch.roll(face(f, d, 1 - side), -1 if side else 1, dims=ax).clone()
                t.select(ax, n[d] - 1 if side else 0).copy_(mine.select(ax, n[d] - 1 if side else 0))
                return t

            ui, Ki = face(u, d, side), face(K, d, side)
            ue, Ke = outer(u, -ui), outer(K, Ki)
            gi = sum(nrm[i] * face(grad[i], d, side) for i in range(3))
            ge = sum(nrm[i] * outer(grad[i], face(grad[i], d, side)) for i in range(3))
            other = torch.sqrt(sum(face(G[..., d, i], d, 1 - side) ** 2 for i in range(3)))
            he = torch.roll(2.0 / other, -1 if side else 1, dims=ax).clone()
            he.select(ax, n[d] - 1 if side else 0).copy_(h.select(ax, n[d] - 1 if side else 0))
            star = 0.5 * (Ki * gi + Ke * ge) - 1.5 * N * N / torch.minimum(h, he) * (Ki * ui - Ke * ue)
            for i in range(3):
                face(v[i], d, side).add_(bf * 0.5 * nrm[i] * (ue - ui) / face(M, d, side))
            faces.append((d, side, nrm, bf, star))
    out = -M * sum(G[..., j, i] * deriv(K * v[i], j) for i in range(3) for j in range(3))
    for d, side, nrm, bf, star in faces:
        nv = face(K, d, side) * sum(nrm[i] * face(v[i], d, side) for i in range(3))
        face(out, d, side).sub_(bf * (star - nv))
    return out.reshape(-1)


def exact(case, seed):
    c = case
    kind = c["kind"]
    lower, upper, n = _box(c)
    N = c["N"]
    dof = n[0] * n[1] * n[2] * N**3
    if kind == "puncture":
        return _puncture(c, seed)
    if kind == "curved":
        return _curved_apply(c, seed, _random(dof, seed, 1))
    if kind == "batch":
        out = []
        for i, (m, order) in enumerate(_batch_shapes(c)):
            g = _Grid((-1.0,) * 3, (1.0,) * 3, m, order)
            out.append(g.vector(g.refined_solve(g.mass() * _source(seed, i, *g.coordinates()))))
        return out
    g = _Grid(lower, upper, n, N, c["neumann"])
    if kind == "apply":
        u = _random(dof, seed, 1, torch.float32 if c["precision"] == "fp32" else torch.float64)
        return g.vector(g.apply(g.tensor(u)))
    b = g.mass() * _source(seed, 1, *g.coordinates())
    if kind == "smooth":
        return g.vector(_Schwarz(g).smooth(b, g.tensor(0.01 * _random(dof, seed, 2)), 3))
    if kind == "vcycle":
        return g.vector(_vcycle(c, b))
    return g.vector(g.refined_solve(b))
