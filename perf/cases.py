"""Measured workloads of the library, through its public entry points.

listed()  the workloads by name, draw(rng)  more of the same ranges;
prepare(case, seed)  what a program holds before the call: the mesh object
(stencils, weights, device tables) and its state on the GPU (or in pinned
host memory where the program works from there);
run(state)  one pass, returning everything the pass computes;
work(case)  bytes and flops a pass cannot do without;
exact(case, seed)  the same outputs in plain FP64 torch.

A case is a dict of plain values: "kind" is the call sequence, "mesh" the
mesh family, "n" the lattice points per side, "precision" the library's
precision argument, and the remaining keys the options of that kind.

The FP32 path's results carry single precision, and a program that chose it
for speed keeps them so: the precision-32 cases store their results as float32.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2102_12933_gb300 import autograd, fdu, inputs

GAMMA = 1.4


# --------------------------------------------------------------------------- cases
def listed():
    return [
        # the smallest published run: the 40 x 40 periodic vortex, one FP64 residual (latency and launches)
        dict(name="residual64_vortex40", kind="residual", mesh="vortex", n=40, precision=64),
        # the headline workload: SSP-RK3 steps of the 250k-vertex vortex, in each of the three precisions
        dict(name="steps64_vortex500", kind="steps", mesh="vortex", n=500, precision=64, steps=10),
        dict(name="steps48_vortex500", kind="steps", mesh="vortex", n=500, precision=48, steps=10),
        dict(name="steps32_vortex500", kind="steps", mesh="vortex", n=500, precision=32, steps=20),
        # one FP32 right-hand side for a caller's own integrator: transmissive box with odd sizes, compact coefficients
        dict(name="residual32_riemann301", kind="residual", mesh="riemann", n=301, precision=32, f32_coef=1),
        # the four-quadrant Riemann problem at full size: adaptive FP32 steps with ghost layers and the safeguard
        dict(name="advance32_riemann1000", kind="advance", mesh="riemann", n=1000, precision=32, steps=16),
        # shock-vortex interaction with Dirichlet ghosts at h = 1/4: adaptive FP64 steps with the safeguard
        dict(name="advance64_shock320", kind="advance", mesh="shock", n=320, precision=64, steps=16),
        # a whole small simulation: 2D Sod on 3025 points, degree-5 least squares, adaptive FP64 steps
        dict(name="advance64_sod55", kind="advance", mesh="sod", n=55, precision=64, steps=64, degree=5),
        # many independent meshes of uneven size advanced together, FP32 residual
        dict(name="batch32_16meshes", kind="batch", mesh="batch", n=16, lo=5000, hi=200000, precision=32, steps=10),
        # hybrid triangle / quadrilateral mesh with artificial edges, FP64 residual
        dict(name="residual64_hybrid181", kind="residual", mesh="hybrid", n=181, precision=64),
        # a coupled host program: pinned state in, one FP64 step, state out, every step
        dict(name="host64_vortex250", kind="host", mesh="vortex", n=250, precision=64, steps=4),
        # training-style use: forward steps and the checkpointed adjoint through torch.autograd
        dict(name="autograd64_vortex400", kind="autograd", mesh="vortex", n=400, precision=64, steps=6, every=3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["residual", "residual", "steps", "steps", "advance", "advance", "batch", "host", "autograd"])
    precision = rng.choice([64, 48, 32])
    if kind == "residual":
        mesh = rng.choice(["vortex", "riemann", "hybrid"])
        n = _log_int(rng, 24, 250 if mesh == "hybrid" else 500)
        c = dict(kind=kind, mesh=mesh, n=n, precision=precision, degree=rng.choice([1, 2, 2, 3]))
    elif kind == "steps":
        c = dict(kind=kind, mesh="vortex", n=_log_int(rng, 24, 500), precision=precision, steps=rng.randint(1, 10))
    elif kind == "advance":
        mesh = rng.choice(["riemann", "shock", "sod"])
        n = {"riemann": _log_int(rng, 60, 600), "shock": 2 * _log_int(rng, 40, 200), "sod": _log_int(rng, 30, 80)}[mesh]
        c = dict(kind=kind, mesh=mesh, n=n, precision=precision, steps=rng.randint(5, 24),
                 degree=5 if mesh == "sod" else 2)
    elif kind == "batch":
        c = dict(kind=kind, mesh="batch", n=rng.randint(2, 16), lo=2000, hi=_log_int(rng, 5000, 100000),
                 precision=precision, steps=rng.randint(1, 10))
    elif kind == "host":
        c = dict(kind=kind, mesh="vortex", n=_log_int(rng, 40, 400), precision=precision, steps=rng.randint(1, 4))
    else:
        c = dict(kind=kind, mesh="vortex", n=_log_int(rng, 24, 300), precision=rng.choice([64, 48]),
                 steps=rng.randint(1, 5), every=rng.randint(1, 3))
    if c["precision"] == 32:
        c["f32_coef"] = rng.choice([0, 0, 1])
    return c


# --------------------------------------------------------------------------- inputs
def _mesh_inputs(case, seed):
    """[(mesh, w0, dt)]: one entry, or one per mesh of a batch.  dt is a CFL number of about 1/2."""
    rng = np.random.default_rng([seed, 17])
    n, kind = case["n"], case["mesh"]
    mseed = int(rng.integers(1 << 30))

    def vortex_state(m):
        return inputs.isentropic_vortex(m.xy, beta=float(rng.uniform(1.0, 5.0)), centre=tuple(rng.uniform(3.0, 7.0, 2)))

    if kind == "batch":
        sizes, beta, centre = inputs.batch_sizes(n, case["lo"], case["hi"], seed=mseed)
        # the lattice sizes are the case's own (spread over its range), so that every seed has the same work
        sizes = np.rint(np.sqrt(np.exp(np.linspace(math.log(case["lo"]), math.log(case["hi"]), n)))).astype(int)
        out = []
        for i in range(n):
            m = inputs.torus_lattice(int(sizes[i]), seed=mseed + i)
            out.append((m, inputs.isentropic_vortex(m.xy, beta=float(beta[i]), centre=tuple(centre[i])), 0.08 * m.h))
        return out
    if kind == "vortex":
        m = inputs.torus_lattice(n, seed=mseed)
        w0 = vortex_state(m)
    elif kind == "hybrid":
        m = inputs.hybrid_lattice(n, seed=mseed)
        w0 = vortex_state(m)
    elif kind == "riemann":
        m, w0 = inputs.riemann_case(n, ghost_layers=5, seed=mseed)
    elif kind == "shock":
        m, w0 = inputs.shock_vortex_case(n)
        w0 = inputs.shock_vortex(m.xy, mach_vortex=float(rng.uniform(0.5, 1.0)),
                                 centre=(float(rng.uniform(3.0, 6.0)), float(rng.uniform(-10.0, 10.0))))
    elif kind == "sod":
        m, w0 = inputs.sod_case(n)
        w0 = w0 * (1.0 + 0.01 * rng.uniform(-1.0, 1.0))  # a density level of its own per seed
    else:
        raise ValueError(kind)
    if case["kind"] == "autograd":
        # every component varies over the whole domain, so that the derivative of the nonlinear weights is smooth
        x, y = m.xy[:, 0], m.xy[:, 1]
        ph = rng.uniform(0.0, 10.0, 2)
        for c in range(4):
            w0[:, c] *= 1.0 + 0.02 * np.sin(2 * np.pi * (x + ph[0] + 1.3 * c) / 10) * np.cos(2 * np.pi * (y + ph[1] - 0.7 * c) / 10)
    return [(m, w0, 0.08 * m.h)]


T_END = {"riemann": 0.3, "shock": 3.0, "sod": 0.6}


def _alpha(case):
    return 0.1 if case["kind"] == "advance" and case["mesh"] in ("riemann", "shock") else 0.0


def _eps(case):
    return 1e-6 if case["kind"] == "autograd" else 1e-40


def _cotangent(nv, seed):
    return np.random.default_rng([seed, 23]).standard_normal((nv, 4))


def prepare(case, seed):
    parts = _mesh_inputs(case, seed)
    if case["mesh"] == "batch":
        M = fdu.Batch([(m.xy, m.tri) for m, _, _ in parts], L=10.0, f32_coef=case.get("f32_coef", 0))
        M.set_dt(np.array([dt for _, _, dt in parts]))
        w0 = np.concatenate([w for _, w, _ in parts])
        dt = None
    else:
        m, w0, dt = parts[0]
        M = fdu.Mesh(m.xy, m.tri, m.Lx, m.Ly, lsq_degree=case.get("degree", 2), ghost_donor=m.ghost_donor,
                     positivity_alpha=_alpha(case), weno_eps=_eps(case), f32_coef=case.get("f32_coef", 0))
    s = dict(case=case, M=M, dt=dt, w=torch.tensor(w0, device="cuda"))
    s["out"] = torch.empty_like(s["w"])
    if case["kind"] == "host":
        s["w_in"] = torch.tensor(w0).pin_memory()
        s["w_out"] = torch.empty(w0.shape, dtype=torch.float64).pin_memory().numpy()
    if case["kind"] == "autograd":
        s["w"].requires_grad_(True)
        s["lam"] = torch.tensor(_cotangent(M.nv, seed), device="cuda")
    return s


def _kept(x, precision):
    return x.to(torch.float32) if precision == 32 else x


def run(s):
    case, M, out, p = s["case"], s["M"], s["out"], s["case"]["precision"]
    if case["kind"] == "residual":
        M.set_state(s["w"])
        M.residual(p, out=out)
        return _kept(out, p)
    if case["kind"] == "steps":
        M.set_state(s["w"])
        M.rk_steps(s["dt"], case["steps"], p)
        M.get_state(out=out)
        return _kept(out, p)
    if case["kind"] == "advance":
        M.set_state(s["w"])
        steps, t = M.advance(0.5, T_END[case["mesh"]], p, max_steps=case["steps"])
        M.get_state(out=out)
        return dict(w=_kept(out, p), steps=steps, t=np.float32(t) if p == 32 else t)
    if case["kind"] == "batch":
        M.set_state(s["w"])
        M.batch_rk_steps(case["steps"], p)
        M.get_state(out=out)
        return _kept(out, p)
    if case["kind"] == "host":
        M.set_state(s["w_in"])
        M.rk_step(s["dt"], p)
        M.get_state(out=s["w_out"])
        for _ in range(case["steps"] - 1):
            M.set_state(s["w_out"])
            M.rk_step(s["dt"], p)
            M.get_state(out=s["w_out"])
        return s["w_out"].astype(np.float32) if p == 32 else s["w_out"]
    # autograd: forward steps, then the gradient of <lam, w_T> with respect to w_0
    wT = autograd.RKSteps.apply(s["w"], M, s["dt"], case["steps"], case["every"], p)
    (g,) = torch.autograd.grad(wT, s["w"], s["lam"])
    return dict(w=wT.detach(), grad=g)


# --------------------------------------------------------------------------- work
def _counts(case):
    """Vertices, edges and mean stencil entries per vertex (vertex, edge) of the two-level stencils."""
    n = case["n"]
    if case["mesh"] == "batch":
        v = float(sum(np.rint(np.sqrt(np.exp(np.linspace(math.log(case["lo"]), math.log(case["hi"]), n)))) ** 2))
        return v, 3 * v, 19, 45
    v = float({"riemann": (n + 10) ** 2, "shock": n * (n + 11)}.get(case["mesh"], n * n))
    if case["mesh"] == "hybrid":
        return v, 3.5 * v, 22, 66
    return v, 3 * v, 18 if case["mesh"] in ("shock", "sod") else 19, 42 if case["mesh"] in ("shock", "sod") else 45


def work(case):
    """Per residual evaluation: six ids, four gaps and the normal per edge; id and weights per divergence entry; the
    state read and the result written once.  Flops: 631 per edge and 16 J + 8 K + 70 per vertex (FMA = 2)."""
    V, E, J, K = _counts(case)
    p = 4 if case["precision"] == 32 else 8
    evals = {"residual": 1, "autograd": 3 * case.get("steps", 1)}.get(case["kind"], 3 * case.get("steps", 1))
    byts = E * (24 + 6 * p) + V * (J * (4 + 2 * p) + K * (4 + p) + 64)
    flops = 631 * E + (16 * J + 8 * K + 70) * V
    if case["kind"] == "autograd":  # forward, then the reverse: recomputation and about twice the forward's operations
        byts, flops = 2 * byts, 4 * flops
    return {"bytes": evals * byts, "flops": evals * flops}


# --------------------------------------------------------------------------- the same in plain FP64
def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


class _Plain:
    """The method (arXiv 2102.12933) in FP64 torch: mesh tables and a differentiable residual."""

    def __init__(self, m, degree, eps, alpha):
        self.eps, self.alpha = eps, alpha
        self.L = torch.tensor([m.Lx, m.Ly], dtype=torch.float64, device=_dev())
        self.xy = torch.tensor(m.xy, device=_dev())
        self.nv = m.nv
        donor = None if m.ghost_donor is None else torch.tensor(m.ghost_donor, device=_dev(), dtype=torch.int64)
        self.real = torch.ones(m.nv, dtype=torch.bool, device=_dev()) if donor is None else donor < 0
        self.src = torch.arange(m.nv, device=_dev())
        if donor is not None:
            self.src = torch.where(donor < 0, self.src, donor)
        self._edges(m)
        self._stencils()
        self._coordinates()
        self._divergence(degree)

    def d(self, a, b):
        """Minimum-image displacement from vertex a to vertex b."""
        e = self.xy[b] - self.xy[a]
        return e - self.L * torch.where(self.L > 0, torch.round(e / torch.where(self.L > 0, self.L, 1.0)), 0.0)

    def _edges(self, m):
        if isinstance(m.tri, tuple):  # cell sides and both diagonals of every quadrilateral
            off, vtx = m.tri
            size, pairs = np.diff(off), []
            for k in (3, 4):
                c = vtx[off[:-1][size == k][:, None] + np.arange(k)]
                pairs += [c[:, [i, (i + 1) % k]] for i in range(k)] + ([c[:, [0, 2]], c[:, [1, 3]]] if k == 4 else [])
        else:
            pairs = [m.tri[:, [i, (i + 1) % 3]] for i in range(3)]
        e = np.unique(np.sort(np.concatenate(pairs).astype(np.int64), axis=1), axis=0)
        self.e = torch.tensor(e, device=_dev())
        ne = len(e)
        ends = np.concatenate([e, e[:, ::-1]])
        ids = np.tile(np.arange(ne), 2)
        order = np.lexsort((ends[:, 1], ends[:, 0]))
        a, b, ids = ends[order, 0], ends[order, 1], ids[order]
        cnt = np.bincount(a, minlength=self.nv)
        col = np.arange(2 * ne) - np.repeat(np.cumsum(cnt) - cnt, cnt)
        nb = np.full((self.nv, cnt.max()), -1)
        nbe = np.full((self.nv, cnt.max()), -1)
        nb[a, col], nbe[a, col] = b, ids
        self.nb, self.nbe = torch.tensor(nb, device=_dev()), torch.tensor(nbe, device=_dev())
        t = self.d(self.e[:, 0], self.e[:, 1])
        self.len = t.norm(dim=1)
        self.nrm = t / self.len[:, None]

    def _next(self, frm, at, used):
        """The unused neighbour straightest ahead (first of those within 1e-12); -1 where none is ahead."""
        dv = self.d(frm, at)
        best = torch.full_like(at, -1)
        cbest = torch.zeros(len(at), dtype=torch.float64, device=at.device)
        for j in range(self.nb.shape[1]):
            q = self.nb[at, j]
            free = q >= 0
            for u in used:
                free &= q != u
            ev = self.d(at, q.clamp(min=0))
            c = (dv * ev).sum(1) / (dv.norm(dim=1) * ev.norm(dim=1))
            take = free & ((best < 0) | (c > cbest + 1e-12))
            best, cbest = torch.where(take, q, best), torch.where(take, c, cbest)
        return torch.where(cbest > 0, best, -1)

    def _stencils(self):
        a, b = self.e[:, 0], self.e[:, 1]
        z = lambda v: v.clamp(min=0)  # noqa: E731
        r2 = self._next(a, b, [a, b])
        r3 = self._next(b, z(r2), [a, b, r2])
        l2 = self._next(b, a, [a, b, r2, r3])
        l3 = self._next(a, z(l2), [a, b, r2, r3, l2])
        s = torch.stack([l3, l2, a, b, r2, r3], 1)
        self.valid = (s >= 0).all(1)
        self.s = torch.where(self.valid[:, None], s, s[:, 2:3])

    def _coordinates(self):
        x, w = np.polynomial.legendre.leggauss(16)
        t = torch.tensor(0.5 * (x + 1.0), device=_dev())[:, None, None]
        w = torch.tensor(0.5 * w, device=_dev())[:, None]
        s = self.s
        P = [None] * 6
        P[2] = torch.zeros_like(self.nrm)
        P[3] = self.d(s[:, 2], s[:, 3])
        P[4] = P[3] + self.d(s[:, 3], s[:, 4])
        P[5] = P[4] + self.d(s[:, 4], s[:, 5])
        P[1] = self.d(s[:, 2], s[:, 1])
        P[0] = P[1] + self.d(s[:, 1], s[:, 0])

        def arc(p0, p1, m0, m1):  # cubic Hermite segment
            v = (6 * t * t - 6 * t) * (p0 - p1) + (3 * t * t - 4 * t + 1) * m0 + (3 * t * t - 2 * t) * m1
            return (w * v.norm(dim=2)).sum(0)

        def side(O, A, B, C):
            u = A - O
            tA = u / u.norm(dim=1, keepdim=True) * (B - A).norm(dim=1, keepdim=True)
            tB = 0.5 * (C - A)
            return arc(A, B, tA, tB) / self.len, arc(B, C, tB, C - B) / self.len

        r1, r2 = side(P[2], P[3], P[4], P[5])
        l1, l2 = side(P[3], P[2], P[1], P[0])
        h = torch.full_like(r1, 0.5)
        xi = torch.stack([-0.5 - l1 - l2, -0.5 - l1, -h, h, 0.5 + r1, 0.5 + r1 + r2], 1)
        plain = torch.tensor([-2.5, -1.5, -0.5, 0.5, 1.5, 2.5], dtype=torch.float64, device=_dev())
        xi = torch.where(self.valid[:, None], xi, plain)  # edges without a stencil carry no flux
        self.left = self._weno_tables(xi[:, :5])
        self.right = self._weno_tables(-xi.flip(1)[:, :5])

    @staticmethod
    def _weno_tables(x):
        """Value, slope, curvature at 0 of the three quadratics [E, 3, 3] and the linear weights [E, 3]."""
        val, der, sec = (torch.empty(len(x), 3, 3, dtype=torch.float64, device=x.device) for _ in range(3))
        for k in range(3):
            for j in range(3):
                p, a, b = (x[:, k + (j + i) % 3] for i in range(3))
                den = (p - a) * (p - b)
                val[:, k, j], der[:, k, j], sec[:, k, j] = a * b / den, -(a + b) / den, 2.0 / den
        c = []
        for i in (0, 4):
            l = torch.ones(len(x), dtype=torch.float64, device=x.device)
            for j in range(5):
                if j != i:
                    l = l * -x[:, j] / (x[:, i] - x[:, j])
            c.append(l / val[:, 0 if i == 0 else 2, 0 if i == 0 else 2])
        return val, der, sec, torch.stack([c[0], 1.0 - c[0] - c[1], c[1]], 1)

    @staticmethod
    def _unique_rows(a):
        """Sorted distinct non-negative entries of each row, padded with -1."""
        a = a.sort(dim=1, descending=True).values
        a[:, 1:] = torch.where(a[:, 1:] == a[:, :-1], -1, a[:, 1:])
        a = a.sort(dim=1, descending=True).values
        return a[:, : max(1, int((a >= 0).sum(1).max()))]

    def _divergence(self, degree):
        nv, D = self.nv, self.nb.shape[1]
        z = self.nb.clamp(min=0)
        # edges between two neighbours of a vertex c: for each edge, the common neighbours of its ends
        a, b = self.nb[self.e[:, 0]], self.nb[self.e[:, 1]]
        common = torch.where((a[:, :, None] == b[:, None, :]).any(2) & (a >= 0), a, -1)
        k, j = torch.nonzero(common >= 0, as_tuple=True)
        c = common[k, j]
        order = torch.argsort(c, stable=True)
        c, k = c[order], k[order]
        cnt = torch.bincount(c, minlength=nv)
        col = torch.arange(len(c), device=c.device) - torch.repeat_interleave(torch.cumsum(cnt, 0) - cnt, cnt)
        link = torch.full((nv, int(cnt.max())), -1, device=c.device)
        link[c, col] = k
        both = torch.cat([self.nbe, link], 1)
        self.parts = []
        for o in torch.nonzero(self.real)[:, 0].split(32768):
            have = self.nb[o] >= 0
            V = torch.where(have[:, :, None], self.nb[z[o]], -1).reshape(len(o), -1)
            V = self._unique_rows(torch.where(V == o[:, None], -1, V))
            E = self._unique_rows(torch.where(have[:, :, None], both[z[o]], -1).reshape(len(o), -1))
            self.parts.append((o, V, E, *self._weights(o, V, E, degree)))

    def _weights(self, o, V, E, p):
        """Sum of the a1 and b2 rows of the pseudo-inverse (columns scaled, orthogonalised twice)."""
        def mono(q):
            return torch.stack([q[..., 0] ** i * q[..., 1] ** (t - i) for t in range(1, p + 1) for i in range(t, -1, -1)], -1)

        fo = lambda q: o[:, None].expand_as(q)  # noqa: E731
        vz, ez = V.clamp(min=0), E.clamp(min=0)
        mv = mono(self.d(fo(V), vz)) * (V >= 0)[..., None]
        e0, e1 = self.e[ez, 0], self.e[ez, 1]
        me = mono(self.d(fo(E), e0) + 0.5 * self.d(e0, e1)) * (E >= 0)[..., None]
        n = self.nrm[ez]
        zero = torch.zeros_like(mv)
        A = torch.cat([torch.cat([mv, zero], 2), torch.cat([zero, mv], 2), torch.cat([n[..., :1] * me, n[..., 1:] * me], 2)], 1)
        scale = 1.0 / A.norm(dim=1)
        A = A * scale[:, None, :]
        N = A.shape[2]
        Q, R = torch.zeros_like(A), torch.zeros(len(o), N, N, dtype=torch.float64, device=A.device)
        for c in range(N):
            v = A[:, :, c]
            for _ in range(2):
                h = torch.einsum("bmn,bm->bn", Q[:, :, :c], v)
                R[:, :c, c] += h
                v = v - torch.einsum("bmn,bn->bm", Q[:, :, :c], h)
            R[:, c, c] = v.norm(dim=1)
            Q[:, :, c] = v / R[:, c, c][:, None]
        rhs = torch.zeros(len(o), N, 1, dtype=torch.float64, device=A.device)
        rhs[:, 0, 0] = scale[:, 0]
        rhs[:, N // 2 + 1, 0] = scale[:, N // 2 + 1]
        y = torch.linalg.solve_triangular(R.transpose(1, 2), rhs, upper=False)
        w = torch.einsum("bmn,bn->bm", Q, y[:, :, 0])
        J = V.shape[1]
        return w[:, :J], w[:, J:2 * J], w[:, 2 * J:]

    @staticmethod
    def _prim(w):
        r, u, v = w[..., 0], w[..., 1] / w[..., 0], w[..., 2] / w[..., 0]
        return r, u, v, (GAMMA - 1.0) * (w[..., 3] - 0.5 * r * (u * u + v * v))

    def _fg(self, w):
        r, u, v, p = self._prim(w)
        return (torch.stack([r * u, r * u * u + p, r * u * v, (w[..., 3] + p) * u], -1),
                torch.stack([r * v, r * v * u, r * v * v + p, (w[..., 3] + p) * v], -1))

    def _roe(self, a, b, n):
        """Right and left eigenvectors at the Roe average, (q - c, q, q, q + c), c."""
        ra, ua, va, pa = self._prim(a)
        rb, ub, vb, pb = self._prim(b)
        sa, sb = ra.sqrt(), rb.sqrt()
        avg = lambda x, y: (sa * x + sb * y) / (sa + sb)  # noqa: E731
        u, v, H = avg(ua, ub), avg(va, vb), avg((a[..., 3] + pa) / ra, (b[..., 3] + pb) / rb)
        k = 0.5 * (u * u + v * v)
        c = ((GAMMA - 1.0) * (H - k)).sqrt()
        nx, ny = n[:, 0], n[:, 1]
        q, t = u * nx + v * ny, v * nx - u * ny
        one, zero = torch.ones_like(u), torch.zeros_like(u)
        R = torch.stack([torch.stack([one, u - c * nx, v - c * ny, H - c * q], -1), torch.stack([one, u, v, k], -1),
                         torch.stack([zero, -ny, nx, t], -1), torch.stack([one, u + c * nx, v + c * ny, H + c * q], -1)], -1)
        b1 = (GAMMA - 1.0) / (c * c)
        phi = torch.stack([b1 * k, -b1 * u, -b1 * v, b1], -1)
        psi = torch.stack([q, -nx, -ny, zero], -1) / c[:, None]
        L = torch.stack([0.5 * (phi + psi), torch.stack([one, zero, zero, zero], -1) - phi,
                         torch.stack([-t, -ny, nx, zero], -1), 0.5 * (phi - psi)], 1)
        return R, L, torch.stack([q - c, q, q, q + c], -1), c

    def _weno(self, u, tables):
        """u: characteristic differences from the shared point [E, 5, 4]."""
        val, der, sec, C = tables
        num = den = 0.0
        for k in range(3):
            uk = u[:, k:k + 3]
            v, s, q = (torch.einsum("ej,ejf->ef", T[:, k], uk) for T in (val, der, sec))
            a = C[:, k, None] / (s * s + 13.0 / 12.0 * q * q + self.eps)
            num, den = num + a * v, den + a
        return num / den

    def edge_flux(self, w):
        n, W = self.nrm, w[self.s]
        L1, R1 = W[:, 2], W[:, 3]
        R, L, _, _ = self._roe(L1, R1, n)
        ch = lambda d: torch.einsum("efc,ejc->ejf", L, d)  # noqa: E731
        wl = L1 + torch.einsum("ecf,ef->ec", R, self._weno(ch(W[:, :5] - W[:, 2:3]), self.left))
        wr = R1 + torch.einsum("ecf,ef->ec", R, self._weno(ch(W.flip(1)[:, :5] - W[:, 3:4]), self.right))
        ok = (wl[:, 0] > 0) & (wr[:, 0] > 0) & (self._prim(wl)[3] > 0) & (self._prim(wr)[3] > 0)
        wl, wr = torch.where(ok[:, None], wl, L1), torch.where(ok[:, None], wr, R1)
        R, L, lam, c = self._roe(wl, wr, n)
        delta = 0.1 * c[:, None]
        mag = torch.where(lam.abs() < delta, (lam * lam + delta * delta) / (2 * delta), lam.abs())
        diss = torch.einsum("ecf,ef->ec", R, mag * torch.einsum("efc,ec->ef", L, wr - wl))
        (fl, gl), (fr, gr) = self._fg(wl), self._fg(wr)
        return 0.5 * (n[:, :1] * (fl + fr) + n[:, 1:] * (gl + gr)) - 0.5 * diss

    def residual(self, w):
        f, g = self._fg(w)
        r = self.edge_flux(w)
        out = torch.zeros_like(w)
        for o, V, E, wf, wg, we in self.parts:
            vz, ez = V.clamp(min=0), E.clamp(min=0)
            fo, go = f[o][:, None], g[o][:, None]
            n = self.nrm[ez]
            div = (wf[..., None] * (f[vz] - fo) + wg[..., None] * (g[vz] - go)).sum(1)
            div = div + (we[..., None] * (r[ez] - n[..., :1] * fo - n[..., 1:] * go)).sum(1)
            out = out.index_put((o,), -div)
        return out

    def step(self, w, dt):
        x = w
        for cn, cs in ((0.0, 1.0), (0.75, 0.25), (1.0 / 3.0, 2.0 / 3.0)):
            res = self.residual(x)
            fe = x + dt * res
            if self.alpha > 0:  # largest theta in 1, 1/2, ..., 2^-20, 0 that keeps density and pressure
                p0, done = self._prim(x)[3], torch.zeros(self.nv, dtype=torch.bool, device=w.device)
                fe = x.clone()
                for k in range(21):
                    t = x + 0.5 ** k * dt * res
                    ok = ~done & (t[:, 0] >= self.alpha * x[:, 0]) & (self._prim(t)[3] >= self.alpha * p0)
                    fe, done = torch.where(ok[:, None], t, fe), done | ok
            x = torch.where(self.real[:, None], cn * w + cs * fe, w)[self.src]
        return x

    def max_dt(self, w):
        h = torch.where(self.nbe >= 0, self.len[self.nbe.clamp(min=0)], math.inf).min(1).values
        r, u, v, p = self._prim(w)
        return float((h / ((u * u + v * v).sqrt() + (GAMMA * p / r).sqrt()))[self.real].min())


def exact(case, seed):
    parts = _mesh_inputs(case, seed)
    if case["mesh"] == "batch":
        one = dict(case, kind="steps")
        return torch.cat([_exact_one(one, seed, *part) for part in parts])
    return _exact_one(case, seed, *parts[0])


def _exact_one(case, seed, m, w0, dt):
    P = _Plain(m, case.get("degree", 2), _eps(case), _alpha(case))
    w = torch.tensor(w0, device=_dev())[P.src]
    kind, steps = case["kind"], case.get("steps", 0)
    if kind == "residual":
        return P.residual(w)
    if kind == "advance":
        t, done, end = 0.0, 0, T_END[case["mesh"]]
        while done < steps and t < end:
            dt = min(0.5 * P.max_dt(w), end - t)
            w, t, done = P.step(w, dt), t + dt, done + 1
        return dict(w=w, steps=None, t=t)
    states = [w]
    for _ in range(steps):
        states.append(P.step(states[-1], dt))
    if kind != "autograd":
        return states[-1].cpu().numpy() if kind == "host" else states[-1]
    g = torch.tensor(_cotangent(m.nv, seed), device=_dev())
    for x in reversed(states[:-1]):
        x = x.clone().requires_grad_(True)
        (g,) = torch.autograd.grad(P.step(x, dt), x, g)
    return dict(w=states[-1], grad=g)
