"""The work a user of this library has it do, as measurable cases.

Every case goes through the public binding (`paper_2409_12483_gb300.capi`): time
loops (`ader_solve`), single steps (`ader_step`), the paper's predictor /
corrector pair (`ader_predict`, `ader_correct`) and the request server, over the
1D, 2D and 3D systems, the schemes and the precision forms that the library has.

    listed()             the named cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  inputs on the GPU and the context a program keeps
    run(state)           one pass; its outputs, whole
    work(case)           bytes and floating-point operations of one pass
    exact(case, seed)    the pass's results by plain torch in 64 bits

`exact` is written from the scheme's equations with dense tensor contractions; it
shares nothing with the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2409_12483_gb300 import capi

GAMMA, CFL = 1.4, 0.4
TWO_PI = 2.0 * math.pi
DEV = "cuda"

# Primitive (rho, u, p) left / right of x = 0.5 of the four classical Riemann problems.
RIEMANN = {1: ((1.000, 0.000, 1.000), (0.125, 0.000, 0.100)),
           2: ((0.445, 0.698, 3.528), (0.500, 0.000, 0.571)),
           3: ((1.000, 1.000, 1.000), (1.000, -1.000, 1.000)),
           4: ((1.000, -1.000, 1.000), (1.000, 1.000, 1.000))}


def listed():
    return [
        # the smallest use: the paper's sine-wave test mesh, advanced a little; launches and latency
        {"name": "dg_n2_100_solve", "kind": "dg", "call": "solve", "degree": 2, "cells": 100,
         "steps": 50, "precision": "fp64"},
        # the paper's two functions (local solution, then corrector) called one after the other on
        # a mesh whose size divides by no tile
        {"name": "dg_n3_20011_parts", "kind": "dg", "call": "parts", "degree": 3, "cells": 20011,
         "steps": 1, "precision": "fp64"},
        # the headline: DG-P5 on 10^5 cells in the device-resident time loop
        {"name": "dg_n5_1e5_solve", "kind": "dg", "call": "solve", "degree": 5, "cells": 100000,
         "steps": 10, "precision": "fp64"},
        # the largest 1D mesh: one DG-P7 step with the CFL time step found on the device
        {"name": "dg_n7_1e6_step", "kind": "dg", "call": "step", "degree": 7, "cells": 1000000,
         "steps": 1, "precision": "fp64"},
        # the fast precision form (FP32 Picard on the correction) on the headline mesh
        {"name": "dg_n5_1e5_incr", "kind": "dg", "call": "solve", "degree": 5, "cells": 100000,
         "steps": 10, "precision": "incr"},
        # finite volumes: WENO5 reconstruction and predictor on 10^6 cells
        {"name": "weno5_1e6_solve", "kind": "weno", "call": "solve", "degree": 4,
         "cells": 1000000, "steps": 4, "precision": "fp64"},
        # shocks: a Sod tube with the subcell limiter and outflow ends
        {"name": "sod_n3_limiter", "kind": "limiter", "degree": 3, "cells": 10007, "steps": 20,
         "test": 1},
        # stiffness-free source terms: the two-component reacting flow
        {"name": "reacting_n5_step", "kind": "reacting", "call": "step", "degree": 5,
         "cells": 100000, "steps": 1, "omega": 1.0},
        # a non-conservative product: a tracer carried by the flow, on a mid-sized mesh
        {"name": "tracer_n3_solve", "kind": "tracer", "call": "solve", "degree": 3,
         "cells": 30011, "steps": 8},
        # 2D: the tensor-product scheme at the degree of the headline
        {"name": "dg2_n5_160_solve", "kind": "dg2", "degree": 5, "nx": 160, "ny": 157, "steps": 2},
        # 3D: the degree most 3D runs take, a large mesh
        {"name": "dg3_n3_48_solve", "kind": "dg3", "degree": 3, "nx": 48, "ny": 47, "nz": 45,
         "steps": 2},
        # serving: independent solves of mixed size and degree, submitted together, host to host
        {"name": "serve_24_mixed", "kind": "serve", "requests": 24, "min_cells": 64,
         "max_cells": 2048, "t_end": 0.002, "precision": "fp64"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    top = max(work(c)["flops"] for c in listed())
    while True:
        kind = rng.choice(["dg", "dg", "dg", "weno", "limiter", "reacting", "tracer", "dg2", "dg2",
                           "dg3", "dg3", "serve"])
        c = {"kind": kind}
        if kind == "dg":
            c["call"] = rng.choice(["solve", "solve", "step", "parts"])
            c["degree"] = rng.randint(1, 7)
            c["cells"] = _log(rng, 60, 1000000)
            c["steps"] = rng.randint(2, 40) if c["call"] == "solve" else 1
            c["precision"] = rng.choice(["fp64", "fp64", "fp64", "incr", "ff", "fp32ff"])
        elif kind == "weno":
            c["call"] = rng.choice(["solve", "step"])
            c["degree"] = rng.choice([2, 4])
            c["cells"] = _log(rng, 300, 1000000)
            c["steps"] = rng.randint(2, 16) if c["call"] == "solve" else 1
            c["precision"] = rng.choice(["fp64", "fp64", "incr"])
        elif kind == "limiter":
            c.update(degree=rng.randint(1, 7), cells=_log(rng, 100, 100000),
                     steps=rng.randint(2, 24), test=rng.randint(1, 4))
        elif kind in ("reacting", "tracer"):
            c["call"] = rng.choice(["solve", "step"])
            c.update(degree=rng.randint(1, 7), cells=_log(rng, 100, 200000))
            c["steps"] = rng.randint(2, 12) if c["call"] == "solve" else 1
            if kind == "reacting":
                c["omega"] = rng.choice([1.0, 10.0])
        elif kind == "dg2":
            c.update(degree=rng.randint(1, 7), nx=_log(rng, 8, 512), ny=_log(rng, 8, 512),
                     steps=rng.randint(1, 6))
        elif kind == "dg3":
            c.update(degree=rng.randint(1, 7), nx=_log(rng, 4, 64), ny=_log(rng, 4, 64),
                     nz=_log(rng, 4, 64), steps=rng.randint(1, 3))
        else:
            c.update(requests=rng.randint(4, 24), min_cells=64, max_cells=_log(rng, 128, 2048),
                     t_end=0.002, precision=rng.choice(["fp64", "incr"]))
        if work(c)["flops"] <= top:
            return c


# --------------------------------------------------------------------------------------
# sizes and work
# --------------------------------------------------------------------------------------

def _dims(c):
    return {"dg2": 2, "dg3": 3}.get(c["kind"], 1)


def _vars(c):
    return {"reacting": 5, "tracer": 4, "dg2": 4, "dg3": 5}.get(c["kind"], 3)


def _cells(c):
    return c.get("cells") or c["nx"] * c["ny"] * c.get("nz", 1)


def _requests(c):
    """(cells, degree) of a serving case's requests: the same for every seed."""
    g = np.random.Generator(np.random.PCG64(12483))
    lo, hi = math.log(c["min_cells"]), math.log(c["max_cells"])
    cells = np.rint(np.exp(g.uniform(lo, hi, size=c["requests"]))).astype(int)
    return list(zip(cells.tolist(), g.integers(1, 8, size=c["requests"]).tolist()))


def _step_flops(degree, dims, M, fv=False):
    """One cell and step, with the two Picard iterations that a tolerance test cannot do
    without (the second one shows that the first was enough)."""
    n, d = degree + 1, dims
    flux = {1: 9, 2: 25, 3: 45}[d]
    first = flux * n ** d + 2 * d * n ** (d + 1) * M + 2 * n ** (d + 1) * M
    second = flux * n ** (d + 1) + (d + 1) * 2 * n ** (d + 2) * M
    traces = 2 * d * 2 * n ** (d + 1) * M
    volume = 0 if fv else flux * n ** (d + 1) + 2 * d * n ** (d + 1) * M + 2 * d * n ** (d + 1) * M
    faces = d * n ** d * 40 + 2 * d * n ** d * M
    weno = 3 * (3 * 2 * n * n + 60) if fv else 0
    return first + second + traces + volume + faces + weno


def work(case):
    c = case
    if c["kind"] == "serve":
        nbytes = flops = 0.0
        for cells, deg in _requests(c):
            steps = math.ceil(c["t_end"] * cells * (2 * deg + 1) * 1.7 / CFL)
            nbytes += 2 * 8.0 * cells * (deg + 1) * 3
            flops += float(cells) * steps * _step_flops(deg, 1, 3)
        return {"bytes": nbytes, "flops": flops}
    d, M, fv = _dims(c), _vars(c), c["kind"] == "weno"
    count = _cells(c) * (1 if fv else (c["degree"] + 1) ** d) * M
    nbytes = 2 * 8.0 * count
    if c.get("call") == "parts":  # q leaves the first call and enters the second
        nbytes += 8.0 * count + 2 * 8.0 * count * (c["degree"] + 1)
    return {"bytes": nbytes,
            "flops": float(_cells(c)) * c["steps"] * _step_flops(c["degree"], d, M, fv)}


# --------------------------------------------------------------------------------------
# inputs (closed-form fields with seeded amplitudes and phases)
# --------------------------------------------------------------------------------------

def _nodes(n):
    return (np.polynomial.legendre.leggauss(n)[0] + 1.0) / 2.0


def _points(n, cells):
    """Coordinates [cells][n] of the Gauss-Legendre nodes on [0, 1], on the GPU."""
    xi = torch.tensor(_nodes(n), dtype=torch.float64, device=DEV)
    return (torch.arange(cells, dtype=torch.float64, device=DEV)[:, None] + xi) / cells


def _modes(rng, count, top):
    return [(float(rng.uniform(0.0, top)), k + 1, float(rng.uniform(0.0, TWO_PI)))
            for k in range(count)]


def _sum(x, modes, fn=torch.sin):
    out = torch.ones_like(x)
    for a, k, ph in modes:
        out = out + a * fn(TWO_PI * k * x + ph)
    return out


def _conserved(rho, vel, p):
    E = p / (GAMMA - 1.0) + 0.5 * rho * sum(v * v for v in vel)
    return torch.stack([rho, *[rho * v for v in vel], E], -1)


def _fields(c, seed):
    """The initial state of a case as a GPU tensor (a list of host arrays for a server)."""
    rng = np.random.default_rng([seed, 7])
    if c["kind"] == "serve":
        out = []
        for cells, deg in _requests(c):
            x = _points(deg + 1, cells)
            u = _conserved(_sum(x, _modes(rng, 3, 0.1 / 3)), [torch.full_like(x, 0.5)],
                           _sum(x, _modes(rng, 3, 0.1 / 3)))
            out.append(u.cpu().numpy())
        return out
    n = c["degree"] + 1
    if c["kind"] == "dg2" or c["kind"] == "dg3":
        # the paper's diagonal sine wave with a second mode, and a smooth shear in the velocities
        d = _dims(c)
        sizes = [c["nx"], c["ny"], c.get("nz")][:d]
        X = []
        for a in range(d):
            shape = [1] * (2 * d)
            shape[d - 1 - a], shape[d + a] = sizes[a], n
            X.append(_points(n, sizes[a]).reshape(shape))
        full = list(reversed(sizes)) + [n] * d
        X = [x.expand(full) for x in X]
        ph = rng.uniform(0.0, TWO_PI, size=2 + d)
        s = sum(X)
        rho = 1.0 + 0.5 * torch.sin(TWO_PI * s + float(ph[0]))
        p = 1.0 + 0.1 * torch.sin(TWO_PI * X[0] + float(ph[1]))
        vel = [1.0 + 0.1 * torch.sin(TWO_PI * X[(a + 1) % d] + float(ph[2 + a])) for a in range(d)]
        return _conserved(rho, vel, p).reshape(-1)
    if c["kind"] == "weno":
        # cell averages: a 5-point Gauss rule over each cell
        xg, wg = np.polynomial.legendre.leggauss(5)
        x = (torch.arange(c["cells"], dtype=torch.float64, device=DEV)[:, None]
             + torch.tensor((xg + 1) / 2, device=DEV)) / c["cells"]
        u = _conserved(_sum(x, _modes(rng, 4, 0.05)), [torch.ones_like(x)], torch.ones_like(x))
        return torch.einsum("cqr,q->cr", u, torch.tensor(wg / 2, device=DEV)).reshape(-1)
    x = _points(n, c["cells"])
    if c["kind"] == "limiter":
        L, R = RIEMANN[c["test"]]
        # the tube's states, each a little off its table value; the jump on the face nearest x = 0.5
        f = 1.0 + 0.05 * rng.uniform(-1.0, 1.0, size=4)
        left = x < (c["cells"] // 2) / c["cells"]
        pick = lambda i, fl, fr: torch.full_like(x, R[i] * fr).masked_fill(left, L[i] * fl)  # noqa: E731
        return _conserved(pick(0, float(f[0]), float(f[1])), [pick(1, 1.0, 1.0)],
                          pick(2, float(f[2]), float(f[3]))).reshape(-1)
    if c["kind"] == "reacting":
        m = _modes(rng, 3, 0.1)
        u = _conserved(_sum(x, m), [torch.full_like(x, 0.5)],
                       _sum(x, [(0.5 * a, k, ph) for a, k, ph in m], torch.cos))
        c1, c2 = 0.5 + 0.3 * torch.sin(TWO_PI * x), 0.2 * torch.cos(TWO_PI * x)
        return torch.cat([u, (u[..., 0] * c1)[..., None], (u[..., 0] * c2)[..., None]], -1).reshape(-1)
    if c["kind"] == "tracer":
        u = _conserved(_sum(x, _modes(rng, 3, 0.1)), [torch.full_like(x, 0.5)],
                       _sum(x, _modes(rng, 3, 0.05)))
        return torch.cat([u, _sum(x, _modes(rng, 3, 0.2))[..., None]], -1).reshape(-1)
    if c["cells"] < 50000:
        # density and pressure waves
        return _conserved(_sum(x, _modes(rng, 3, 0.1)), [torch.full_like(x, 0.5)],
                          _sum(x, _modes(rng, 3, 0.1))).reshape(-1)
    # the advected density modes of the benchmark meshes
    one = torch.ones_like(x)
    return _conserved(_sum(x, _modes(rng, 4, 0.05)), [one], one).reshape(-1)


# --------------------------------------------------------------------------------------
# the passes
# --------------------------------------------------------------------------------------

def prepare(case, seed):
    c = case
    s = {"case": c}
    if c["kind"] == "serve":
        need = sum(capi.Server.request_bytes(deg, cells) for cells, deg in _requests(c))
        s["u0"] = _fields(c, seed)
        s["server"] = capi.Server(pool_bytes=need + (64 << 20), max_slots=64,
                                  precision=c["precision"], cfl=CFL, gamma=GAMMA)
        return s
    s["u0"] = _fields(c, seed)
    if c["kind"] == "dg2":
        s["ctx"] = capi.Context2D(c["nx"], c["ny"], c["degree"])
    elif c["kind"] == "dg3":
        s["ctx"] = capi.Context3D(c["nx"], c["ny"], c["nz"], c["degree"])
    else:
        opt = {"weno": {}, "dg": {},
               "limiter": {"limiter": 1, "bc": "outflow"},
               "reacting": {"system": "reacting", "omega": c.get("omega")},
               "tracer": {"system": "tracer"}}[c["kind"]]
        s["ctx"] = capi.Context(c["cells"], c["degree"], "weno" if c["kind"] == "weno" else "dg",
                                precision=c.get("precision", "fp64"), **opt)
    s["u"] = torch.empty_like(s["u0"])
    if c.get("call") == "parts":
        s["q"] = torch.empty(s["ctx"].predictor_count, dtype=torch.float64, device=DEV)
        s["dt"] = 0.9 * CFL / ((2 * c["degree"] + 1) * c["cells"] * 2.0)
    return s


def run(state):
    c = state["case"]
    if c["kind"] == "serve":
        srv = state["server"]
        ids = [srv.submit(deg, u0, c["t_end"])
               for (cells, deg), u0 in zip(_requests(c), state["u0"])]
        while sum(srv.progress(0.0)):
            pass
        out = [srv.poll(i, want_state=True) for i in ids]
        for i in ids:
            srv.release(i)
        return {"u": [r["u"] for r in out], "steps": [r["steps"] for r in out]}
    ctx, u = state["ctx"], state["u"]
    if c.get("call") == "parts":
        ctx.ader_predict(state["u0"], state["dt"], state["q"])
        ctx.ader_correct(state["u0"], state["q"], state["dt"], u)
        return {"q": state["q"], "u": u}
    if c.get("call") == "step":
        ctx.ader_step(state["u0"], u)
        return {"u": u}
    u.copy_(state["u0"])
    steps, t, _ = ctx.ader_solve(u, max_steps=c["steps"])
    return {"u": u, "steps": steps, "t": t}


# --------------------------------------------------------------------------------------
# the same by plain torch in 64 bits
# --------------------------------------------------------------------------------------

class _Basis:
    """Lagrange basis on the Gauss-Legendre nodes of [0, 1] and the operators built from it."""

    def __init__(self, N):
        n = self.n = N + 1
        self.N = N
        x = _nodes(n)
        w = np.polynomial.legendre.leggauss(n)[1] / 2.0
        bw = np.array([1.0 / np.prod([x[k] - x[j] for j in range(n) if j != k]) for k in range(n)])

        def phi(t):  # [points][k]
            t = np.atleast_1d(t)
            return np.stack([bw[k] * np.prod([t - x[j] for j in range(n) if j != k], axis=0)
                             * np.ones_like(t) for k in range(n)], -1)

        D = np.array([[bw[j] / bw[i] / (x[i] - x[j]) if i != j else 0.0 for j in range(n)]
                      for i in range(n)])
        D -= np.diag(D.sum(1))  # D[i][j] = phi_j'(x_i)
        one, zero = phi(1.0)[0], phi(0.0)[0]
        ups = np.outer(one, one) - D.T * w[None, :]
        Ns = 2 * N + 1
        P = np.stack([Ns * (w / Ns) @ phi((j + x) / Ns) for j in range(Ns)])
        g = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device=DEV)  # noqa: E731
        self.x, self.w, self.D = g(x), g(w), g(D)
        self.one, self.zero = g(one), g(zero)
        self.kap = g(np.linalg.solve(ups, np.diag(w)))
        self.vol = g(D.T * w[None, :] / w[:, None])  # (w_l phi_k'(x_l)) / w_k
        self.P = g(P)
        self.R = g(np.linalg.pinv(P))
        self.Ns = Ns


def _apply(A, x, axis):
    """sum_j A[i][j] x[.. j ..] along `axis`."""
    return torch.movedim(torch.tensordot(A, x, dims=([1], [axis])), 0, axis)


def _dot(a, x, axis):
    return torch.tensordot(a, x, dims=([0], [axis]))


def _pressure(U, d):
    return (GAMMA - 1.0) * (U[..., d + 1] - 0.5 * (U[..., 1:d + 1] ** 2).sum(-1) / U[..., 0])


def _flux(U, a, d):
    p = _pressure(U, d)
    v = U[..., 1 + a] / U[..., 0]
    F = U * v[..., None]
    F[..., 0] = U[..., 1 + a]
    F[..., 1 + a] += p
    F[..., d + 1] += p * v
    return F


def _speed(U, a, d):
    return (U[..., 1 + a] / U[..., 0]).abs() + (GAMMA * _pressure(U, d) / U[..., 0]).sqrt()


def _rusanov(A, B, a, d):
    s = torch.maximum(_speed(A, a, d), _speed(B, a, d))[..., None]
    return 0.5 * (_flux(A, a, d) + _flux(B, a, d)) - 0.5 * s * (B - A)


class _Scheme:
    """One system on one mesh: u has shape [cells (z, y, x)] + [n] * d + [M]."""

    def __init__(self, kind, N, sizes, omega=0.0, outflow=False, limiter=False):
        self.kind, self.d, self.sizes = kind, len(sizes), sizes
        self.b = _Basis(N)
        self.N, self.n = N, N + 1
        self.h = [1.0 / s for s in sizes]
        self.om2, self.outflow, self.limiter = omega * omega, outflow, limiter
        self.sub = _Basis(1) if limiter else None

    def flux(self, U, a):
        d = self.d
        F = _flux(U, a, d)
        if self.kind == "tracer":
            F[..., 3] = 0.0
        return F

    def source(self, q):
        S = torch.zeros_like(q)
        S[..., 3] = q[..., 4]
        S[..., 4] = -self.om2 * q[..., 3]
        return S

    def speed_h(self, U):
        return torch.stack([_speed(U, a, self.d) / self.h[a] for a in range(self.d)]).max()

    def dt(self, u):
        if self.kind == "weno":
            return float(CFL / self.speed_h(u))
        v = u
        for a in range(self.d):
            v = _apply(self.b.P, v, self.d + a)
        return float(CFL / (self.d * (2 * self.N + 1)) / self.speed_h(v))

    def predict(self, u, dt, b=None, lam=None):
        """q[tau][...]: the Picard iteration to its fixed point."""
        b, d = b or self.b, self.d
        lam = lam or [dt / h for h in self.h]
        q = u[None].expand(b.n, *u.shape).clone()
        last = math.inf
        for it in range(4 * b.n + 24):
            s = 0.0
            for a in range(d):
                s = s + lam[a] * _apply(b.D, self.flux(q, a), 1 + d + a)
            if self.kind == "reacting":
                s = s - dt * self.source(q)
            if self.kind == "tracer":
                s[..., 3] += lam[0] * q[..., 1] / q[..., 0] * _apply(b.D, q[..., 3], 2)
            new = u[None] - _apply(b.kap, s, 0)
            move = float((new - q).abs().max())
            q = new
            if move <= 2e-16 or (move >= 0.5 * last and move < 1e-13):
                break
            last = move
        return q

    def neighbours(self, qR, qL, u, a):
        """Both sides of every low face along direction a (1D outflow: also the last one)."""
        axis = 1 + self.d - 1 - a
        if not self.outflow:
            return torch.roll(qR, 1, axis), qL
        w = self.b.w
        gl = torch.einsum("k,kr->r", w, u[0]).expand_as(qL[:, :1])
        gr = torch.einsum("k,kr->r", w, u[-1]).expand_as(qR[:, :1])
        return torch.cat([gl, qR], 1), torch.cat([qL, gr], 1)

    def correct(self, u, q, dt):
        b, d = self.b, self.d
        new = u.clone()
        self.G = None
        for a in range(d):
            lam, node = dt / self.h[a], 1 + d + a
            Fb = lam * _dot(b.w, self.flux(q, a), 0)
            new += _apply(b.vol, Fb, node - 1)
            A, B = self.neighbours(_dot(b.one, q, node), _dot(b.zero, q, node), u, a)
            G = lam * _dot(b.w, _rusanov(A, B, a, d), 0)
            lo = hi = G
            if self.kind == "tracer":
                G[..., 3] = lam * _dot(b.w, -0.5 * torch.maximum(_speed(A, 0, 1), _speed(B, 0, 1))
                                       * (B[..., 3] - A[..., 3]), 0)
                xs, ws = np.polynomial.legendre.leggauss(3)
                ub = 0.0
                for x, w in zip((xs + 1) / 2, ws / 2):
                    m = A + x * (B - A)
                    ub = ub + w * m[..., 1] / m[..., 0]
                Bt = lam * _dot(b.w, ub * (B[..., 3] - A[..., 3]), 0)
                lo, hi = G.clone(), G.clone()
                lo[..., 3] -= 0.5 * Bt  # the cell on the plus side of the face
                hi[..., 3] += 0.5 * Bt  # the cell on the minus side
            if self.outflow:
                self.G = G
                lo, hi = G[:-1], G[1:]
            else:
                hi = torch.roll(hi, -1, d - 1 - a)
            shape = [1] * (2 * d + 1)
            shape[d + a] = self.n
            new -= ((b.one / b.w).reshape(shape) * hi.unsqueeze(d + a)
                    - (b.zero / b.w).reshape(shape) * lo.unsqueeze(d + a))
        if self.kind == "reacting":
            new += dt * _dot(b.w, self.source(q), 0)
        if self.kind == "tracer":
            new[..., 3] -= dt / self.h[0] * _dot(
                b.w, q[..., 1] / q[..., 0] * _apply(b.D, q[..., 3], 2), 0)
        return new

    # -- the subcell limiter (1D, outflow) --
    def limit(self, u, new, dt):
        b, Ns, s1 = self.b, self.b.Ns, self.sub
        lam = dt / self.h[0]
        v, vs = _apply(b.P, u, 1), _apply(b.P, new, 1)

        def bad(x):
            e = x[..., 2] - 0.5 * x[..., 1] ** 2 / x[..., 0]
            return ~((x[..., 0] > 0) & (e > 0) & torch.isfinite(x[..., 0]) & torch.isfinite(e))

        lo, hi = v.min(1).values, v.max(1).values
        pad = lambda x: torch.cat([x[:1], x, x[-1:]])  # noqa: E731
        lo = torch.minimum(torch.minimum(pad(lo)[:-2], pad(lo)[2:]), lo)
        hi = torch.maximum(torch.maximum(pad(hi)[:-2], pad(hi)[2:]), hi)
        delta = torch.clamp(1e-3 * (hi - lo), min=1e-4)
        out = (vs < (lo - delta)[:, None]) | (vs > (hi + delta)[:, None])
        tr = bad(vs).any(1) | out.any(2).any(1)
        # ADER-WENO2 on every subcell (two ghost subcells at each end)
        V = pad(pad(v.reshape(-1, 3)))
        sl, sr = V[1:-1] - V[:-2], V[2:] - V[1:-1]
        al, ar = (sl * sl + 1e-14) ** -8.0, (sr * sr + 1e-14) ** -8.0
        slope = (al * sl + ar * sr) / (al + ar)
        wn = V[1:-1, None] + slope[:, None] * (s1.x[None, :, None] - 0.5)
        q = self.predict(wn, dt, s1, [Ns * lam])
        F = lam * _dot(s1.w, _rusanov(_dot(s1.one, q, 2)[:, :-1], _dot(s1.zero, q, 2)[:, 1:], 0, 1), 0)
        no = torch.zeros(1, dtype=torch.bool, device=DEV)
        at = torch.cat([no, tr]) | torch.cat([tr, no])
        dG = torch.where(at[:, None], F[::Ns] - self.G, 0.0)
        dgn = new - ((b.one / b.w)[None, :, None] * dG[1:, None]
                     - (b.zero / b.w)[None, :, None] * dG[:-1, None])
        vn = v - Ns * (F[1:] - F[:-1]).reshape(v.shape)
        lim = _apply(b.R, vn, 1)
        mean = vn.mean(1, keepdim=True).expand_as(lim)
        lim = torch.where(bad(_apply(b.P, lim, 1)).any(1)[:, None, None], mean, lim)
        return torch.where(tr[:, None, None], lim, dgn)

    # -- finite volumes --
    def reconstruct(self, v):
        """WENO of degree N from the central, left and right stencils; nodal values."""
        N, n = self.N, self.n
        t = 2.0 * _nodes(n) - 1.0
        V = torch.tensor(np.vander(t, n, increasing=True), device=DEV)
        S = np.zeros((n, n))  # sigma = a S a: all derivatives in xi (d/dxi = 2 d/dt), squared
        tq, wq = np.polynomial.legendre.leggauss(n)
        for a in range(1, n):
            rows = np.array([[math.prod(range(j - a + 1, j + 1)) * x ** (j - a) if j >= a else 0.0
                              for j in range(n)] for x in tq]) * 2.0 ** a
            S += rows.T @ np.diag(wq / 2) @ rows
        S = torch.tensor(S, device=DEV)
        num = den = 0.0
        for start, lin in ((-(N // 2), 1e5), (-N, 1.0), (0, 1.0)):
            A = np.array([[((2 * o + 1.0) ** (j + 1) - (2 * o - 1.0) ** (j + 1)) / (2 * (j + 1))
                           for j in range(n)] for o in range(start, start + n)])
            st = torch.stack([torch.roll(v, -o, 0) for o in range(start, start + n)])
            a = torch.tensordot(torch.tensor(np.linalg.inv(A), device=DEV), st, dims=1)
            sig = (a * torch.tensordot(S, a, dims=1)).sum(0)
            w = lin / (sig + 1e-14) ** 8
            num, den = num + w * a, den + w
        return torch.movedim(torch.tensordot(V, num / den, dims=1), 0, 1)

    def step(self, u, dt):
        if self.kind == "weno":
            q = self.predict(self.reconstruct(u), dt)
            A, B = torch.roll(_dot(self.b.one, q, 2), 1, 1), _dot(self.b.zero, q, 2)
            G = dt / self.h[0] * _dot(self.b.w, _rusanov(A, B, 0, 1), 0)
            return u - (torch.roll(G, -1, 0) - G)
        new = self.correct(u, self.predict(u, dt), dt)
        return self.limit(u, new, dt) if self.limiter else new

    def solve(self, u, t_end=0.0, steps=0):
        t, k = 0.0, 0
        while (not steps or k < steps) and (not t_end or t < t_end):
            dt = self.dt(u)
            clip = t_end and t + dt >= t_end
            if clip:
                dt = t_end - t
            u = self.step(u, dt)
            t, k = (t_end if clip else t + dt), k + 1
        return u, k, t


def exact(case, seed):
    c = case
    u0 = _fields(c, seed)
    if c["kind"] == "serve":
        out = []
        for (cells, deg), u in zip(_requests(c), u0):
            out.append(_Scheme("dg", deg, [cells]).solve(torch.tensor(u, device=DEV), c["t_end"]))
        return {"u": [u.reshape(-1) for u, _, _ in out], "steps": [k for _, k, _ in out]}
    d, n = _dims(c), c["degree"] + 1
    sizes = [c["nx"], c["ny"], c.get("nz")][:d] if d > 1 else [c["cells"]]
    s = _Scheme(c["kind"], c["degree"], sizes, omega=c.get("omega", 0.0),
                outflow=c["kind"] == "limiter", limiter=c["kind"] == "limiter")
    u = u0.reshape(sizes[::-1] + ([] if c["kind"] == "weno" else [n] * d) + [_vars(c)])
    if c.get("call") == "parts":
        dt = 0.9 * CFL / ((2 * c["degree"] + 1) * c["cells"] * 2.0)
        q = s.predict(u, dt)
        return {"q": q.movedim(0, 1).reshape(-1), "u": s.correct(u, q, dt).reshape(-1)}
    if c.get("call") == "step":
        return {"u": s.step(u, s.dt(u)).reshape(-1)}
    u, k, t = s.solve(u, steps=c["steps"])
    return {"u": u.reshape(-1), "steps": k, "t": t}
