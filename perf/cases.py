"""The work this library is used for, as cases that can be timed and compared.

A case is one call of a public entry point: SpMV, the stationary methods, the
Krylov solvers, mixed-precision refinement, the batched solver, and the
differentiable diffusion solve with its backward pass.  Right-hand sides are
U(-1, 1) per node and log k ~ N(0, sigma^2) per cell, as in the library's
benchmark.  Iterations are fixed (tol = 0) so that a pass always does the same
work; refinement and the adjoint run to a tolerance far below the accuracy at
which their results are compared, since that is the only way to call them.
"""
import math
import random

import numpy as np
import torch

import paper_2305_05988_gb300 as hs
from paper_2305_05988_gb300 import inputs

PECLET = 0.5

# Minimum FP64 traffic per unknown of one SpMV, sweep or iteration, every
# vector of the method read or written once (bench.py's accounting), and the
# flops of the 7-point forms.
BYTES = {"spmv": 16.0, "jacobi": 24.0, "gs": 24.0, "cg": 64.0, "bicgstab": 136.0}
FLOPS = {"spmv": 10.0, "jacobi": 9.0, "gs": 9.0, "cg": 19.0, "bicgstab": 48.0}


def listed():
    return [
        # the smallest call: a few sweeps on a coarse 2-D grid (a smoother, a
        # host program's inner step), where launches and host time are all
        {"name": "jacobi_2d_small", "call": "jacobi", "op": "laplacian", "nx": 33, "ny": 17, "nz": 0, "dtype": "f64",
         "its": 20},
        # the 2-D Poisson problem of the benchmark: many short iterations,
        # bound by the grid-wide reductions
        {"name": "cg_2d_128", "call": "cg", "op": "laplacian", "nx": 128, "ny": 128, "nz": 0, "dtype": "f64",
         "its": 100},
        # one operator application on a grid of odd sizes, as a user's own
        # iteration calls it
        {"name": "spmv_3d_ragged", "call": "spmv", "op": "laplacian", "nx": 251, "ny": 187, "nz": 142, "dtype": "f64",
         "its": 1},
        # the 256^3 benchmark's sweeps and solvers, shortened
        {"name": "jacobi_3d_256", "call": "jacobi", "op": "laplacian", "nx": 256, "ny": 256, "nz": 256,
         "dtype": "f64", "its": 20},
        {"name": "gs_3d_256", "call": "gs", "op": "laplacian", "nx": 256, "ny": 256, "nz": 256, "dtype": "f64",
         "its": 20, "mode": "forward"},
        {"name": "cg_3d_256", "call": "cg", "op": "laplacian", "nx": 256, "ny": 256, "nz": 256, "dtype": "f64",
         "its": 20},
        {"name": "bicgstab_3d_256", "call": "bicgstab", "op": "upwind", "nx": 256, "ny": 256, "nz": 256,
         "dtype": "f64", "its": 8},
        # the paper's symmetric sweeps as a smoother on an odd-sized
        # convection-diffusion grid: alternating directions cannot overlap
        {"name": "gs_symmetric_ragged", "call": "gs", "op": "upwind", "nx": 121, "ny": 90, "nz": 67, "dtype": "f64",
         "its": 4, "mode": "symmetric"},
        # the paper's own benchmark matrix (27 points), a slab of its node grid
        {"name": "cg_hpcg27", "call": "cg", "op": "hpcg27", "nx": 128, "ny": 128, "nz": 512, "dtype": "f64",
         "its": 10},
        # FP32-inner / FP64-outer refinement on variable-coefficient
        # diffusion, the whole call to tolerance
        {"name": "mixed_diffusion_256", "call": "mixed", "op": "diffusion", "nx": 256, "ny": 256, "nz": 256,
         "dtype": "f64", "its": 0, "sigma": 1.0, "tol": 1e-12},
        # many systems of mixed sizes in one call (even systems CG, odd
        # systems BiCGStab, 2-D and 3-D)
        {"name": "batch_mixed_sizes", "call": "batch", "systems": 48, "side_max": 128, "layout": 3, "its": 10},
        # forward and backward pass of the differentiable solve
        {"name": "adjoint_64", "call": "adjoint", "op": "diffusion", "nx": 64, "ny": 64, "nz": 64, "dtype": "f64",
         "its": 0, "sigma": 0.5, "tol": 1e-12},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    """One more case of the same calls: 2-D and 3-D grids from 16 nodes a side
    to 256^3 unknowns, any aspect ratio, odd sizes, FP64 and FP32."""
    call = rng.choice(["spmv", "jacobi", "gs", "cg", "bicgstab", "cg", "jacobi", "mixed", "batch", "adjoint"])
    if call == "batch":
        return {"call": "batch", "systems": rng.randint(4, 48), "side_max": _log_int(rng, 24, 128),
                "layout": rng.randint(0, 1 << 20), "its": rng.randint(6, 10)}
    if call in ("mixed", "adjoint"):
        side = [rng.randint(24, 72) for _ in range(3)]
        return {"call": call, "op": "diffusion", "nx": side[0], "ny": side[1], "nz": side[2], "dtype": "f64",
                "its": 0, "sigma": rng.choice([0.5, 1.0]), "tol": 1e-12}
    three = rng.random() < 0.7
    top = 256 if three else 1024
    side = [_log_int(rng, 16, top) for _ in range(3 if three else 2)]
    op = {"spmv": ["laplacian", "upwind", "diffusion"], "jacobi": ["laplacian", "upwind", "diffusion"],
          "gs": ["laplacian", "upwind"], "cg": ["laplacian", "diffusion"] + (["hpcg27"] if three else []),
          "bicgstab": ["upwind"]}[call]
    c = {"call": call, "op": rng.choice(op), "nx": side[0], "ny": side[1], "nz": side[2] if three else 0,
         "dtype": rng.choice(["f64", "f64", "f32"]), "its": 1}
    if call in ("jacobi", "gs"):
        c["its"] = rng.randint(3, 20)
    elif call == "cg":
        c["its"] = rng.randint(6, 20)
    elif call == "bicgstab":
        c["its"] = rng.randint(3, 6)
    if c["op"] == "diffusion":
        c["sigma"] = rng.choice([0.5, 1.0])
    if call == "gs":
        c["mode"] = rng.choice(["forward", "forward", "backward", "symmetric"])
        if c["mode"] == "symmetric":
            c["its"] = min(c["its"], 5)
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _shape(c):
    return (c["nx"], c["ny"], c["nz"]) if c["nz"] else (c["nx"], c["ny"])


def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1000003 + stream)
    return g


def _rhs(N, seed, stream=1):
    return torch.rand(N, dtype=torch.float64, device="cuda", generator=_gen(seed, stream)) * 2.0 - 1.0


def _logk(c, N, seed):
    return torch.randn(N, dtype=torch.float64, device="cuda", generator=_gen(seed, 2)) * c["sigma"]


def _systems(c):
    return inputs.batch_systems(c["systems"], c["layout"], 16, c["side_max"])


def prepare(c, seed):
    """The operator and the vectors a program holds before it calls."""
    if c["call"] == "batch":
        ops, bs = [], []
        systems = _systems(c)
        for s in systems:
            ops.append(hs.Operator.laplacian(s.shape) if s.solver == "cg" else
                       hs.Operator.upwind(s.shape, inputs.upwind_beta(s.shape, s.peclet)))
            bs.append(_rhs(s.N, seed, 16 + s.index))
        return {"c": c, "batch": hs.Batch(ops, [s.solver for s in systems]), "bs": bs}
    shape = _shape(c)
    N = int(np.prod(shape))
    b = _rhs(N, seed)
    if c["call"] == "adjoint":
        w = _rhs(N, seed, 3)
        return {"c": c, "logk": _logk(c, N, seed).requires_grad_(True), "f": b.requires_grad_(True), "w": w}
    if c["op"] == "laplacian":
        A = hs.Operator.laplacian(shape)
    elif c["op"] == "upwind":
        A = hs.Operator.upwind(shape, inputs.upwind_beta(shape, PECLET))
    elif c["op"] == "hpcg27":
        A = hs.Operator.hpcg(shape, 27)
    else:
        A = hs.Operator.diffusion(shape, torch.exp(_logk(c, N, seed)))
    if c["dtype"] == "f32":
        b = b.float()
    return {"c": c, "A": A, "b": b}


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(state):
    c = state["c"]
    call = c["call"]
    if call == "batch":
        xs, infos = state["batch"].solve(state["bs"], tol=0.0, maxit=c["its"])
        return {"x": xs, "iters": np.array([i.iters for i in infos])}
    if call == "adjoint":
        logk, f = state["logk"], state["f"]
        logk.grad = f.grad = None
        u = hs.diffusion_solve(logk, f, _shape(c), tol=c["tol"])
        (state["w"] * u).sum().backward()
        return {"u": u.detach(), "grad_logk": logk.grad, "grad_f": f.grad}
    A, b = state["A"], state["b"]
    if call == "spmv":
        return A.spmv(b)
    if call == "jacobi":
        x, info = hs.jacobi(A, b, maxit=c["its"])
    elif call == "gs":
        x, info = hs.gauss_seidel(A, b, maxit=c["its"], mode=c["mode"])
    elif call == "cg":
        x, info = hs.cg(A, b, tol=0.0, maxit=c["its"])
    elif call == "bicgstab":
        x, info = hs.bicgstab(A, b, tol=0.0, maxit=c["its"])
    else:
        x, info = hs.solve_mixed(A, b, tol=c["tol"])
        return {"x": x}
    return {"x": x, "rel_res": info.rel_res, "iters": info.iters}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(c):
    if c["call"] == "batch":
        by = fl = 0.0
        for s in _systems(c):
            by += BYTES[s.solver] * s.N * c["its"]
            fl += FLOPS[s.solver] * s.N * c["its"]
        return {"bytes": by, "flops": fl}
    N = float(np.prod(_shape(c)))
    half = 0.5 if c["dtype"] == "f32" else 1.0
    if c["call"] in ("mixed", "adjoint"):
        # CG to tolerance takes about 5.5 (sigma 0.5) or 13 (sigma 1)
        # iterations per node of the longest side; FP32 vectors and
        # coefficients: 40 + 16 bytes
        its = (13.0 if c["sigma"] >= 1.0 else 5.5) * max(_shape(c))
        if c["call"] == "mixed":
            return {"bytes": 56.0 * N * its, "flops": 19.0 * N * its}
        return {"bytes": 2 * 96.0 * N * its, "flops": 2 * 19.0 * N * its}
    its = c["its"] * (2 if c.get("mode") == "symmetric" else 1)
    by = BYTES[c["call"]] * half
    if c["op"] == "diffusion":
        by += (8.0 if c["call"] == "spmv" else 32.0 * half)   # k once, or four coefficient arrays
    return {"bytes": by * N * its, "flops": FLOPS[c["call"]] * N * its}


# ---------------------------------------------------------------------------
# the same results in plain torch, 64 bits
# ---------------------------------------------------------------------------

class _Plain:
    """A x on a padded grid: constant couplings, or faces formed from k."""

    def __init__(self, shape, op, k=None, beta=None):
        self.dims = tuple(reversed(tuple(shape) + (1,) * (3 - len(shape))))   # (nz, ny, nx)
        self.nd = len(shape)
        h = [1.0 / (n + 1) for n in shape]
        self.op = op
        if op in ("laplacian", "upwind"):
            self.lo, self.up, self.d = [], [], 0.0
            for q in range(self.nd):
                ih2 = 1.0 / (h[q] * h[q])
                bh = beta[q] / h[q] if op == "upwind" else 0.0
                self.lo.append(-ih2 - bh)
                self.up.append(-ih2)
                self.d += 2.0 * ih2 + bh
        elif op == "diffusion":
            k = k.reshape(self.dims)
            self.lo, self.up, self.d = [], [], torch.zeros_like(k)
            for q in range(self.nd):
                ax, ih2 = 2 - q, 1.0 / (h[q] * h[q])
                n = k.shape[ax]
                a, b = k.narrow(ax, 0, n - 1), k.narrow(ax, 1, n - 1)
                face = 2.0 * a * b / (a + b)
                lo = torch.cat([k.narrow(ax, 0, 1), face], ax) * ih2
                up = torch.cat([face, k.narrow(ax, n - 1, 1)], ax) * ih2
                self.lo.append(-lo)
                self.up.append(-up)
                self.d = self.d + lo + up

    @staticmethod
    def _shift(x, ax, by):
        """x at the neighbour `by` along ax, zero outside."""
        y = torch.zeros_like(x)
        n = x.shape[ax]
        if n > 1:
            if by < 0:
                y.narrow(ax, 1, n - 1).copy_(x.narrow(ax, 0, n - 1))
            else:
                y.narrow(ax, 0, n - 1).copy_(x.narrow(ax, 1, n - 1))
        return y

    def neighbours(self, x):
        y = torch.zeros_like(x)
        for q in range(self.nd):
            y += self.lo[q] * self._shift(x, 2 - q, -1)
            y += self.up[q] * self._shift(x, 2 - q, +1)
        return y

    def apply(self, v):
        x = v.reshape(self.dims)
        if self.op == "hpcg27":
            s = x
            for ax in range(3):
                s = s + self._shift(s, ax, -1) + self._shift(s, ax, +1)
            return (28.0 * x - s).reshape(-1)
        return (self.d * x + self.neighbours(x)).reshape(-1)


def _plain_gs(P, b, its, mode):
    """Lexicographic sweeps, one point hyperplane i + j + k at a time, on a
    grid padded by one node of zeros."""
    nz, ny, nx = P.dims
    dev = b.device
    sy, sz = nx + 2, (nx + 2) * (ny + 2)
    x = torch.zeros(sz * (nz + 2), dtype=torch.float64, device=dev)
    k, j, i = torch.meshgrid(torch.arange(nz, device=dev), torch.arange(ny, device=dev),
                             torch.arange(nx, device=dev), indexing="ij")
    level = (i + j + k).reshape(-1)
    order = torch.argsort(level, stable=True)
    pad = ((k + 1) * sz + (j + 1) * sy + i + 1).reshape(-1)[order]
    bs = b[order]
    counts = torch.bincount(level).tolist()
    cuts = np.concatenate([[0], np.cumsum(counts)]).tolist()
    steps = [1, sy, sz][: P.nd]

    def sweep(levels):
        for s in levels:
            p, r = pad[cuts[s]:cuts[s + 1]], bs[cuts[s]:cuts[s + 1]].clone()
            for q in range(P.nd):
                r -= P.lo[q] * x[p - steps[q]] + P.up[q] * x[p + steps[q]]
            x[p] = r / P.d

    up, down = range(len(counts)), range(len(counts) - 1, -1, -1)
    for _ in range(its):
        if mode in ("forward", "symmetric"):
            sweep(up)
        if mode in ("backward", "symmetric"):
            sweep(down)
    out = torch.empty_like(b)
    out[order] = x[pad]
    return out


def _plain_cg(P, b, its, tol=0.0):
    x, r = torch.zeros_like(b), b.clone()
    p, rr = r.clone(), torch.dot(b, b)
    bb, n = float(rr), 0
    while n < its:
        w = P.apply(p)
        a = rr / torch.dot(p, w)
        x += a * p
        r -= a * w
        new = torch.dot(r, r)
        n += 1
        if tol and n % 16 == 0 and math.sqrt(float(new) / bb) <= tol:
            break
        p = r + (new / rr) * p
        rr = new
    return x, math.sqrt(float(torch.dot(r, r)) / bb)


def _plain_solve(P, b, tol):
    """CG restarted on the true residual."""
    x = torch.zeros_like(b)
    for _ in range(4):
        r = b - P.apply(x)
        if float(r.norm() / b.norm()) < tol:
            break
        x += _plain_cg(P, r, 20000, max(1e-9, 0.2 * tol / float(r.norm() / b.norm())))[0]
    return x


def _plain_bicgstab(P, b, its):
    x, r = torch.zeros_like(b), b.clone()
    rs = r / r.norm()
    p, an = r.clone(), torch.dot(r, rs)
    for n in range(its):
        v = P.apply(p)
        ad = torch.dot(v, rs)
        al = an / ad
        s = r - al * v
        t = P.apply(s)
        om = torch.dot(t, s) / torch.dot(t, t)
        x += al * p + om * s
        r = s - om * t
        new = torch.dot(r, rs)
        if math.sqrt(abs(float(new))) < 1e-5:            # the default restart rule
            rs = r / r.norm()
            p, an = r.clone(), torch.dot(r, rs)
        else:
            p = r + (new / (ad * om)) * (p - om * v)
            an = new
    return x, float(r.norm() / b.norm())


def exact(c, seed):
    if c["call"] == "batch":
        out = []
        for s in _systems(c):
            b = _rhs(s.N, seed, 16 + s.index)
            if s.solver == "cg":
                out.append(_plain_cg(_Plain(s.shape, "laplacian"), b, c["its"])[0])
            else:
                P = _Plain(s.shape, "upwind", beta=inputs.upwind_beta(s.shape, s.peclet))
                out.append(_plain_bicgstab(P, b, c["its"])[0])
        return {"x": out, "iters": None}
    shape = _shape(c)
    N = int(np.prod(shape))
    b = _rhs(N, seed)
    if c["dtype"] == "f32":
        b = b.float().double()
    k = torch.exp(_logk(c, N, seed)) if c["op"] == "diffusion" else None
    beta = inputs.upwind_beta(shape, PECLET) if c["op"] == "upwind" else None
    P = _Plain(shape, c["op"], k, beta)
    if c["call"] == "adjoint":
        u = _plain_solve(P, b, 1e-14)
        lam = _plain_solve(P, _rhs(N, seed, 3), 1e-14)
        kd = k.reshape(P.dims).clone().requires_grad_(True)
        # d/dk of -lam . A(k) u with u and lam held fixed
        dk, = torch.autograd.grad(-torch.dot(lam, _Plain(shape, "diffusion", kd).apply(u)), kd)
        return {"u": u, "grad_logk": dk.reshape(-1) * k, "grad_f": lam}
    if c["call"] == "mixed":
        return {"x": _plain_solve(P, b, 1e-14)}
    if c["call"] == "spmv":
        return P.apply(b)
    if c["call"] == "jacobi":
        x = torch.zeros(P.dims, dtype=torch.float64, device=b.device)
        for _ in range(c["its"]):
            x = (b.reshape(P.dims) - P.neighbours(x)) / P.d
        x = x.reshape(-1)
        rel = float((b - P.apply(x)).norm() / b.norm())
    elif c["call"] == "gs":
        x = _plain_gs(P, b, c["its"], c["mode"])
        rel = float((b - P.apply(x)).norm() / b.norm())
    elif c["call"] == "cg":
        x, rel = _plain_cg(P, b, c["its"])
    else:
        x, rel = _plain_bicgstab(P, b, c["its"])
    return {"x": x, "rel_res": rel, "iters": None}
