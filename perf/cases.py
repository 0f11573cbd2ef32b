"""Measured workloads of the library: whole time steps and single line inversions through the public
classes of ``paper_1611_04214_gb300.molt``.

``listed()`` names the fixed cases and ``draw(rng)`` gives further ones of the same ranges.
``prepare`` builds what a program holds before the call (the seeded state on the GPU and the
solver handle), ``run`` is one pass through the public entry points, ``work`` its unavoidable
traffic and arithmetic, and ``exact`` the same pass in 64 bits with plain torch operations.

Every step case advances a copy of the prepared state, as a program does that tries step sizes or
runs an ensemble, so that each pass does the same work.
"""
import math
from functools import lru_cache

import numpy as np
import torch

from paper_1611_04214_gb300 import molt

TWO_PI = 2.0 * math.pi
STAGES = {"be": 1, "bdf2": 1, "bdf3": 1, "sdirk2": 2, "sdirk3": 3}


def listed():
    return [
        # the 1D Neumann run (256 nodes, eps 0.1), stepped to its tolerance: the smallest call,
        # a latency chain of many iterations
        {"name": "line256_fp64", "kind": "solver", "nx": 256, "ny": 1, "bc": "neumann", "eps": 0.1, "dt": 1e-3,
         "scheme": "be", "precision": "fp64", "M": 4, "tol": 1e-10, "iters": 400, "steps": 4, "state": "smooth"},
        # a small 2D run in 64 bits on the paper's scale of grids, Dirichlet walls, to its tolerance
        {"name": "ch2d_200x136_dirichlet_fp64", "kind": "solver", "nx": 200, "ny": 136, "bc": "dirichlet", "eps": 0.18,
         "dt": 2e-3, "scheme": "sdirk2", "precision": "fp64", "M": 6, "tol": 1e-9, "iters": 400, "steps": 1,
         "state": "smooth"},
        # the 1024^2 Neumann BDF2 run once its state is smooth: a few iterations per step to the
        # tolerance 1e-6, so that the work around the iterations counts as much as they do
        {"name": "ch2d_1024_neumann_fp32", "kind": "solver", "nx": 1024, "ny": 1024, "bc": "neumann", "eps": 0.05,
         "dt": 1e-4, "scheme": "bdf2", "precision": "fp32", "M": 4, "tol": 1e-6, "iters": 400, "steps": 4,
         "state": "smooth"},
        # odd node counts with walls (N + 1 nodes for an even N), a capped iteration count
        {"name": "ch2d_1001x777_dirichlet_fp32", "kind": "solver", "nx": 1001, "ny": 777, "bc": "dirichlet",
         "eps": 0.05, "dt": 2e-4, "scheme": "sdirk2", "precision": "fp32", "M": 4, "tol": 1e-30, "iters": 12,
         "steps": 1, "state": "noise"},
        # the same kind of grid in 64 bits
        {"name": "ch2d_1024_periodic_fp64", "kind": "solver", "nx": 1024, "ny": 1024, "bc": "periodic", "eps": 0.05,
         "dt": 1e-4, "scheme": "bdf2", "precision": "fp64", "M": 4, "tol": 1e-30, "iters": 8, "steps": 1,
         "state": "noise"},
        # the headline run: 8192^2 periodic, SDIRK3, 10 iterations per stage
        {"name": "ch2d_8192_sdirk3_fp32", "kind": "solver", "nx": 8192, "ny": 8192, "bc": "periodic", "eps": 0.02,
         "dt": 5e-5, "scheme": "sdirk3", "precision": "fp32", "M": 4, "tol": 1e-30, "iters": 10, "steps": 1,
         "state": "noise"},
        # the three-phase model at 4096^2 on a grid-scale mixture, 10 iterations per step
        {"name": "vch_4096_neumann_fp32", "kind": "vch", "nx": 4096, "ny": 4096, "bc": "neumann", "eps": 0.03,
         "dt": 1e-6, "scheme": "bdf2", "precision": "fp32", "M": 4, "tol": 1e-30, "iters": 10, "steps": 2},
        # independent instances of mixed sizes stepped together
        {"name": "batch48_neumann_fp32", "kind": "batch", "count": 48, "smin": 128, "smax": 1024, "bc": "neumann",
         "scheme": "be", "M": 4, "tol": 1e-30, "iters": 20},
        # the 3D split stage
        {"name": "split3d_256_fp32", "kind": "split3d", "nx": 256, "ny": 256, "nz": 256, "bc": "periodic", "eps": 0.05,
         "dt": 1e-4, "scheme": "be", "M": 4, "tol": 1e-30, "iters": 10},
        # the sixth-order model on many independent lines, and on a grid
        {"name": "fch1d_16384x1024_fp32", "kind": "fch1d", "nx": 1024, "lines": 16384, "bc": "periodic", "eps": 0.18,
         "dt": 0.05, "precision": "fp32", "M": 6, "tol": 1e-30, "iters": 20},
        {"name": "fch2d_2048_fp32", "kind": "fch2d", "nx": 2048, "ny": 2048, "bc": "periodic", "eps": 0.18,
         "dt": 0.05, "precision": "fp32", "M": 6, "tol": 1e-30, "iters": 10},
        # one line inversion along each axis, the building block that the header exports
        {"name": "sweeps_8192x4096_neumann_fp32", "kind": "sweep", "nx": 8192, "ny": 4096, "bc": "neumann", "nu": 0.08,
         "precision": "fp32", "M": 4},
    ]


def _size(rng, lo, hi):
    """A node count spread over the logarithm of [lo, hi], odd ones among them."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if rng.random() < 0.4:
        return n
    step = 64 if n >= 512 else 8
    return min(hi, max(lo, (n + step // 2) // step * step))


def draw(rng):
    kind = rng.choice(["line", "solver32", "solver32", "solver64", "vch", "batch", "split3d", "fch1d", "fch2d", "sweep"])
    bc = rng.choice(["periodic", "neumann", "dirichlet"])
    closed = rng.choice(["periodic", "neumann"])
    M = rng.choice([2, 4, 4, 6])
    eps = round(rng.uniform(0.03, 0.12), 4)
    dt = eps * eps * 10 ** rng.uniform(-2.5, 0.3)
    if kind == "line":
        return {"kind": "solver", "nx": _size(rng, 64, 8192), "ny": 1, "bc": bc, "eps": eps, "dt": dt,
                "scheme": rng.choice(["be", "bdf2", "sdirk2", "sdirk3"]), "precision": rng.choice(["fp32", "fp64"]),
                "M": M, "tol": 1e-30, "iters": rng.randint(8, 60), "steps": rng.randint(1, 4), "state": "noise"}
    if kind in ("solver32", "solver64"):
        hi = 8192 if kind == "solver32" else 2048
        nx, ny = _size(rng, 64, hi), _size(rng, 64, hi)
        return {"kind": "solver", "nx": nx, "ny": ny, "bc": bc, "eps": eps, "dt": dt,
                "scheme": rng.choice(["be", "bdf2", "sdirk2", "sdirk3"]), "precision": "fp" + kind[-2:], "M": M,
                "tol": 1e-30, "iters": rng.randint(4, 10), "steps": 1, "state": "noise"}
    if kind == "vch":
        nx, ny = _size(rng, 128, 4096), _size(rng, 128, 4096)
        return {"kind": "vch", "nx": nx, "ny": ny, "bc": closed, "eps": 0.03, "dt": 1e-6 * 10 ** rng.uniform(-0.5, 0.5),
                "scheme": rng.choice(["be", "bdf2"]), "precision": "fp32", "M": M, "tol": 1e-30,
                "iters": rng.randint(4, 10), "steps": rng.randint(1, 2)}
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(4, 64), "smin": rng.randint(64, 200), "smax": rng.randint(400, 1024),
                "bc": bc, "scheme": rng.choice(["be", "bdf2"]), "M": M, "tol": 1e-30, "iters": rng.randint(8, 20)}
    if kind == "split3d":
        return {"kind": "split3d", "nx": _size(rng, 48, 320), "ny": _size(rng, 48, 320), "nz": _size(rng, 48, 320),
                "bc": closed, "eps": eps, "dt": dt, "scheme": rng.choice(["be", "bdf2"]), "M": M, "tol": 1e-30,
                "iters": rng.randint(4, 10)}
    if kind == "fch1d":
        nx = _size(rng, 128, 8192)
        return {"kind": "fch1d", "nx": nx, "lines": max(1, min(_size(rng, 1, 16384), 16777216 // nx)), "bc": closed,
                "eps": 0.18, "dt": 0.05, "precision": rng.choice(["fp32", "fp32", "fp64"]), "M": M, "tol": 1e-30,
                "iters": rng.randint(5, 20)}
    if kind == "fch2d":
        return {"kind": "fch2d", "nx": _size(rng, 64, 2048), "ny": _size(rng, 64, 2048), "bc": closed, "eps": 0.18,
                "dt": 0.05, "precision": rng.choice(["fp32", "fp32", "fp64"]), "M": M, "tol": 1e-30,
                "iters": rng.randint(4, 10)}
    return {"kind": "sweep", "nx": _size(rng, 64, 8192), "ny": _size(rng, 64, 8192), "bc": bc,
            "nu": 10 ** rng.uniform(-2, 0.6), "precision": rng.choice(["fp32", "fp32", "fp64"]), "M": M}


# ---- inputs ---------------------------------------------------------------------------------------


def _dtype(case):
    return torch.float64 if case.get("precision", "fp32") == "fp64" else torch.float32


def _nodes(n, bc):
    h = TWO_PI / (n if bc == "periodic" else n - 1)
    return torch.arange(n, dtype=torch.float64, device="cuda") * h


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _smooth(shape, bc, g):
    """A few low modes of random amplitude that satisfy the boundary condition, |u| below 0.5."""
    out = torch.zeros(shape, dtype=torch.float64, device="cuda")
    for _ in range(6):
        a = 0.08 * (2.0 * torch.rand((), generator=g, device="cuda", dtype=torch.float64) - 1.0)
        mode = torch.ones((), dtype=torch.float64, device="cuda")
        for axis, n in enumerate(shape):
            if n == 1:
                continue
            k = int(torch.randint(1, 5, (), generator=g, device="cuda"))
            x = _nodes(n, bc) * (1.0 if bc == "periodic" else 0.5)
            f = torch.sin(k * x) if bc == "dirichlet" else torch.cos(k * x)
            mode = mode * f.reshape([-1 if i == axis else 1 for i in range(len(shape))])
        out += a * mode
    return out


def _state(case, shape, seed):
    """The starting field (the physical variable u; Dirichlet walls hold u = -1)."""
    g = _generator(seed)
    bc = case["bc"]
    if case.get("state") == "smooth":
        u = _smooth(shape, bc, g)
        if bc == "dirichlet":
            u = u - 1.0 + 0.5 * torch.ones_like(u)
            bump = torch.ones((), dtype=torch.float64, device="cuda")
            for axis, n in enumerate(shape):
                if n > 1:
                    s = torch.sin(_nodes(n, bc) * 0.5)
                    bump = bump * s.reshape([-1 if i == axis else 1 for i in range(len(shape))])
            u = -1.0 + (u + 1.0) * bump
    else:
        u = 0.1 + 0.05 * torch.randn(shape, generator=g, device="cuda", dtype=torch.float32).double()
    if bc == "dirichlet":
        for axis, n in enumerate(shape):
            if n > 1:
                u.select(axis, 0).fill_(-1.0)
                u.select(axis, n - 1).fill_(-1.0)
    return u.to(_dtype(case)).contiguous()


def _mixture(case, seed):
    """A grid-scale three-phase mixture: random phase fractions at their barycentre of the roots."""
    shape = (case["ny"], case["nx"])
    g = _generator(seed)
    e = [-torch.log(torch.rand(shape, generator=g, device="cuda", dtype=torch.float32).clamp_min(1e-7)).double()
         for _ in range(3)]
    tot = e[0] + e[1] + e[2]
    roots = [(1.0, 0.0), (-0.5, math.sqrt(3.0) / 2.0), (-0.5, -math.sqrt(3.0) / 2.0)]
    u1 = sum(e[i] * roots[i][0] for i in range(3)) / tot
    u2 = sum(e[i] * roots[i][1] for i in range(3)) / tot
    return u1.to(_dtype(case)).contiguous(), u2.to(_dtype(case)).contiguous()


def _instances(case, seed):
    """(nx, ny, Lx, Ly, eps) and dt of every instance: sides at the node spacing of 2 pi / 512.  The
    sizes belong to the case, the fields to the seed."""
    r = np.random.default_rng(case["count"] * 7919 + case["smin"] * 31 + case["smax"])
    inst, dts = [], []
    for _ in range(case["count"]):
        nx, ny = (int(round(math.exp(r.uniform(math.log(case["smin"]), math.log(case["smax"]))) / 8)) * 8 for _ in range(2))
        nx, ny = max(nx, 16), max(ny, 16)
        nx, ny = min(nx, 1024), min(ny, 1024)
        h = TWO_PI / 512
        m = 0 if case["bc"] == "periodic" else 1
        inst.append((nx, ny, h * (nx - m), h * (ny - m), float(r.uniform(0.04, 0.1))))
        dts.append(float(10 ** r.uniform(-5, -3)))
    return inst, dts


def _fch_state(case, seed):
    shape = (case["lines"], case["nx"]) if case["kind"] == "fch1d" else (case["ny"], case["nx"])
    g = _generator(seed)
    x = _nodes(case["nx"], case["bc"]) * (1.0 if case["bc"] == "periodic" else 0.5)
    u = (0.3 * torch.cos(2.0 * x))[None, :] * torch.ones((shape[0], 1), dtype=torch.float64, device="cuda")
    u = u + 0.05 * (2.0 * torch.rand(shape, generator=g, device="cuda", dtype=torch.float32) - 1.0).double()
    return (u - 1.0).to(_dtype(case)).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    common = dict(bc=case["bc"], quad_order=case["M"])
    if kind == "sweep":
        common["precision"] = case["precision"]
        s = molt.Solver(nx=case["nx"], ny=case["ny"], Lx=TWO_PI, Ly=TWO_PI, **common)
        f = (1.0 + torch.rand((case["ny"], case["nx"]), generator=_generator(seed), device="cuda",
                              dtype=torch.float32)).to(_dtype(case))
        return {"case": case, "solver": s, "in": f, "ox": torch.empty_like(f), "oy": torch.empty_like(f)}
    common.update(tol=case["tol"], max_iter=case["iters"])
    if kind == "solver":
        s = molt.Solver(nx=case["nx"], ny=case["ny"], eps=case["eps"], precision=case["precision"], **common)
        u0 = _state(case, (case["ny"], case["nx"]), seed)
        return {"case": case, "solver": s, "u0": [u0], "u": [torch.empty_like(u0)]}
    if kind == "vch":
        s = molt.Solver(nx=case["nx"], ny=case["ny"], eps=case["eps"], precision=case["precision"], **common)
        u0 = list(_mixture(case, seed))
        return {"case": case, "solver": s, "u0": u0, "u": [torch.empty_like(x) for x in u0]}
    if kind == "batch":
        inst, dts = _instances(case, seed)
        b = molt.Batch(inst, **common)
        u0 = torch.cat([_state(case, (ny, nx), seed * 1009 + i).reshape(-1) for i, (nx, ny, *_r) in enumerate(inst)])
        return {"case": case, "solver": b, "dt": dts, "u0": [u0], "u": [torch.empty_like(u0)]}
    if kind == "split3d":
        s = molt.Solver3D(case["nx"], case["ny"], case["nz"], eps=case["eps"], **common)
        u0 = _state(case, (case["nz"], case["ny"], case["nx"]), seed)
        return {"case": case, "solver": s, "u0": [u0], "u": [torch.empty_like(u0)]}
    common["precision"] = case["precision"]
    u0 = _fch_state(case, seed)
    # (the sixth-order solvers carry their Laplacian from step to step; a pass carries it over from
    # the pass before, as the steps of a run do)
    if kind == "fch1d":
        s = molt.Fch1D(case["nx"], case["lines"], eps=case["eps"], **common)
    else:
        s = molt.Fch2D(case["nx"], case["ny"], eps=case["eps"], **common)
    return {"case": case, "solver": s, "u0": [u0], "u": [torch.empty_like(u0)]}


def run(state):
    case = state["case"]
    kind, s = case["kind"], state["solver"]
    if kind == "sweep":
        h = [TWO_PI / (n if case["bc"] == "periodic" else n - 1) for n in (case["nx"], case["ny"])]
        s.helmholtz_apply(0, (h[0] / case["nu"]) ** 2, state["in"], state["ox"])
        s.helmholtz_apply(1, (h[1] / case["nu"]) ** 2, state["in"], state["oy"])
        return [state["ox"], state["oy"]]
    for dst, src in zip(state["u"], state["u0"]):
        dst.copy_(src)
    u = state["u"]
    if kind == "solver":
        s.reset_history()
        for _ in range(case["steps"]):
            s.step(u[0], case["dt"], case["scheme"], raise_on_nonconvergence=False)
    elif kind == "vch":
        s.reset_history()
        for _ in range(case["steps"]):
            s.vch_step(u[0], u[1], case["dt"], case["scheme"], raise_on_nonconvergence=False)
    elif kind == "batch":
        s.step(u[0], state["dt"], case["scheme"], raise_on_nonconvergence=False)
    elif kind == "split3d":
        s.step(u[0], case["dt"], case["scheme"], raise_on_nonconvergence=False)
    else:
        s.step(u[0], case["dt"], raise_on_nonconvergence=False)
    return list(u)


# ---- what a pass cannot do without ----------------------------------------------------------------


def work(case):
    kind, M = case["kind"], case["M"]
    size = 8 if case.get("precision", "fp32") == "fp64" else 4
    sweep = 2 * 2 * (M + 1) + 4 + 1        # two local integrals, two recurrences, their sum
    if kind == "sweep":
        pts = case["nx"] * case["ny"]
        return {"bytes": 3 * pts * size, "flops": 2 * pts * sweep}
    if kind == "batch":
        inst, _ = _instances(case, 0)
        pts = sum(i[0] * i[1] for i in inst)
    else:
        pts = case["nx"] * case.get("ny", 1) * case.get("nz", 1) * case.get("lines", 1)
    stages = STAGES[case["scheme"]] * case.get("steps", 1) if "scheme" in case else 1
    iters = case["iters"] if case["tol"] < 1e-20 else 4     # converged runs: about what they take
    # an iteration reads the iterate and the stage's right side and writes the iterate; a step
    # reads and writes the state
    comps = 2 if kind == "vch" else 1
    dim = {"fch1d": 1, "split3d": 3}.get(kind, 1 if case.get("ny", 1) == 1 and kind != "batch" else 2)
    per_iter = {1: 2, 2: 6, 3: 12}[dim] * sweep
    return {"bytes": comps * pts * size * (2 + 3 * iters * stages),
            "flops": comps * pts * per_iter * iters * stages}


# ---- the same passes in 64 bits -------------------------------------------------------------------


def _lagrange_weights(nu, offsets, sign):
    """(nu/2) int_0^1 e^{-nu t} l_o(sign t) dt for each offset o, by Gauss-Legendre panels."""
    panels = 1 + int(math.ceil(nu / 8.0))
    xg, wg = np.polynomial.legendre.leggauss(40)
    t = np.concatenate([(p + (xg + 1) / 2) / panels for p in range(panels)])
    w = np.concatenate([wg / 2 / panels for _ in range(panels)])
    kern = w * (nu / 2.0) * np.exp(-nu * t)
    out = []
    for i, xo in enumerate(offsets):
        b = np.ones_like(t)
        for k, xk in enumerate(offsets):
            if k != i:
                b = b * (sign * t - xk) / (xo - xk)
        out.append(float(np.sum(kern * b)))
    return out


@lru_cache(maxsize=64)
def _line(n, c, L, bc, M):
    periodic = bc == "periodic"
    N = n if periodic else n - 1
    nu = (L / N) / math.sqrt(c)
    H = M // 2
    mid = list(range(-H, H + 1))
    wl, wr = _lagrange_weights(nu, mid, -1.0), _lagrange_weights(nu, mid, 1.0)
    walls = []
    if not periodic:
        for j in list(range(H)) + list(range(N - H + 1, N + 1)):
            s = min(max(j - H, 0), N - M)
            offs = [s + k - j for k in range(M + 1)]
            walls.append((j, s, _lagrange_weights(nu, offs, -1.0) if j >= 1 else None,
                          _lagrange_weights(nu, offs, 1.0) if j < N else None))
    return nu, N, wl, wr, walls


def _scan(J, d, reverse):
    """y_j = d y_{j-1} + J_j along the last axis (reversed: from the other end) by doubling."""
    n, s, y, p = J.shape[-1], 1, J, d
    while s < n and p > 1e-19:
        z = y.clone()
        if reverse:
            z[..., : n - s].add_(y[..., s:], alpha=p)
        else:
            z[..., s:].add_(y[..., : n - s], alpha=p)
        y, s, p = z, 2 * s, p * p
    return y


def _H(f, c, L, bc, M, axis):
    """(I - c d_xx)^{-1} by fast convolution along one axis."""
    f = f.movedim(axis, -1).contiguous()
    n = f.shape[-1]
    nu, N, wl, wr, walls = _line(n, float(c), float(L), bc, M)
    H, d = M // 2, math.exp(-nu)
    JL, JR = torch.zeros_like(f), torch.zeros_like(f)
    if bc == "periodic":
        e = torch.cat([f[..., n - H:], f, f[..., :H]], -1)
    else:
        e = torch.cat([f[..., :1].expand(*f.shape[:-1], H), f, f[..., -1:].expand(*f.shape[:-1], H)], -1)
    for o in range(M + 1):
        JL.add_(e[..., o:o + n], alpha=wl[o])
        JR.add_(e[..., o:o + n], alpha=wr[o])
    del e
    for j, s, a, b in walls:
        nodes = f[..., s:s + M + 1]
        zero = torch.zeros((), dtype=f.dtype, device=f.device)
        JL[..., j] = zero if a is None else (nodes * torch.tensor(a, dtype=f.dtype, device=f.device)).sum(-1)
        JR[..., j] = zero if b is None else (nodes * torch.tensor(b, dtype=f.dtype, device=f.device)).sum(-1)
    IL, IR = _scan(JL, d, False), _scan(JR, d, True)
    i = torch.arange(n, dtype=f.dtype, device=f.device)
    mu = math.exp(-nu * N)
    if bc == "periodic":
        ba, bb = IL[..., -1:] / (1 - mu), IR[..., :1] / (1 - mu)
        out = IL + IR + ba * torch.exp(-nu * (i + 1)) + bb * torch.exp(-nu * (n - i))
    else:
        I0, IN = IR[..., :1], IL[..., -1:]
        sg = 1.0 if bc == "neumann" else -1.0
        ba, bb = sg * (I0 + sg * mu * IN) / (1 - mu * mu), sg * (IN + sg * mu * I0) / (1 - mu * mu)
        out = IL + IR + ba * torch.exp(-nu * i) + bb * torch.exp(-nu * (N - i))
    return out.movedim(-1, axis)


class _Grid:
    def __init__(self, bc, M, lengths, dims):
        self.bc, self.M, self.L, self.axes = bc, M, lengths, [a for a, n in enumerate(dims) if n > 1]

    def H(self, f, c, a):
        return _H(f, c, self.L[a], self.bc, self.M, a)

    def minv(self, f, c):
        for a in self.axes:
            f = self.H(f, c, a)
        return f

    def X(self, f, c):
        """M^{-1} P: the remainder of the split product."""
        D = lambda g, a: g - self.H(g, c, a)  # noqa: E731
        if len(self.axes) == 1:
            return torch.zeros_like(f)
        if len(self.axes) == 2:
            return D(D(f, self.axes[0]), self.axes[1])
        z, y, x = self.axes
        dz, dy = D(f, z), D(f, y)
        dyz = D(dz, y)
        return D(dy, x) + D(dz, x) + dyz - 2.0 * D(dyz, x)


def _cs(tau, eps, k=1.0):
    """The two Helmholtz parameters of a stage: k^2 tau^2 - eps^2 tau is the discriminant."""
    if k * k * tau >= eps * eps:
        disc = math.sqrt(k * k * tau * tau - eps * eps * tau)
        return k * tau + disc, k * tau - disc
    c = math.sqrt(eps * eps * tau)
    return c, c


def _iterate(grid, case, tau, eps, vs, Ys, lag, k=1.0):
    ci, co = _cs(tau, eps, k)
    beta = tau / ci
    for _ in range(case["iters"]):
        new = []
        for v, Y, g in zip(vs, Ys, lag(vs, (ci + co) / tau)):
            inner = beta * (grid.minv(g, ci) - g + grid.X(g, ci))
            out = Y + grid.minv(inner, co)
            if len(grid.axes) > 1:
                xi = grid.X(v, ci)
                out = out + grid.X(v, co) + xi - grid.X(xi, co)
            new.append(out)
        res = max(float((a - b).abs().max()) for a, b in zip(new, vs))
        vs = new
        if res < case["tol"]:
            break
    return vs


def _ch_stage(grid, case, tau, eps, r, v):
    ci, co = _cs(tau, eps)
    Y = grid.minv(grid.minv(r, ci), co)
    return _iterate(grid, case, tau, eps, [v], [Y], lambda vs, s: [vs[0] ** 3 - 3 * vs[0] ** 2 + (2 - s) * vs[0]])[0]


def _eta3():
    lo, hi = 0.4, 0.5
    p = lambda x: ((x - 3) * x + 1.5) * x - 1 / 6  # noqa: E731
    for _ in range(200):
        m = 0.5 * (lo + hi)
        lo, hi = (lo, m) if p(lo) * p(m) <= 0 else (m, hi)
    return 0.5 * (lo + hi)


def _ch_steps(grid, case, u, dt, eps, steps):
    v, prev = u.double() + 1.0, None
    for _ in range(steps):
        scheme = case["scheme"]
        if scheme == "be" or (scheme == "bdf2" and prev is None):
            new = _ch_stage(grid, case, dt, eps, v, v)
        elif scheme == "bdf2":
            new = _ch_stage(grid, case, 2 * dt / 3, eps, (4 * v - prev) / 3, v)
        else:
            if scheme == "sdirk2":
                e = 1 - math.sqrt(2) / 2
                A = [[e], [1 - e, e]]
            else:
                e = _eta3()
                A = [[e], [(1 - e) / 2, e], [-(6 * e * e - 16 * e + 1) / 4, (6 * e * e - 20 * e + 5) / 4, e]]
            K, new = [], v
            for row in A:
                r = v + dt * sum(a * k for a, k in zip(row, K)) if K else v
                new = _ch_stage(grid, case, e * dt, eps, r, new)
                K.append((new - r) / (e * dt))
        prev, v = v, new
    return v - 1.0


def _vch_lag(vs, s):
    a, b = vs[0] - 0.5, vs[1] - math.sqrt(3) / 2
    fr, fi = a * (a * a - 3 * b * b) - 1, b * (3 * a * a - b * b)
    zr, zi = a * a - b * b, 2 * a * b
    return [6 * (fr * zr + fi * zi) - s * vs[0], 6 * (fi * zr - fr * zi) - s * vs[1]]


def _fch1d(case, u):
    eps, dt, eta = case["eps"], case["dt"], 1.0
    a = (dt * eps ** 4) ** (1 / 3)
    ce, cf, cp = dt * eta * eps ** 4 / a ** 2, dt * eps ** 2 / a ** 2, dt / a
    H = lambda f: _H(f, a, TWO_PI, case["bc"], case["M"], 1)  # noqa: E731
    vn = u.double() + 1.0
    hv = H(vn)
    h2 = H(hv)
    v, lap = vn, (hv - vn) / a
    for _ in range(case["iters"]):
        f, fp = v * (v * (v - 3) + 2), 3 * v * v - 6 * v + 2
        p = -eps ** 2 * fp * lap + f * fp - eta * eps ** 2 * f
        dv, df, dp = H(v) - v, H(f) - f, H(p) - p
        hdv = H(dv)
        z = h2 + (3 + ce) * (hdv - dv) - 3 * hdv - cf * (H(df) - df) + cp * H(dp)
        v = H(z)
        lap = (v - z) / a
    return v - 1.0


def _fch2d(case, u):
    eps, dt, eta = case["eps"], case["dt"], 1.0
    a = (dt * eps ** 4) ** (1 / 3)
    ce, cf, cp = dt * eta * eps ** 4 / a ** 2, dt * eps ** 2 / a ** 2, dt / a
    Hy = lambda f: _H(f, a, TWO_PI, case["bc"], case["M"], 0)  # noqa: E731
    Hx = lambda f: _H(f, a, TWO_PI, case["bc"], case["M"], 1)  # noqa: E731

    def parts(f):
        hy = Hy(f)
        return Hx(f), hy, Hx(hy)

    def K(f):
        x, y, m = parts(f)
        return 2 * m - x - y, m

    def X(f):
        x, y, m = parts(f)
        return m - x - y + f

    vn = u.double() + 1.0
    m2 = parts(parts(vn)[2])[2]
    W = vn
    x, y, v = parts(W)
    lap, xw = (2 * v - x - y) / a, v - x - y + W
    for _ in range(case["iters"]):
        f, fp = v * (v * (v - 3) + 2), 3 * v * v - 6 * v + 2
        p = -eps ** 2 * fp * lap + f * fp - eta * eps ** 2 * f
        kv = K(v)[0]
        kkv, mkv = K(kv)
        kkf = K(K(f)[0])[0]
        mkp = parts(K(p)[0])[2]
        x2 = X(xw)
        x3 = X(x2)
        W = m2 - 3 * mkv + (3 + ce) * kkv - cf * kkf + cp * mkp + 3 * xw - 3 * x2 + x3
        x, y, v = parts(W)
        lap, xw = (2 * v - x - y) / a, v - x - y + W
    return v - 1.0


def exact(case, seed):
    kind, bc, M = case["kind"], case["bc"], case["M"]
    if kind == "sweep":
        f = (1.0 + torch.rand((case["ny"], case["nx"]), generator=_generator(seed), device="cuda",
                              dtype=torch.float32)).double()
        h = [TWO_PI / (n if bc == "periodic" else n - 1) for n in (case["nx"], case["ny"])]
        return [_H(f, (h[0] / case["nu"]) ** 2, TWO_PI, bc, M, 1), _H(f, (h[1] / case["nu"]) ** 2, TWO_PI, bc, M, 0)]
    if kind == "solver":
        dims = (case["ny"], case["nx"])
        grid = _Grid(bc, M, (TWO_PI, TWO_PI), dims)
        return [_ch_steps(grid, case, _state(case, dims, seed), case["dt"], case["eps"], case["steps"])]
    if kind == "split3d":
        dims = (case["nz"], case["ny"], case["nx"])
        grid = _Grid(bc, M, (TWO_PI,) * 3, dims)
        return [_ch_steps(grid, case, _state(case, dims, seed), case["dt"], case["eps"], 1)]
    if kind == "batch":
        inst, dts = _instances(case, seed)
        if sum(i[0] * i[1] for i in inst) * case["iters"] > 4e8 * 2:
            return None
        out = []
        for i, ((nx, ny, Lx, Ly, eps), dt) in enumerate(zip(inst, dts)):
            u = _state(case, (ny, nx), seed * 1009 + i)
            out.append(_ch_steps(_Grid(bc, M, (Ly, Lx), (ny, nx)), case, u, dt, eps, 1).reshape(-1))
        return [torch.cat(out)]
    if kind == "vch":
        dims = (case["ny"], case["nx"])
        grid = _Grid(bc, M, (TWO_PI, TWO_PI), dims)
        z = (-0.5, -math.sqrt(3) / 2)
        v, prev, eps, dt = [u.double() - z[i] for i, u in enumerate(_mixture(case, seed))], None, case["eps"], case["dt"]
        for _ in range(case["steps"]):
            tau, r = dt, v
            if case["scheme"] == "bdf2" and prev is not None:
                tau, r = 2 * dt / 3, [(4 * a - b) / 3 for a, b in zip(v, prev)]
            ci, co = _cs(tau, eps, 9.0)
            Y = [grid.minv(grid.minv(a, ci), co) for a in r]
            prev, v = v, _iterate(grid, case, tau, eps, v, Y, _vch_lag, 9.0)
        return [v[0] + z[0], v[1] + z[1]]
    if kind == "fch1d":
        return [_fch1d(case, _fch_state(case, seed))]
    return [_fch2d(case, _fch_state(case, seed))]
