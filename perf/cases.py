"""What this library's performance is measured on: the calls its users make.

Each case is one pass through the public binding (``paper_1403_1937_gb300``):
a solve with a new forcing field on a kept handle (plain FP64, mixed with the
Jacobi inner CG, mixed with the multigrid inner CG; 2D and 3D), a batch of
uneven instances, a training step through the autograd layer, path planning
on a distance field, and the FFT perturbation series.  Sizes, spacings,
source counts and hbar follow the workloads module, the tests and the bench;
the tolerances (1e-9 for the mixed solves, as in the tests, 2e-10 with the
multigrid inner solve in 2D, 1e-12 in FP64) are tight enough that two correct
solvers agree to 1e-9 in S, and hbar is where the FP32 inner solves reach
them for every field drawn here (2048^2 with hbar = 10 h and 256^3 with
multigrid and hbar = 5 h stall above 1e-9 on a few of them).

``prepare`` makes the inputs on the GPU from the seed alone; ``exact``
computes the same results in 64 bits with plain torch: a block-tridiagonal
Cholesky elimination of the finite-difference system (2D), a restarted
conjugate-gradient iteration (3D and the largest 2D grids), torch.fft for the
series and the stepwise Euler integration for the paths.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1403_1937_gb300 import autograd, eik

F64 = torch.float64


# ------------------------------------------------------------------ cases
def listed():
    return [
        # the smallest grids of the paper's tests (one source, f from a cost
        # map): a few hundred short iterations, so launch latency decides
        {"name": "fp64_2d_small", "kind": "solve", "mode": "fp64", "nx": 129, "ny": 129, "nz": 1,
         "nsrc": 1, "hb": 1.28, "tol": 1e-12, "heights": False, "phi": False},
        # an ordinary rectangular map in plain FP64 (the default precision and
        # tolerance), several seeds with prescribed values, phi wanted too
        {"name": "fp64_2d_ragged", "kind": "solve", "mode": "fp64", "nx": 733, "ny": 517, "nz": 1,
         "nsrc": 5, "hb": 6.0, "tol": 1e-12, "heights": True, "phi": True},
        # a 3D cost volume (boxes as obstacles) in plain FP64
        {"name": "fp64_3d", "kind": "solve", "mode": "fp64", "nx": 120, "ny": 97, "nz": 85,
         "nsrc": 4, "hb": 4.0, "tol": 1e-12, "heights": False, "phi": False},
        # the grid of the bench's 2048^2 workload: mixed precision, Jacobi inner CG
        {"name": "mixed_2d_2048", "kind": "solve", "mode": "mixed", "nx": 2048, "ny": 2048,
         "nz": 1, "nsrc": 16, "hb": 16.0, "tol": 1e-9, "heights": False, "phi": False},
        # an ordinary mixed solve whose phi spans a wide range (hbar = 4 h):
        # level-set sweeps, odd sizes
        {"name": "mixed_2d_wide", "kind": "solve", "mode": "mixed", "nx": 611, "ny": 733, "nz": 1,
         "nsrc": 3, "hb": 4.0, "tol": 1e-9, "heights": False, "phi": False},
        # the 256^3 workload of the bench: mixed precision, Jacobi inner CG
        {"name": "mixed_3d_256", "kind": "solve", "mode": "mixed", "nx": 256, "ny": 256, "nz": 256,
         "nsrc": 4, "hb": 5.1, "tol": 1e-9, "heights": False, "phi": False},
        # the same two grids with the multigrid inner solve, the library's
        # fastest mode for large grids
        {"name": "mg_2d_2048", "kind": "solve", "mode": "mg", "nx": 2048, "ny": 2048, "nz": 1,
         "nsrc": 16, "hb": 10.235, "tol": 2e-10, "heights": False, "phi": False},
        {"name": "mg_3d_256", "kind": "solve", "mode": "mg", "nx": 256, "ny": 256, "nz": 256,
         "nsrc": 4, "hb": 8.0, "tol": 1e-9, "heights": False, "phi": False},
        # many maps at once: uneven sides 64 .. 1024, hbar 8 h or 12 h, 1 .. 8
        # seeds each, solved as one packed batch
        {"name": "batch_2d", "kind": "batch", "count": 12, "lo": 64, "hi": 1024, "tol": 1e-9},
        # one step of fitting a cost map to travel times at receivers: forward
        # solve and adjoint through the autograd layer (hbar = 0.04: with a
        # much smaller one the FP64 adjoint's own rounding, about 5e-9 of the
        # gradient at hbar = 0.01, would be larger than what is compared)
        {"name": "train_2d_512", "kind": "train", "nx": 512, "ny": 512, "hb": 20.44, "nrecv": 4096,
         "tol": 1e-12},
        # path planning on a solved map: nodal gradient and 4096 Euler paths
        {"name": "paths_2d_2048", "kind": "paths", "nx": 2048, "ny": 2048, "nsrc": 16,
         "npaths": 4096, "max_steps": 8192},
        # the paper's FFT series, six terms
        {"name": "fft_2d_513", "kind": "fft", "nx": 513, "ny": 513, "nsrc": 8, "hbar": 0.08,
         "terms": 6},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fp64_2d", "fp64_3d", "mixed_2d", "mixed_2d", "mixed_3d", "mg_2d", "mg_3d",
                       "batch", "train", "paths", "fft"])
    if kind == "fp64_2d":
        nx, ny = _log_int(rng, 33, 1024), _log_int(rng, 33, 1024)
        return {"kind": "solve", "mode": "fp64", "nx": nx, "ny": ny, "nz": 1,
                "nsrc": rng.randint(1, 8), "hb": round(max(1.28, 0.01 * max(nx, ny)), 3),
                "tol": 1e-12, "heights": rng.random() < 0.3, "phi": rng.random() < 0.3}
    if kind in ("fp64_3d", "mixed_3d", "mg_3d"):
        top = 128 if kind == "fp64_3d" else 256
        d = [_log_int(rng, 24, top) for _ in range(3)]
        return {"kind": "solve", "mode": kind[:-3], "nx": d[0], "ny": d[1], "nz": d[2],
                "nsrc": rng.randint(1, 4),
                "hb": round(rng.uniform(7.0, 10.0) if kind == "mg_3d" else rng.uniform(4.0, 6.0), 3),
                "tol": 1e-12 if kind == "fp64_3d" else 1e-9, "heights": rng.random() < 0.3,
                "phi": rng.random() < 0.3}
    if kind in ("mixed_2d", "mg_2d"):
        nx, ny = _log_int(rng, 64, 2048), _log_int(rng, 64, 2048)
        hb = rng.choice([4.0, 8.0, 10.235]) if max(nx, ny) <= 1024 else 16.0
        return {"kind": "solve", "mode": kind[:-3], "nx": nx, "ny": ny, "nz": 1,
                "nsrc": rng.randint(1, 16), "hb": hb, "tol": 1e-9 if kind == "mixed_2d" else 2e-10,
                "heights": rng.random() < 0.3, "phi": rng.random() < 0.3}
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(4, 12), "lo": 64,
                "hi": _log_int(rng, 128, 1024), "tol": 1e-9}
    if kind == "train":
        nx, ny = _log_int(rng, 96, 512), _log_int(rng, 96, 512)
        return {"kind": "train", "nx": nx, "ny": ny, "hb": round(0.04 * max(nx, ny), 3),
                "nrecv": _log_int(rng, 64, 4096), "tol": 1e-12}
    if kind == "paths":
        return {"kind": "paths", "nx": _log_int(rng, 128, 2048), "ny": _log_int(rng, 128, 2048),
                "nsrc": rng.randint(1, 16), "npaths": _log_int(rng, 16, 4096), "max_steps": 8192}
    return {"kind": "fft", "nx": _log_int(rng, 65, 600), "ny": _log_int(rng, 65, 600),
            "nsrc": rng.randint(5, 10), "hbar": round(rng.uniform(0.08, 0.12), 3),
            "terms": rng.randint(2, 6)}


# ----------------------------------------------------------------- inputs
def _fourier(rng, nx, ny, h):
    """Smooth cost map in [0.5, 1.5]: eight Fourier modes of low wave number,
    min-max normalised (x fastest, shape (ny, nx))."""
    ks = rng.integers(-4, 5, size=(64, 2))
    nk = (ks ** 2).sum(1)
    ks = ks[(nk >= 1) & (nk <= 16)][:8]
    amp, phase = rng.standard_normal(len(ks)), rng.uniform(0, 2 * np.pi, len(ks))
    x = (torch.arange(nx, dtype=F64, device="cuda") * h)[None, :]
    y = (torch.arange(ny, dtype=F64, device="cuda") * h)[:, None]
    g = torch.zeros((ny, nx), dtype=F64, device="cuda")
    for (kx, ky), a, p in zip(ks.tolist(), amp.tolist(), phase.tolist()):
        g += a * torch.cos(p + 2 * math.pi * (kx * x + ky * y))
    lo, hi = g.min(), g.max()
    return torch.clamp(1.0 + 0.5 * (2 * (g - lo) / (hi - lo) - 1), 0.5, 1.5).contiguous()


def _boxes(rng, nx, ny, nz, h):
    """Cost volume: background 1 and 32 axis-aligned boxes in [0.5, 2]."""
    f = torch.ones((nz, ny, nx), dtype=F64, device="cuda")
    ext = [(n - 1) * h for n in (nx, ny, nz)]
    for _ in range(32):
        lo = [rng.uniform(0.0, 0.8) * e for e in ext]
        a, b = zip(*((int(l / h), min(n - 1, int((l + rng.uniform(0.05, 0.3) * e) / h)))
                     for l, e, n in zip(lo, ext, (nx, ny, nz))))
        f[a[2]:b[2] + 1, a[1]:b[1] + 1, a[0]:b[0] + 1] = rng.uniform(0.5, 2.0)
    return f.contiguous()


def _sources(rng, n, k):
    return np.sort(rng.choice(n, size=min(k, n), replace=False)).astype(np.int64)


def _solve_inputs(case, seed):
    rng = np.random.default_rng([1937, seed])
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    h = 1.0 / (max(nx, ny, nz) - 1)
    f = _fourier(rng, nx, ny, h) if nz == 1 else _boxes(rng, nx, ny, nz, h)
    src = _sources(rng, nx * ny * nz, case["nsrc"])
    U = rng.uniform(0.0, 0.05, len(src)) if case["heights"] else np.zeros(len(src))
    dims = (nx, ny) if nz == 1 else (nx, ny, nz)
    return dims, h, case["hb"] * h, f, src, U


def _batch_inputs(case, seed):
    rng = np.random.default_rng([1941, seed])
    # the sizes are the case's, the fields and seeds the seed's
    shape = np.random.default_rng([7, case["count"], case["lo"], case["hi"]])
    out = []
    for _ in range(case["count"]):
        nx, ny = (int(v) for v in shape.integers(case["lo"], case["hi"] + 1, size=2))
        hb, nsrc = float(shape.choice([8.0, 12.0])), int(shape.integers(1, 9))
        h = 1.0 / (max(nx, ny) - 1)
        out.append(((nx, ny), h, hb * h, _fourier(rng, nx, ny, h), _sources(rng, nx * ny, nsrc),
                    np.zeros(nsrc)))
    return out


def _train_inputs(case, seed):
    rng = np.random.default_rng([1942, seed])
    nx, ny = case["nx"], case["ny"]
    h = 1.0 / (max(nx, ny) - 1)
    f = _fourier(rng, nx, ny, h)
    src = _sources(rng, nx * ny, 1)
    pool = np.setdiff1d(np.arange(nx * ny, dtype=np.int64), src)
    recv = np.sort(rng.choice(pool, size=min(case["nrecv"], len(pool)), replace=False))
    # observed travel times: the distance to the source, with noise
    sx, sy = int(src[0]) % nx, int(src[0]) // nx
    T = h * np.hypot(recv % nx - sx, recv // nx - sy) + 0.01 * rng.standard_normal(len(recv))
    return (nx, ny), h, case["hb"] * h, f, src, torch.from_numpy(recv).cuda(), \
        torch.from_numpy(T).cuda()


def _paths_inputs(case, seed):
    """A distance field as a solve returns it: S = -hbar log of a sum of
    exp(-distance / hbar) over the sources."""
    rng = np.random.default_rng([1943, seed])
    nx, ny = case["nx"], case["ny"]
    h = 1.0 / (max(nx, ny) - 1)
    hbar = 0.005
    src = _sources(rng, nx * ny, case["nsrc"])
    x = (torch.arange(nx, dtype=F64, device="cuda") * h)[None, :]
    y = (torch.arange(ny, dtype=F64, device="cuda") * h)[:, None]
    S = None
    for k in src.tolist():
        d = -torch.sqrt((x - (k % nx) * h) ** 2 + (y - (k // nx) * h) ** 2) / hbar
        S = d if S is None else torch.logaddexp(S, d)
    S = (-hbar * S).reshape(-1).contiguous()
    starts = rng.uniform(0, 1, (case["npaths"], 2)) * np.array([(nx - 1) * h, (ny - 1) * h])
    return (nx, ny), h, S, src, torch.from_numpy(starts).cuda()


def _fft_inputs(case, seed):
    rng = np.random.default_rng([1944, seed])
    nx, ny = case["nx"], case["ny"]
    h = 1.0 / (max(nx, ny) - 1)
    return (nx, ny), h, _fourier(rng, nx, ny, h), _sources(rng, nx * ny, case["nsrc"])


def _options(mode, tol):
    if mode == "mg":
        return eik.make_options(precision="mixed", tol=tol, precond="multigrid")
    return eik.make_options(precision=mode, tol=tol)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "solve":
        dims, h, hbar, f, src, U = _solve_inputs(case, seed)
        hd = eik.eik_create(dims, h, hbar, f, src, U, _options(case["mode"], case["tol"]))
        return {"kind": kind, "h": hd, "f": f, "phi": case["phi"]}
    if kind == "batch":
        inst = [SimpleNamespace(dims=d, h=h, hbar=hb, f=f.cpu().numpy(), src_idx=s, src_U=U)
                for d, h, hb, f, s, U in _batch_inputs(case, seed)]
        b = eik.eik_create_batch(inst, _options("mixed", case["tol"]))
        f = torch.from_numpy(np.concatenate([i.f.ravel() for i in inst])).cuda()
        return {"kind": kind, "b": b, "f": f}
    if kind == "train":
        dims, h, hbar, f, src, recv, T = _train_inputs(case, seed)
        layer = autograd.Eikonal(dims, h, hbar, src, precision="mixed", tol=case["tol"])
        return {"kind": kind, "layer": layer, "f": f, "recv": recv, "T": T}
    if kind == "paths":
        dims, h, S, src, starts = _paths_inputs(case, seed)
        return {"kind": kind, "dims": dims, "h": h, "S": S, "src": src, "starts": starts,
                "max_steps": case["max_steps"]}
    dims, h, f, src = _fft_inputs(case, seed)
    return {"kind": kind, "dims": dims, "h": h, "f": f, "src": src, "hbar": case["hbar"],
            "terms": case["terms"]}


# -------------------------------------------------------------------- run
def run(st):
    kind = st["kind"]
    if kind == "solve":
        eik.eik_set_f(st["h"], st["f"])
        S, phi, _ = eik.eik_solve(st["h"], want_phi=st["phi"])
        return (S, phi) if st["phi"] else S
    if kind == "batch":
        eik.eik_set_f_batch(st["b"], st["f"])
        S, _ = eik.eik_solve_batch(st["b"])
        return S
    if kind == "train":
        f = st["f"].detach().requires_grad_(True)
        S = st["layer"](f)
        loss = ((S.reshape(-1)[st["recv"]] - st["T"]) ** 2).sum()
        loss.backward()
        return {"S": S.detach(), "grad": f.grad}
    if kind == "paths":
        G = eik.grad_S(st["S"], st["dims"], st["h"])
        P, L, status = eik.backtrack(G, st["dims"], st["h"], st["starts"], st["src"],
                                     0.5 * st["h"], st["max_steps"], 2.0 * st["h"])
        return {"G": G, "paths": P, "lengths": L, "status": status}
    S, phi, _ = eik.fft_series(st["dims"], st["h"], st["hbar"], st["f"], st["src"], st["terms"])
    return {"S": S, "phi": phi}


# ------------------------------------------------------------------- work
def work(case):
    """One pass reads its inputs and writes its outputs once.  The solves'
    operations count two multigrid-like sweeps over the grid (~100 per node),
    the least that an O(N) method spends; the series its real transforms."""
    kind = case["kind"]
    if kind == "solve":
        n = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": 8 * n * (3 if case["phi"] else 2), "flops": 100 * n}
    if kind == "batch":
        shape = np.random.default_rng([7, case["count"], case["lo"], case["hi"]])
        n = 0
        for _ in range(case["count"]):
            nx, ny = (int(v) for v in shape.integers(case["lo"], case["hi"] + 1, size=2))
            shape.choice([8.0, 12.0]), shape.integers(1, 9)
            n += nx * ny
        return {"bytes": 16 * n, "flops": 100 * n}
    if kind == "train":
        n = case["nx"] * case["ny"]
        return {"bytes": 32 * n, "flops": 200 * n}
    if kind == "paths":
        n = case["nx"] * case["ny"]
        pts = case["npaths"] * (case["max_steps"] + 1)
        return {"bytes": 24 * n + 16 * pts, "flops": 4 * n + 40 * pts // 16}
    n = case["nx"] * case["ny"]
    return {"bytes": 24 * n, "flops": (3 + 2 * case["terms"]) * 4 * n * 2.5 * math.log2(4 * n)}


# ------------------------------------------------------------------ exact
class _System:
    """The finite-difference system of one 2D or 3D grid (half-cell faces) as
    coefficient arrays: diagonal a, edge weights along each axis, Dirichlet
    sources."""

    def __init__(self, dims, h, hbar, f, src, U):
        nx, ny = dims[0], dims[1]
        nz = dims[2] if len(dims) == 3 else 1
        self.shape, self.nd, self.hbar = (nz, ny, nx), len(dims), hbar
        self.c = (hbar / h) ** 2

        def half(n, axis):
            w = torch.ones(n, dtype=F64, device="cuda")
            if n > 1:
                w[0] = w[-1] = 0.5
            return w.reshape([-1 if k == axis else 1 for k in range(3)])

        hz, hy, hx = half(nz, 0), half(ny, 1), half(nx, 2)
        one = torch.ones(self.shape, dtype=F64, device="cuda")
        f = f.reshape(self.shape)
        self.w = hx * hy * hz * one
        src = torch.from_numpy(src).cuda()
        U = torch.from_numpy(np.asarray(U, dtype=np.float64)).cuda()
        self.U_min = U.min()
        free = torch.ones(nz * ny * nx, dtype=F64, device="cuda")
        free[src] = 0.0
        phi0 = torch.zeros(nz * ny * nx, dtype=F64, device="cuda")
        phi0[src] = torch.exp(-(U - self.U_min) / hbar)
        self.src, self.U = src, U
        self.free, self.phi0 = free.reshape(self.shape), phi0.reshape(self.shape)
        self.edge = [self.c * w for w in (hx * hy * one[:-1], hx * hz * one[:, :-1],
                                          hy * hz * one[:, :, :-1])]
        a = self.w * f * f
        for ax, e in enumerate(self.edge):
            if self.shape[ax] > 1:
                a.narrow(ax, 0, e.shape[ax]).add_(e)
                a.narrow(ax, 1, e.shape[ax]).add_(e)
        self.a = a
        self.f = f

    def off(self, v):
        """sum over the neighbours of edge weight times v."""
        out = torch.zeros_like(v)
        for ax, e in enumerate(self.edge):
            k = e.shape[ax]
            if self.shape[ax] > 1:
                out.narrow(ax, 0, k).add_(e * v.narrow(ax, 1, k))
                out.narrow(ax, 1, k).add_(e * v.narrow(ax, 0, k))
        return out

    def S_of(self, phi):
        S = (self.U_min - self.hbar * torch.log(phi)).reshape(-1)
        S[self.src] = self.U
        return S

    # 2D: eliminate one line of nodes after the other; every block is an
    # M-matrix, so the Cholesky steps lose no relative accuracy
    def lines(self):
        a, free = self.a[0], self.free[0]
        ey, ex = self.edge[1][0], self.edge[2][0]
        turn = a.shape[1] > a.shape[0]          # blocks along the shorter axis
        if turn:
            a, free, ey, ex = a.t(), free.t(), ex.t(), ey.t()
        a = torch.where(free > 0, a, torch.ones_like(a))
        ex = ex * free[:, :-1] * free[:, 1:]
        ey = ey * free[:-1] * free[1:]
        inv, prev = [], None
        for k in range(a.shape[0]):
            D = torch.diag(a[k]) - torch.diag(ex[k], 1) - torch.diag(ex[k], -1)
            if prev is not None:
                D = D - ey[k - 1][:, None] * prev * ey[k - 1][None, :]
            prev = torch.cholesky_inverse(torch.linalg.cholesky(D))
            inv.append(prev)
        return turn, ey, inv

    @staticmethod
    def line_solve(fac, b):
        turn, ey, inv = fac
        y = (b.t() if turn else b).clone()
        for k in range(1, y.shape[0]):
            y[k] += ey[k - 1] * (inv[k - 1] @ y[k - 1])
        x = torch.empty_like(y)
        x[-1] = inv[-1] @ y[-1]
        for k in range(y.shape[0] - 2, -1, -1):
            x[k] = inv[k] @ (y[k] + ey[k] * x[k + 1])
        return x.t() if turn else x

    def rhs(self):
        return torch.where(self.free > 0, self.off(self.phi0), self.phi0)

    def solve_lines(self):
        fac = self.lines()
        return fac, self.line_solve(fac, self.rhs()[0])[None]

    # Jacobi-scaled conjugate gradients, restarted from the true residual
    # until every row's residual is 1e-13 of its diagonal term
    def solve_cg(self, tol=1e-13, restarts=40, steps=4000):
        b = self.off(self.phi0) * self.free
        s = self.free / torch.sqrt(self.a)
        x = torch.zeros_like(b)
        A = lambda v: v * self.free - s * self.off(s * v)  # noqa: E731
        bh, best = s * b, math.inf
        for _ in range(restarts):
            r = bh - A(x)
            cw = torch.where((self.free > 0) & (x <= 0), math.inf,
                             (r.abs() / x).masked_fill(self.free == 0, 0.0)).max().item()
            if cw <= tol or (math.isfinite(cw) and cw > 0.5 * best):
                break
            best = min(best, cw) if math.isfinite(cw) else best
            p, rr = r.clone(), (r * r).sum()
            for k in range(steps):
                q = A(p)
                al = rr / (p * q).sum()
                x += al * p
                r -= al * q
                new = (r * r).sum()
                p = r + (new / rr) * p
                rr = new
                if k % 50 == 49 and bool((r.abs() <= 0.3 * tol * x.abs()).all()):
                    break
        phi = torch.where(self.free > 0, s * x, self.phi0)
        return phi


def _lines_seconds(nx, ny):
    k = min(nx, ny)
    return max(nx, ny) * (1e-3 + 2.5e-11 * k ** 3)


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        dims, h, hbar, f, src, U = _solve_inputs(case, seed)
        sys_ = _System(dims, h, hbar, f, src, U)
        if len(dims) == 2 and _lines_seconds(*dims) < 10.0:
            phi = sys_.solve_lines()[1]
        else:
            phi = sys_.solve_cg()
        S = sys_.S_of(phi)
        shape = dims[::-1]
        S = S.reshape(shape)
        return (S, phi.reshape(shape)) if case["phi"] else S
    if kind == "batch":
        inst = _batch_inputs(case, seed)
        if sum(_lines_seconds(*i[0]) for i in inst if i[2] < 7 * i[1]) > 18.0:
            return None
        out = []
        for dims, h, hbar, f, src, U in inst:
            sys_ = _System(dims, h, hbar, f, src, U)
            out.append(sys_.S_of(sys_.solve_lines()[1] if hbar < 7 * h else sys_.solve_cg()))
        return torch.cat(out)
    if kind == "train":
        dims, h, hbar, f, src, recv, T = _train_inputs(case, seed)
        sys_ = _System(dims, h, hbar, f, src, np.zeros(1))
        fac, phi = sys_.solve_lines()
        S = sys_.S_of(phi)
        dS = torch.zeros_like(S)
        dS[recv] = 2.0 * (S[recv] - T)
        g = (-hbar * dS.reshape(phi.shape) / phi) * sys_.free
        lam = sys_.line_solve(fac, g[0])[None] * sys_.free
        grad = -2.0 * sys_.w * sys_.f * phi * lam
        return {"S": S.reshape(dims[::-1]), "grad": grad.reshape(dims[::-1])}
    if kind == "paths":
        return _exact_paths(case, seed)
    return _exact_fft(case, seed)


def _exact_paths(case, seed):
    """The same rounded Euler steps, all paths at once."""
    (nx, ny), h, S, src, starts = _paths_inputs(case, seed)
    step, eps, ms = 0.5 * h, 2.0 * h, case["max_steps"]
    S = S.reshape(ny, nx)
    G = torch.empty((2, ny, nx), dtype=F64, device="cuda")
    G[0, :, 1:-1] = (S[:, 2:] - S[:, :-2]) / (2 * h)
    G[0, :, 0], G[0, :, -1] = (S[:, 1] - S[:, 0]) / h, (S[:, -1] - S[:, -2]) / h
    G[1, 1:-1] = (S[2:] - S[:-2]) / (2 * h)
    G[1, 0], G[1, -1] = (S[1] - S[0]) / h, (S[-1] - S[-2]) / h
    gx, gy = G[0].reshape(-1), G[1].reshape(-1)
    sx = torch.from_numpy(src % nx).cuda().to(F64) * h
    sy = torch.from_numpy(src // nx).cuda().to(F64) * h
    x, y = starts[:, 0].clone(), starts[:, 1].clone()
    n = len(x)
    P = torch.full((n, ms + 1, 2), math.nan, dtype=F64, device="cuda")
    P[:, 0, 0], P[:, 0, 1] = x, y
    length = torch.zeros(n, dtype=torch.int32, device="cuda")
    status = torch.ones(n, dtype=torch.int32, device="cuda")
    live = torch.ones(n, dtype=torch.bool, device="cuda")

    def near():
        dx, dy = x[:, None] - sx[None, :], y[:, None] - sy[None, :]
        return torch.sqrt(dx * dx + dy * dy).amin(1) < eps

    for k in range(ms):
        hit = live & near()
        status[hit] = 0
        live &= ~hit
        u, v = x / h, y / h
        cu, cv = u.floor().clamp(0, nx - 2), v.floor().clamp(0, ny - 2)
        tu, tv = u - cu, v - cv
        at = cu.long() + nx * cv.long()
        a, b = torch.zeros_like(x), torch.zeros_like(x)
        for q in range(4):
            w = (tu if q & 1 else 1.0 - tu) * (tv if q & 2 else 1.0 - tv)
            j = at + (q & 1) + nx * (q >> 1)
            a, b = a + w * gx[j], b + w * gy[j]
        gn = torch.sqrt(a * a + b * b)
        flat = live & ~(gn > 0)
        status[flat] = 2
        live &= ~flat
        nxt, nyt = x - step * a / gn, y - step * b / gn
        x = torch.where(live, nxt.clamp(0.0, (nx - 1) * h), x)
        y = torch.where(live, nyt.clamp(0.0, (ny - 1) * h), y)
        length += live
        P[:, k + 1, 0] = torch.where(live, x, P[:, k + 1, 0])
        P[:, k + 1, 1] = torch.where(live, y, P[:, k + 1, 1])
        if k % 64 == 63 and not bool(live.any()):
            break
    status[live & near()] = 0
    return {"G": G.reshape(2, -1), "paths": P, "lengths": length, "status": status}


def _exact_fft(case, seed):
    """Table 1 with torch.fft on arrays padded to 2n - 1, Bessel functions
    from torch.special, the origin's cell average by Gauss-Legendre rays."""
    (nx, ny), h, f, src = _fft_inputs(case, seed)
    hbar, terms = case["hbar"], case["terms"]
    ft = math.sqrt(0.5 * (float(f.min()) ** 2 + float(f.max()) ** 2))
    ix = torch.arange(2 * nx - 1, device="cuda", dtype=F64) - (nx - 1)
    iy = torch.arange(2 * ny - 1, device="cuda", dtype=F64) - (ny - 1)
    r = h * torch.hypot(ix[None, :], iy[:, None])

    def conv(kern, g):
        s = (3 * ny - 2, 3 * nx - 2)
        full = torch.fft.irfft2(torch.fft.rfft2(kern, s) * torch.fft.rfft2(g, s), s)
        return full[ny - 1:2 * ny - 1, nx - 1:2 * nx - 1]

    delta = torch.zeros(ny * nx, dtype=F64, device="cuda")
    delta[torch.from_numpy(src).cuda()] = 1.0
    term = conv(torch.exp(-ft * r / hbar), delta.reshape(ny, nx))
    phi = term.clone()
    a = ft / hbar
    xg, wg = np.polynomial.legendre.leggauss(64)
    R = torch.from_numpy(0.5 * h / np.cos(np.pi / 8 * (xg + 1))).cuda()
    ray = (1.0 - a * R * torch.special.modified_bessel_k1(a * R)) / (a * a)
    g0 = 8.0 * float((ray * torch.from_numpy(wg * np.pi / 8).cuda()).sum()) / (h * h)
    K = torch.special.modified_bessel_k0(a * r)
    K[ny - 1, nx - 1] = g0
    K = K / (2.0 * math.pi * hbar * hbar)
    for i in range(1, terms + 1):
        term = conv(K, (f * f - ft * ft) * term) * h * h
        phi = phi + (-1) ** i * term
    phi = phi.reshape(-1)
    return {"S": -hbar * torch.log(phi), "phi": phi}
