"""Performance cases: what a user of the solver has it do, through its public Python front end.

Kinds of case
    apply   one preconditioner application z = M r to the sources of one medium (the step every
            Krylov iteration spends most of its time in); a solver of the user's own calls it so
    medium  a new velocity model: set-up, factorisation of every box and the first application
    matvec  the global operator y = A x on its own (residual checks, a user's own Krylov loop)
    solve   a whole FGMRES solve of the right-hand sides of given sources on a factored medium

Grids are N x N interior cells in nb x nb boxes at 10 cells per wavelength.  Local factors are
complex FP32 in upper-tile storage ("c64", the default), complex FP64 ("c128", the plain path), or
TF32 pairs for the tensor cores ("x3", many sources sharing one medium).

Results of the FP32 paths are returned as complex64: an application computes and sums the local
solutions in FP32 and widens them on the store, so the cast drops nothing, and a wavefield solved to
a relative residual of 1e-8 or coarser is kept in single precision.  FP64 paths return complex128.
"""
import math

import numpy as np
import torch

from paper_1508_02897_gb300.solver import HelmholtzDDM

_DEV = "cuda"


def _case(name, kind, N, nb, precision="c64", nrhs=1, medium="random", npml=16, overlap=8, restart=10, rtol=1e-8,
          max_iters=400, graphs=False):
    c = dict(kind=kind, N=N, nb=nb, precision=precision, nrhs=nrhs, medium=medium, npml=npml, overlap=overlap)
    if kind == "solve":
        c.update(restart=restart, rtol=rtol, max_iters=max_iters, graphs=graphs)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call of the preconditioner: a 128^2 test problem, four boxes
        _case("apply_128", "apply", 128, 2, medium="homogeneous"),
        # an ordinary single-source application whose grid the boxes do not divide: uneven odd boxes
        _case("apply_1003", "apply", 1003, 8),
        # the large single-source application: 1024 boxes, the factors far larger than any cache
        _case("apply_4096", "apply", 4096, 32),
        # the plain FP64 path on an ordinary grid
        _case("apply_1024_c128", "apply", 1024, 8, precision="c128", medium="three_layer"),
        # a shot record of a few sources solved together on the default storage
        _case("apply_2048_4src", "apply", 2048, 16, nrhs=4),
        # many sources sharing one medium on the tensor cores
        _case("apply_1984_64src", "apply", 1984, 16, precision="x3", nrhs=64),
        # a new velocity model: set-up and factorisation, then the first application
        _case("medium_2048", "medium", 2048, 16),
        # the operator alone on the large grid
        _case("matvec_4096", "matvec", 4096, 32),
        # the smallest whole solve: launches and host round trips between short kernels
        _case("solve_128", "solve", 128, 2, medium="homogeneous", restart=50),
        # an ordinary whole solve of one source, three layers
        _case("solve_1024", "solve", 1024, 8, medium="three_layer", restart=50),
        # a request of 16 sources solved in lockstep, every step replayed as a CUDA graph
        _case("solve_1024_16src", "solve", 1024, 8, precision="x3", nrhs=16, restart=10, graphs=True),
        # two restart cycles of the large single-source solve (a fixed number of steps)
        _case("solve_4096_20it", "solve", 4096, 32, restart=10, rtol=1e-12, max_iters=20),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges: grid sizes over their logarithm, boxes that need not
    divide the grid, thinner PMLs and overlaps now and then."""
    kind = rng.choice(["apply", "apply", "apply", "medium", "matvec", "solve", "solve"])
    npml, overlap = rng.choice([(16, 8), (16, 8), (16, 8), (12, 6), (16, 0)])
    medium = rng.choice(["random", "random", "three_layer", "homogeneous"])
    precision, nrhs = "c64", 1
    if kind == "matvec":
        N, nrhs = _log_int(rng, 128, 3600), rng.choice([1, 1, 2, 3])
        if N > 2000:
            nrhs = 1
    elif kind == "medium":
        N = _log_int(rng, 128, 2100)
    elif kind == "apply":
        precision = rng.choice(["c64", "c64", "c64", "c128", "x3"])
        if precision == "c64":
            nrhs = rng.choice([1, 1, 1, 2, 3, 5, 8])
            N = _log_int(rng, 128, 3600 if nrhs == 1 else 2048)
        elif precision == "c128":
            N = _log_int(rng, 128, 1024)
        else:
            N, nrhs = _log_int(rng, 256, 1536), rng.randint(8, 64)
    else:
        precision = rng.choice(["c64", "c64", "x3"])
        nrhs = 1 if precision == "c64" else rng.randint(8, 20)
        N = _log_int(rng, 128, 1200 if precision == "c64" else 800)
    own = rng.uniform(88.0, 128.0)   # owned cells per box; box widths stay within 176
    nb = max(1 if kind == "matvec" else 2, int(math.ceil(N / own)))
    return _case(None, kind, N, nb, precision=precision, nrhs=nrhs, medium=medium, npml=npml, overlap=overlap,
                 restart=rng.choice([10, 20, 50]) if nrhs == 1 else 10, graphs=nrhs > 1)


# ---------------------------------------------------------------- inputs
def _gen(seed, salt):
    return torch.Generator(device=_DEV).manual_seed(1000003 * (int(seed) + 1) + salt)


def _velocity(case, seed):
    """Velocity on the whole truncated grid (float64 [n][n]).  homogeneous: c = 1; three_layer:
    1 / 1.5 / 2 from top to bottom with seeded interfaces; random: 1 + 0.3 clip(g, -1, 1), g white
    noise smoothed by a Gaussian of length 0.05 and scaled to unit deviation."""
    N, npml = case["N"], case["npml"]
    n = N + 2 * npml
    g = _gen(seed, 1)
    if case["medium"] == "homogeneous":
        return torch.ones((n, n), dtype=torch.float64, device=_DEV)
    if case["medium"] == "three_layer":
        y = (torch.arange(n, dtype=torch.float64, device=_DEV) - npml + 0.5) / N
        b = torch.rand(2, generator=g, device=_DEV, dtype=torch.float64) * 0.1
        c = 1.0 + 0.5 * (y >= 0.28 + b[0]).double() + 0.5 * (y >= 0.61 + b[1]).double()
        return c[:, None].expand(n, n).contiguous()
    noise = torch.randn((n, n), generator=g, device=_DEV, dtype=torch.float32)
    k = torch.arange(n, device=_DEV)
    d = torch.minimum(k, n - k).to(torch.float32) / N
    e = torch.exp(-d * d / (2.0 * 0.05 * 0.05))
    ker = torch.fft.fft(e).real.contiguous()
    f = torch.fft.ifft2(torch.fft.fft2(noise) * ker[:, None] * ker[None, :]).real.double()
    f = (f - f.mean()) / f.std()
    return 1.0 + 0.3 * f.clamp(-1.0, 1.0)


def _omega(case, c):
    return 2.0 * math.pi * float(c.min()) * case["N"] / 10.0   # 10 cells per wavelength at the slowest speed


def _sources(case, seed):
    """Unit-mass Gaussian sources (two cells wide) at seeded points, complex128 [nrhs][n][n]."""
    N, npml = case["N"], case["npml"]
    n = N + 2 * npml
    x = (torch.arange(n, dtype=torch.float64, device=_DEV) - npml + 0.5) / N
    p = torch.rand((case["nrhs"], 2), generator=_gen(seed, 2), device=_DEV, dtype=torch.float64) * 0.9 + 0.05
    w = 2.0 / N
    gx = torch.exp(-((x[None, :] - p[:, :1]) ** 2) / (2.0 * w * w))
    gy = torch.exp(-((x[None, :] - p[:, 1:]) ** 2) / (2.0 * w * w))
    return (gy[:, :, None] * gx[:, None, :] / (2.0 * math.pi * w * w)).to(torch.complex128)


def _field(case, seed):
    """Complex normal vectors, as the tests and Krylov bases feed them: complex128 [nrhs][n][n]."""
    n = case["N"] + 2 * case["npml"]
    r = torch.randn((case["nrhs"], n, n, 2), generator=_gen(seed, 3), device=_DEV, dtype=torch.float32)
    return torch.view_as_complex(r.double())


def _solver(case, c, omega):
    x3 = case["precision"] == "x3"
    return HelmholtzDDM(case["N"], case["npml"], omega, c, case["nb"], case["nb"], case["overlap"],
                        precision="c64" if x3 else case["precision"], tcore="x3" if x3 else False, symmetric=not x3,
                        factor=case["kind"] != "matvec")


def prepare(case, seed):
    c = _velocity(case, seed)
    omega = _omega(case, c)
    if case["kind"] == "medium":   # the new model arrives; nothing of it is set up yet
        return dict(case=case, c=c, omega=omega, r=_field(case, seed))
    s = _solver(case, c, omega)
    if case["kind"] == "solve":
        return dict(case=case, s=s, b=s.rhs(_sources(case, seed)))
    return dict(case=case, s=s, r=_field(case, seed))


def _out(case, z):
    return z if case["precision"] == "c128" else z.to(torch.complex64)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "matvec":
        return state["s"].matvec(state["r"])
    if kind == "apply":
        s = state["s"]
        # one step of the overlapping DDM is the preconditioner; with several sources this
        # entry point gives the library room for all of them at once
        return _out(case, s.apply_precond(state["r"]) if case["nrhs"] == 1 else s.apply_ddm(state["r"], 1))
    if kind == "medium":
        s = _solver(case, state["c"], state["omega"])
        z = s.apply_precond(state["r"])
        s.close()
        return _out(case, z)
    x, _ = state["s"].solve(state["b"], restart=case["restart"], rtol=case["rtol"], max_iters=case["max_iters"],
                            graphs=case["graphs"])
    return _out(case, x)


# ---------------------------------------------------------------- work
def _axis(case):
    """Per box along one axis: owned range and extent (even cuts; edge boxes own the outer PML)."""
    N, npml, nb, lo = case["N"], case["npml"], case["nb"], case["overlap"]
    cut = [npml + (i * N) // nb for i in range(nb + 1)]
    out = []
    for i in range(nb):
        o0, o1 = cut[i], cut[i + 1]
        e0, e1 = o0 - npml - (lo if i else 0), o1 + npml + (lo if i < nb - 1 else 0)
        out.append((0 if i == 0 else o0, N + 2 * npml if i == nb - 1 else o1, e0, e1))
    return out


def work(case):
    """Each input read once and each output written once.  A stored inverse is complex symmetric:
    m (m + 1) / 2 entries per grid row of a box of width m."""
    n2 = float((case["N"] + 2 * case["npml"]) ** 2)
    B = case["nrhs"]
    if case["kind"] == "matvec":
        return dict(bytes=n2 * (32.0 * B + 8.0), flops=n2 * 18.0 * B)
    w = [e1 - e0 for _, _, e0, e1 in _axis(case)]
    item = 16 if case["precision"] == "c128" else 8
    entries = sum(r * m * (m + 1) / 2.0 for m in w for r in w)
    mac = sum((2 * r - 1) * float(m) * m for m in w for r in w)
    ab, af = entries * item, 8.0 * mac * B
    if case["kind"] == "apply":
        return dict(bytes=ab + 32.0 * n2 * B, flops=af)
    if case["kind"] == "medium":
        return dict(bytes=2.0 * ab + (8.0 + 32.0) * n2, flops=af + 8.0 * sum(r * float(m) ** 3 for m in w for r in w))
    # about six steps per box and direction at a residual of 1e-8, each one application, one
    # operator, and the new vector against half a cycle of earlier ones
    it = min(case["max_iters"], 6 * case["nb"])
    vec = 16.0 * n2 * B
    half = min(case["restart"], it) / 2.0
    return dict(bytes=it * (ab + vec * (2.0 * half + 8.0)), flops=it * (af + n2 * B * (16.0 * half + 18.0)))


# ---------------------------------------------------------------- 64-bit values
def _alpha(ncell, npml):
    """PML stretching 1 + 20 i (xi / npml)^2 at the centres and faces of a segment of ncell cells."""
    c, f = np.arange(ncell) + 0.5, np.arange(ncell + 1.0)
    xi = [np.maximum(0.0, np.maximum(npml - t, t - (ncell - npml))) for t in (c, f)]
    return [1.0 + 20j * (t / npml) ** 2 for t in xi]


class _Plain64:
    """The operator and the one-step preconditioner in complex FP64 with plain torch: every box padded
    to the largest (identity rows), the blocks of its block-tridiagonal matrix inverted row by row."""

    def __init__(self, case, c, omega, precond=True):
        self.N, self.npml = case["N"], case["npml"]
        n = self.n = self.N + 2 * self.npml
        self.h2 = 1.0 / self.N ** 2
        self.k2 = (omega / c) ** 2
        ac, af = (torch.from_numpy(np.ascontiguousarray(t)).to(_DEV) for t in _alpha(n, self.npml))
        self.west, self.east = ac[:, None] / af[None, :-1], ac[:, None] / af[None, 1:]
        self.south, self.north = ac[None, :] / af[:-1, None], ac[None, :] / af[1:, None]
        self.jac = ac[:, None] * ac[None, :]
        self.centre = -(self.west + self.east + self.south + self.north) + self.h2 * self.jac * self.k2
        if precond:
            self._boxes(case)

    def mul(self, x):   # [B][n][n]
        y = self.centre * x
        y[:, :, 1:] += self.west[:, 1:] * x[:, :, :-1]
        y[:, :, :-1] += self.east[:, :-1] * x[:, :, 1:]
        y[:, 1:] += self.south[1:] * x[:, :-1]
        y[:, :-1] += self.north[:-1] * x[:, 1:]
        return y

    def _boxes(self, case):
        ax = _axis(case)
        self.box = [(x, y) for y in ax for x in ax]
        nbx, m = len(self.box), max(e1 - e0 for _, _, e0, e1 in ax)
        self.m = m
        diag = torch.ones((m, nbx, m), dtype=torch.complex128, device=_DEV)
        side = torch.zeros((m, nbx, m - 1), dtype=torch.complex128, device=_DEV)
        self.low = torch.zeros((m + 1, nbx, m), dtype=torch.complex128, device=_DEV)   # row j to row j - 1
        for b, (x, y) in enumerate(self.box):
            ex, ey = x[3] - x[2], y[3] - y[2]
            (c1, f1), (c2, f2) = _alpha(ex, self.npml), _alpha(ey, self.npml)
            c1, f1, c2, f2 = (torch.from_numpy(np.ascontiguousarray(t)).to(_DEV) for t in (c1, f1, c2, f2))
            w, e = c2[:, None] / f1[None, :-1], c2[:, None] / f1[None, 1:]
            s, nn = c1[None, :] / f2[:-1, None], c1[None, :] / f2[1:, None]
            diag[:ey, b, :ex] = -(w + e + s + nn) + self.h2 * c2[:, None] * c1[None, :] * self.k2[y[2]:y[3], x[2]:x[3]]
            side[:ey, b, :ex - 1] = e[:, :-1]
            self.low[1:ey, b, :ex] = s[1:]
        self.inv = torch.empty((m, nbx, m, m), dtype=torch.complex128, device=_DEV)
        for j in range(m):
            S = torch.diag_embed(diag[j]) + torch.diag_embed(side[j], 1) + torch.diag_embed(side[j], -1)
            if j:
                S = S - self.low[j][:, :, None] * self.inv[j - 1] * self.low[j][:, None, :]
            self.inv[j] = torch.linalg.inv(S)

    def apply(self, r):   # [B][n][n]
        B, m = r.shape[0], self.m
        rho = torch.zeros((m, len(self.box), m, B), dtype=torch.complex128, device=_DEV)
        for b, (x, y) in enumerate(self.box):
            rho[y[0] - y[2]:y[1] - y[2], b, x[0] - x[2]:x[1] - x[2]] = r[:, y[0]:y[1], x[0]:x[1]].permute(1, 2, 0)
        for j in range(m):
            if j:
                rho[j] -= self.low[j][:, :, None] * rho[j - 1]
            rho[j] = torch.bmm(self.inv[j], rho[j])
        for j in range(m - 2, -1, -1):
            rho[j] -= torch.bmm(self.inv[j], self.low[j + 1][:, :, None] * rho[j + 1])
        z = torch.zeros_like(r)
        for b, (x, y) in enumerate(self.box):
            z[:, y[2]:y[3], x[2]:x[3]] += rho[:y[3] - y[2], b, :x[3] - x[2]].permute(2, 0, 1)
        return z

    def solve(self, b, tol=1e-12, most=160):
        """Right-preconditioned GMRES (Gram-Schmidt twice), the sources side by side."""
        B = b.shape[0]
        x = torch.zeros_like(b)
        bn = torch.linalg.vector_norm(b.reshape(B, -1), dim=1)
        for _ in range(3):
            r = (b - self.mul(x)).reshape(B, -1)
            beta = torch.linalg.vector_norm(r, dim=1)
            if bool((beta <= tol * bn).all()):
                break
            V = [r / beta[:, None]]
            H = torch.zeros((B, most + 1, most), dtype=torch.complex128, device=_DEV)
            for k in range(most):
                w = self.mul(self.apply(V[k].reshape(b.shape))).reshape(B, -1)
                for _pass in range(2):
                    hs = [torch.einsum("bi,bi->b", v.conj(), w) for v in V]
                    for i, v in enumerate(V):
                        w = w - hs[i][:, None] * v
                        H[:, i, k] += hs[i]
                nw = torch.linalg.vector_norm(w, dim=1)
                H[:, k + 1, k] = nw
                V.append(w / nw[:, None])
                if k % 8 == 7 or k == most - 1:
                    e1 = torch.zeros((B, k + 2, 1), dtype=torch.complex128, device=_DEV)
                    e1[:, 0, 0] = beta
                    h = H[:, :k + 2, :k + 1].cpu()
                    y = torch.linalg.lstsq(h, e1.cpu()).solution
                    res = torch.linalg.vector_norm((e1.cpu() - h @ y).reshape(B, -1), dim=1).to(_DEV)
                    if bool((res <= 0.5 * tol * bn).all()):
                        break
            y = y.to(_DEV)
            u = sum(y[:, i, 0][:, None] * V[i] for i in range(y.shape[1]))
            x = x + self.apply(u.reshape(b.shape))
        return x


def exact(case, seed):
    w = [e1 - e0 for _, _, e0, e1 in _axis(case)]
    if case["kind"] == "matvec":
        c = _velocity(case, seed)
        return _Plain64(case, c, _omega(case, c), precond=False).mul(_field(case, seed))
    if case["nb"] ** 2 * max(w) ** 4 > 3.0e11:   # the block inverses in FP64 would take too long
        return None
    if case["kind"] == "solve" and (case["rtol"] < 1e-9 or case["nrhs"] > 1):
        return None   # a fixed number of steps has no converged value; many sources would take too long
    c = _velocity(case, seed)
    p = _Plain64(case, c, _omega(case, c))
    if case["kind"] == "solve":
        return p.solve(p.h2 * p.jac * _sources(case, seed))
    return p.apply(_field(case, seed))
