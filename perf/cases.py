"""What is timed of this framework, and what its results are in plain 64-bit arithmetic.

A case is one call (or one short sequence of calls) that a program using the
library makes on the GPU: a whole FGMRES solve, one V-cycle used as a
preconditioner, one relaxation sweep, a residual, a solve with its gradient, a
batch of solves.  Grids are n = coarse_n * 2^k, the sizes the library takes; the
work is the manufactured boundary data with an N(0, 1) nodal force of the
project's benchmark, and its C1 .. C5 sizes.

The mixed-precision solves run at rtol 1e-11, the tolerance at which a solve
with a reduced-precision cycle stands in for an FP64 one (at 1e-8 two solves
differ by the conditioning of the grid times 1e-8, whatever their arithmetic).
"""
from __future__ import annotations

import math
import random

import torch

import paper_2401_06277_gb300.autograd as autograd
import paper_2401_06277_gb300.stokes as stokes

PREC = {"fp64": stokes.STOKES_FP64, "fp32": stokes.STOKES_MIXED_FP32, "bf16": stokes.STOKES_MIXED_BF16}
SMOOTHER = {"vanka": stokes.STOKES_SMOOTHER_SHARED, "bs": stokes.STOKES_SMOOTHER_BRAESS_SARAZIN}


def listed():
    return [
        # the headline workload: a 2048 x 2048 solve to 1e-8 in FP64 (38 million unknowns)
        _solve("solve_fp64_2048", 2048, 4, "fp64", 1e-8),
        # a mid-sized grid whose coarsest grid is odd, so that no level is a multiple of a tile
        _solve("solve_fp64_640", 640, 5, "fp64", 1e-8),
        # the smallest problem in use (a first experiment, an inner loop): launches and latency
        _solve("solve_fp64_32", 32, 4, "fp64", 1e-8),
        # the mixed-precision forms as FP64 replacements, large, tensor-core and small
        _solve("solve_mixed_fp32_2048", 2048, 4, "fp32", 1e-11),
        _solve("solve_mixed_bf16_1024", 1024, 4, "bf16", 1e-11),
        _solve("solve_mixed_fp32_128", 128, 4, "fp32", 1e-11),
        # the other smoother of the FP64 form
        _solve("solve_braess_sarazin_512", 512, 4, "fp64", 1e-8, smoother="bs"),
        # the cycle as a preconditioner of somebody else's Krylov method
        {"name": "vcycle_fp64_1024", "kind": "vcycle", "n": 1024, "coarse_n": 4},
        # the parts a program composes itself: a sweep on a ragged grid, the operator on the largest
        {"name": "sweep_fp64_896", "kind": "sweep", "n": 896, "coarse_n": 7},
        {"name": "residual_fp64_2048", "kind": "residual", "n": 2048, "coarse_n": 4},
        # solve and gradient of a misfit (forward and backward of the autograd function)
        {"name": "gradient_fp64_512", "kind": "gradient", "n": 512, "coarse_n": 4, "rtol": 1e-8},
        # many independent problems of different sizes
        {"name": "batch_mixed_uneven_8", "kind": "batch", "count": 8, "largest": 1024, "prec": "fp32",
         "rtol": 1e-11},
    ]


def _solve(name, n, coarse_n, prec, rtol, smoother="vanka"):
    c = {"kind": "solve", "n": n, "coarse_n": coarse_n, "prec": prec, "rtol": rtol, "smoother": smoother}
    return {"name": name, **c} if name else c


def _size(rng, lo, hi):
    """(n, coarse_n) with n = coarse_n 2^k, log-uniform in lo..hi over coarse grids of 4..7 elements."""
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    sizes = [(c << k, c) for c in (4, 5, 6, 7) for k in range(1, 12) if lo <= c << k <= hi]
    near = sorted(sizes, key=lambda s: abs(math.log(s[0] / want)))
    return near[rng.randrange(2)]


def draw(rng: random.Random):
    kind = rng.choice(["solve", "solve", "solve", "mixed", "bs", "vcycle", "sweep", "residual", "gradient", "batch"])
    if kind == "solve":
        return _solve(None, *_size(rng, 32, 1792), "fp64", 1e-8)
    if kind == "mixed":
        return _solve(None, *_size(rng, 64, 1792), rng.choice(["fp32", "bf16"]), 1e-11)
    if kind == "bs":
        return _solve(None, *_size(rng, 32, 1024), "fp64", 1e-8, smoother="bs")
    if kind == "batch":
        prec = rng.choice(["fp32", "fp64"])
        return {"kind": "batch", "count": rng.randint(2, 8), "prec": prec, "rtol": 1e-11,
                "largest": rng.choice([256, 512] if prec == "fp64" else [256, 512, 1024])}
    lo, hi = {"vcycle": (32, 2048), "sweep": (32, 2048), "residual": (64, 2048), "gradient": (32, 1024)}[kind]
    n, cn = _size(rng, lo, hi)
    c = {"kind": kind, "n": n, "coarse_n": cn}
    return {**c, "rtol": 1e-8} if kind == "gradient" else c


def _batch_sizes(case):
    """Grid sizes of a batch: halving from the largest to 128, then again."""
    per = [case["largest"] >> k for k in range(8) if case["largest"] >> k >= 128]
    return [per[k % len(per)] for k in range(case["count"])]


# ---- inputs ----

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _boundary(n):
    """Nodal velocity (sin pi x cos pi y, -cos pi x sin pi y), its normal component exactly 0 on the boundary."""
    t = torch.arange(2 * n + 1, device="cuda", dtype=torch.float64) / (2 * n)
    s, c = torch.sin(math.pi * t), torch.sin(math.pi * (0.5 - t))
    s[0] = s[-1] = 0.0
    c[n] = 0.0
    return torch.stack([c[:, None] * s[None, :], -(s[:, None] * c[None, :])]).contiguous()


def _force(n, gen):
    return torch.randn((2, 2 * n + 1, 2 * n + 1), generator=gen, device="cuda", dtype=torch.float64)


def _hierarchy(case):
    return stokes.Hierarchy(case["n"], coarse_n=case["coarse_n"], prec=PREC[case.get("prec", "fp64")],
                            smoother=SMOOTHER[case.get("smoother", "vanka")], rtol=case.get("rtol", 1e-8))


def _near_solution(n, gen):
    """An iterate as a sweep or a residual meets it: the smooth field plus a rough error of a few percent."""
    x = 0.03 * torch.randn(stokes.vec_len(n), generator=gen, device="cuda", dtype=torch.float64)
    nq, nv = 2 * n + 1, (2 * n + 1) ** 2
    u = _boundary(n)
    rough = x[: 2 * nv].view(2, nq, nq)
    rough[:, 0] = rough[:, -1] = 0.0
    rough[:, :, 0] = rough[:, :, -1] = 0.0
    x[: 2 * nv] += u.reshape(-1)
    return x


def _krylov_vector(n, gen):
    """A residual as the preconditioner meets it after the first iterations: rough, zero on Dirichlet rows."""
    r = torch.randn(stokes.vec_len(n), generator=gen, device="cuda", dtype=torch.float64)
    nq, nv = 2 * n + 1, (2 * n + 1) ** 2
    u = r[: 2 * nv].view(2, nq, nq)
    u[:, 0] = u[:, -1] = 0.0
    u[:, :, 0] = u[:, :, -1] = 0.0
    r[2 * nv:] *= 1.0 / n          # pressure rows carry a factor h
    r[2 * nv:] -= r[2 * nv:].mean()
    return r / r.norm()


def prepare(case, seed):
    gen = _generator(seed)
    kind = case["kind"]
    if kind == "batch":
        ns = _batch_sizes(case)
        batch = stokes.Batch(ns, prec=PREC[case["prec"]], rtol=case["rtol"])
        rhs = [batch.assemble_rhs(k, _force(n, gen), _boundary(n)) for k, n in enumerate(ns)]
        return {"kind": kind, "batch": batch, "rhs": rhs}
    n = case["n"]
    H = _hierarchy(case)
    st = {"kind": kind, "h": H}
    if kind == "vcycle":
        st["r"] = _krylov_vector(n, gen)
        return st
    f, ud = _force(n, gen), _boundary(n)
    if kind == "gradient":
        st["f"], st["ud"] = f.requires_grad_(True), ud
        # dJ/dx of a velocity misfit with noisy data: zero on pressures and Dirichlet rows
        g = _krylov_vector(n, gen)
        g[2 * (2 * n + 1) ** 2:] = 0.0
        st["g"] = g
        return st
    st["b"] = H.assemble_rhs(f, ud)
    if kind in ("sweep", "residual"):
        st["x"] = _near_solution(n, gen)
    return st


def _zero_mean(x, n):
    """The pressure is determined up to a constant: a program fixes it by the mean."""
    p = x[2 * (2 * n + 1) ** 2:]
    p -= p.mean()
    return x


def run(state):
    kind = state["kind"]
    if kind == "solve":
        return _zero_mean(state["h"].solve(state["b"])[0], state["h"].n)
    if kind == "vcycle":
        return state["h"].vcycle(state["r"])
    if kind == "sweep":
        return state["h"].sweep(state["x"], state["b"])
    if kind == "residual":
        return state["h"].residual(state["b"], state["x"])
    if kind == "gradient":
        x = autograd.stokes_solve(state["f"], state["ud"], state["h"])
        (grad,) = torch.autograd.grad(x, state["f"], state["g"])
        return {"x": x, "grad": grad}
    xs = state["batch"].solve(state["rhs"])[0]
    return [_zero_mean(x, n) for x, n in zip(xs, state["batch"].ns)]


# ---- the work that cannot be left out ----

def _cycle_work(n, coarse_n, sweeps, size, sweep_flops):
    """Bytes and operations of one V(2,2): per level, each sweep reads x and b and writes x, the residual
    does the same, restriction reads a fine and writes a coarse vector, prolongation reads a coarse vector
    and updates a fine one."""
    by = fl = 0.0
    while n > coarse_n:
        N, Nc, V = stokes.vec_len(n), stokes.vec_len(n // 2), (n + 1) ** 2
        by += size * (sweeps * 3 * N - N + 3 * N + N + Nc + Nc + 2 * N)
        fl += V * (sweeps * sweep_flops + 361 + 120)
        n //= 2
    return by, fl


def _iterations(case):
    """FGMRES iterations to the tolerance (they do not depend on the grid): 6 or 8 to 1e-8, 12 to 1e-11."""
    return 6 if case.get("smoother") == "bs" else 8 if case.get("rtol", 1e-8) >= 1e-9 else 12


def _solve_work(n, coarse_n, prec, smoother, its):
    N, V = stokes.vec_len(n), (n + 1) ** 2
    cb, cf = _cycle_work(n, coarse_n, 4, 8 if prec == "fp64" else 4, 1681 if smoother == "vanka" else 620)
    # an iteration: the cycle, its input and output, A z, one pass over the basis, the new basis vector
    by = sum(cb + 8 * N * (2 + 2 + (j + 1) + 2) for j in range(its)) + 8 * N * (its + 6)
    fl = sum(cf + 334 * V + 4 * N * (j + 1) + 3 * N for j in range(its)) + 2 * N * its + 668 * V
    return by, fl


def work(case):
    kind = case["kind"]
    if kind == "batch":
        w = [_solve_work(n, 4, case["prec"], "vanka", _iterations(case)) for n in _batch_sizes(case)]
        return {"bytes": sum(a for a, _ in w), "flops": sum(b for _, b in w)}
    n, N, V = case["n"], stokes.vec_len(case["n"]), (case["n"] + 1) ** 2
    if kind == "solve":
        by, fl = _solve_work(n, case["coarse_n"], case["prec"], case["smoother"], _iterations(case))
    elif kind == "gradient":
        by, fl = (2 * v for v in _solve_work(n, case["coarse_n"], "fp64", "vanka", _iterations(case)))
        by += 8 * 4 * N
        fl += 4 * 50 * V
    elif kind == "vcycle":
        by, fl = _cycle_work(n, case["coarse_n"], 4, 8, 1681)
    else:
        by, fl = 3 * 8 * N, V * (1681 if kind == "sweep" else 361)
    return {"bytes": by, "flops": fl}


# ---- the same results in plain torch, 64 bits ----
# Fields are [J, I] arrays (y first).  Every block of the operator is a Kronecker product of 1D
# matrices, applied here as banded 1D operators; a Vanka sweep gathers the 51 unknowns of every
# vertex patch and multiplies by dense inverses, one for each distinct patch matrix.

_KE = [[7.0, -8.0, 1.0], [-8.0, 16.0, -8.0], [1.0, -8.0, 7.0]]       # / (3 h)
_ME = [[4.0, 2.0, -1.0], [2.0, 16.0, 2.0], [-1.0, 2.0, 4.0]]         # h / 30
_CE = [[-5 / 6, 2 / 3, 1 / 6], [-1 / 6, -2 / 3, 5 / 6]]              # int q_a psi'
_NE = [[1 / 6, 1 / 3, 0.0], [0.0, 1 / 3, 1 / 6]]                     # h


def _bands(elem, n, rows):
    """Element matrices (rows x 3) assembled on n elements as bands [row, offset + 2] of the Q2 columns."""
    step = 2 if rows == 3 else 1
    m = torch.zeros((step * n + 1, 5), dtype=torch.float64)
    e = torch.arange(n)
    for a in range(rows):
        for b in range(3):
            off = b - a if rows == 3 else b - 2 * a
            m.index_put_((step * e + a, torch.full((n,), off + 2)), torch.full((n,), elem[a][b], dtype=torch.float64),
                         accumulate=True)
    return m.cuda()


def _mul(m, x, step):
    """Banded 1D operator along the last axis: y[r] = sum_o m[r, o] x[step r + o - 2]."""
    rows = m.shape[0]
    xp = torch.nn.functional.pad(x, (2, 2))
    y = torch.zeros(*x.shape[:-1], rows, dtype=torch.float64, device=x.device)
    for o in range(5):
        y += m[:, o] * xp[..., o: o + step * (rows - 1) + 1: step]
    return y


def _mul_t(m, x, step, cols):
    """The transpose: y[step r + o - 2] += m[r, o] x[r]."""
    rows = m.shape[0]
    y = torch.zeros(*x.shape[:-1], cols + 4, dtype=torch.float64, device=x.device)
    for o in range(5):
        y[..., o: o + step * (rows - 1) + 1: step] += m[:, o] * x
    return y[..., 2:-2]


def _t(x):
    return x.transpose(-1, -2)


class _Plain:
    """One level: operator, sweep and transfers."""

    def __init__(self, n, smoother="vanka"):
        self.n, self.nq, self.np, self.nv = n, 2 * n + 1, n + 1, (2 * n + 1) ** 2
        h = 1.0 / n
        self.K, self.M = _bands(_KE, n, 3) / (3 * h), _bands(_ME, n, 3) * (h / 30)
        self.C, self.N = _bands(_CE, n, 2), _bands(_NE, n, 2) * h
        self.free = torch.zeros((self.nq, self.nq), dtype=torch.float64, device="cuda")
        self.free[1:-1, 1:-1] = 1.0
        self.smoother = smoother
        if smoother == "vanka":
            self._patches()
        elif smoother == "bs":
            k, m = self.K[:, 2], self.M[:, 2]
            self.D = self.free * (m[:, None] * k[None, :] + k[:, None] * m[None, :]) + (1 - self.free)
            w = self.free / self.D
            self.dS = -(_t(_mul(self.N ** 2, _t(_mul(self.C ** 2, w, 2)), 2))
                        + _t(_mul(self.C ** 2, _t(_mul(self.N ** 2, w, 2)), 2)))

    def split(self, x):
        return x[: 2 * self.nv].view(2, self.nq, self.nq), x[2 * self.nv:].view(self.np, self.np)

    def lap(self, u):
        return _t(_mul(self.M, _t(_mul(self.K, u, 1)), 1)) + _t(_mul(self.K, _t(_mul(self.M, u, 1)), 1))

    def div(self, u):
        return -(_t(_mul(self.N, _t(_mul(self.C, u[0], 2)), 2)) + _t(_mul(self.C, _t(_mul(self.N, u[1], 2)), 2)))

    def grad(self, p):
        q = self.nq
        return torch.stack([-_t(_mul_t(self.N, _t(_mul_t(self.C, p, 2, q)), 2, q)),
                            -_t(_mul_t(self.C, _t(_mul_t(self.N, p, 2, q)), 2, q))])

    def apply(self, x):
        u, p = self.split(x)
        uf = u * self.free
        v = self.free * (self.lap(uf) + self.grad(p)) + (1 - self.free) * u
        return torch.cat([v.reshape(-1), self.div(uf).reshape(-1)])

    def rhs(self, f, ud):
        g = ud * (1 - self.free)
        mass = _t(_mul(self.M, _t(_mul(self.M, f, 1)), 1))
        v = self.free * (mass - self.lap(g)) + g
        return torch.cat([v.reshape(-1), -self.div(g).reshape(-1)])

    def rhs_t(self, lam):
        u, _ = self.split(lam)
        return _t(_mul(self.M, _t(_mul(self.M, u * self.free, 1)), 1))

    def _dense(self, m, r0, rows, c0, step):
        d = torch.zeros((rows, 5), dtype=torch.float64)
        for r in range(rows):
            for o in range(5):
                c = step * (r0 + r) + o - 2 - c0
                if 0 <= r0 + r < m.shape[0] and 0 <= c < 5:
                    d[r, c] = m[r0 + r, o]
        return d

    def _axis(self, i):
        """(K, M, C, N, free) of the 5-node window of vertex i."""
        c0 = 2 * i - 2
        fr = torch.tensor([1.0 if 0 < c0 + k < self.nq - 1 else 0.0 for k in range(5)], dtype=torch.float64)
        K, M, C, N = (self._dense(m.cpu(), r, k, c0, s) for m, r, k, s in
                      ((self.K, c0, 5, 1), (self.M, c0, 5, 1), (self.C, i, 1, 2), (self.N, i, 1, 2)))
        return K, M, C, N, fr

    def _patches(self):
        n = self.n
        ax = {c: self._axis(i) for c, i in enumerate((0, 1, 2, n - 1, n))}
        self.inv = {}
        for cy in range(5):
            for cx in range(5):
                Kx, Mx, Cx, Nx, fx = ax[cx]
                Ky, My, Cy, Ny, fy = ax[cy]
                f = torch.kron(fy, fx)
                L = (torch.kron(Ky, Mx) + torch.kron(My, Kx)) * f[:, None] * f[None, :] + torch.diag(1 - f)
                A = torch.zeros((51, 51), dtype=torch.float64)
                A[:25, :25] = A[25:50, 25:50] = L
                A[50, :25] = -torch.kron(Ny, Cx)[0] * f
                A[50, 25:50] = -torch.kron(Cy, Nx)[0] * f
                A[:50, 50] = A[50, :50]
                self.inv[cy, cx] = torch.linalg.inv(A).cuda()
        one = torch.ones((self.np, self.np, 25), dtype=torch.float64, device="cuda")
        self.mult = self._fold(one)

    def _fold(self, w):
        y = torch.zeros((self.nq + 4, self.nq + 4), dtype=torch.float64, device="cuda")
        for s in range(25):
            J, I = divmod(s, 5)
            y[J: J + 2 * self.np - 1: 2, I: I + 2 * self.np - 1: 2] += w[:, :, s]
        return y[2:-2, 2:-2]

    def sweep(self, x, b):
        r = b if x is None else b - self.apply(x)
        ru, rp = self.split(r)
        if self.smoother == "vanka":
            R = torch.empty((self.np, self.np, 51), dtype=torch.float64, device="cuda")
            for c in range(2):
                w = torch.nn.functional.pad(ru[c], (2, 2, 2, 2)).unfold(0, 5, 2).unfold(1, 5, 2)
                R[:, :, 25 * c: 25 * c + 25] = w.reshape(self.np, self.np, 25)
            R[:, :, 50] = rp
            n, D = self.n, torch.empty_like(R)
            span = [slice(0, 1), slice(1, 2), slice(2, n - 1), slice(n - 1, n), slice(n, n + 1)]
            for (cy, cx), inv in self.inv.items():
                D[span[cy], span[cx]] = R[span[cy], span[cx]] @ inv.T
            du = torch.stack([self._fold(D[:, :, :25]), self._fold(D[:, :, 25:50])]) / self.mult
            d = 0.7 * torch.cat([du.reshape(-1), D[:, :, 50].reshape(-1)])
        else:
            g = rp - self.div(self.free * ru / self.D)
            dp = torch.zeros_like(rp)
            for _ in range(2):
                dp = dp + (g + self.div(self.free * self.grad(dp) / self.D)) / self.dS
            d = torch.cat([((ru - self.free * self.grad(dp)) / self.D).reshape(-1), dp.reshape(-1)])
        return d if x is None else x + d


def _interp(nc, quadratic):
    """1D interpolation from nc to 2 nc elements, dense."""
    if quadratic:
        P = torch.zeros((4 * nc + 1, 2 * nc + 1), dtype=torch.float64)
        k = torch.arange(2 * nc + 1)
        P[2 * k, k] = 1.0
        e = torch.arange(nc)
        for f, w in ((1, (0.375, 0.75, -0.125)), (3, (-0.125, 0.75, 0.375))):
            for g in range(3):
                P[4 * e + f, 2 * e + g] = w[g]
    else:
        P = torch.zeros((2 * nc + 1, nc + 1), dtype=torch.float64)
        k = torch.arange(nc + 1)
        P[2 * k, k] = 1.0
        e = torch.arange(nc)
        P[2 * e + 1, e] = P[2 * e + 1, e + 1] = 0.5
    return P.cuda()


class _PlainSolver:
    def __init__(self, n, coarse_n, smoother="vanka"):
        self.lv = []
        while n >= coarse_n:
            self.lv.insert(0, _Plain(n, smoother if n > coarse_n else "none"))
            n //= 2
        self.P = [None] + [(_interp(L.n // 2, True), _interp(L.n // 2, False)) for L in self.lv[1:]]
        C = self.lv[0]
        N = stokes.vec_len(C.n)
        A = torch.zeros((N + 1, N + 1), dtype=torch.float64, device="cuda")
        A[:N, :N] = torch.stack([C.apply(e) for e in torch.eye(N, dtype=torch.float64, device="cuda")]).T
        w = torch.ones(C.np, dtype=torch.float64, device="cuda") / C.n
        w[0] = w[-1] = 0.5 / C.n
        A[N, 2 * C.nv: N] = A[2 * C.nv: N, N] = (w[:, None] * w[None, :]).reshape(-1)
        self.G = torch.linalg.inv(A)[:N, :N]

    def cycle(self, r, l=None):
        l = len(self.lv) - 1 if l is None else l
        if l == 0:
            return self.G @ r
        L, C, (P2, P1) = self.lv[l], self.lv[l - 1], self.P[l]
        x = L.sweep(L.sweep(None, r), r)
        u, p = L.split(r - L.apply(x))
        rc = torch.cat([(C.free * (P2.T @ (u * L.free) @ P2)).reshape(-1), (P1.T @ p @ P1).reshape(-1)])
        eu, ep = C.split(self.cycle(rc, l - 1))
        x = x + torch.cat([(L.free * (P2 @ (eu * C.free) @ P2.T)).reshape(-1), (P1 @ ep @ P1.T).reshape(-1)])
        return L.sweep(L.sweep(x, r), r)

    def solve(self, b, x, rtol, m=30):
        """FGMRES(m), modified Gram-Schmidt (one cycle suffices for the tolerances in use)."""
        A = self.lv[-1].apply
        r = b - A(x)
        beta = r.norm().item()
        if beta == 0.0:
            return x
        V, Z, H, g = [r / beta], [], torch.zeros((m + 1, m), dtype=torch.float64), None
        for j in range(m):
            Z.append(self.cycle(V[j]))
            w = A(Z[j])
            for i in range(j + 1):
                H[i, j] = torch.dot(V[i], w).item()
                w -= H[i, j].item() * V[i]
            H[j + 1, j] = w.norm().item()
            V.append(w / H[j + 1, j].item())
            e = torch.zeros(j + 2, dtype=torch.float64)
            e[0] = beta
            g = torch.linalg.lstsq(H[: j + 2, : j + 1], e[:, None]).solution[:, 0]
            if (e - H[: j + 2, : j + 1] @ g).norm().item() <= rtol * beta:
                break
        for z, y in zip(Z, g.tolist()):
            x = x + y * z
        return x


def _start(L, b):
    u, _ = L.split(b)
    return torch.cat([((1 - L.free) * u).reshape(-1), torch.zeros(L.np ** 2, dtype=torch.float64, device="cuda")])


def exact(case, seed):
    """What run() returns, in plain torch.  None for the mixed-precision forms: two solves of one system
    stopped by the same tolerance differ by their arithmetic times the grid's conditioning."""
    kind = case["kind"]
    if kind == "batch" or case.get("prec", "fp64") != "fp64":
        return None
    n, gen = case["n"], _generator(seed)
    if kind == "vcycle":
        return _PlainSolver(n, case["coarse_n"]).cycle(_krylov_vector(n, gen))
    f, ud = _force(n, gen), _boundary(n)
    if kind in ("sweep", "residual"):
        L = _Plain(n, "vanka" if kind == "sweep" else "none")
        b = L.rhs(f, ud)
        x = _near_solution(n, gen)
        return L.sweep(x, b) if kind == "sweep" else b - L.apply(x)
    S = _PlainSolver(n, case["coarse_n"], case.get("smoother", "vanka"))
    L = S.lv[-1]
    b = L.rhs(f, ud)
    x = S.solve(b, _start(L, b), case["rtol"])
    if kind == "solve":
        return _zero_mean(x, n)
    g = _krylov_vector(n, gen)
    g[2 * L.nv:] = 0.0
    lam = S.solve(g, _start(L, g), case["rtol"])
    return {"x": x, "grad": L.rhs_t(lam)}
