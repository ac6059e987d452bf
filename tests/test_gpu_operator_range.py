"""The tensor-core FP64 operator (n >= 192) entry by entry, for data whose size changes
within a strip of 128 cells or differs between the components.

Bar: 66 u sum |a| |x| per row (u = 2^-53), plus 4 u |b|.  31 u is the a-priori bound of
the FP64 kernel (25 + 6 multiply-adds), which the contraction keeps with 30 u; the
reference, the exact integer stencil in FP64, takes another 31, the final roundings 4.
Inputs far below the normal range are scaled so that every product stays normal."""
import numpy as np
import pytest
import scipy.sparse as sp
import torch

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
_MAT = {}


def matrices(n):
    """Integer stencils (K (x) M + M (x) K, couplings) with the Dirichlet nodes eliminated."""
    if n in _MAT:
        return _MAT[n]
    nq, npv = 2 * n + 1, n + 1

    def rows(even, odd):
        m = sp.lil_matrix((nq, nq))
        for i in range(nq):
            t = odd if i & 1 else even
            for k, v in enumerate(t):
                j = i + k - len(t) // 2
                if 0 <= j < nq:
                    m[i, j] = v
        return m.tocsr()

    K, M = rows([1, -8, 14, -8, 1], [-8, 16, -8]), rows([-1, 2, 8, 2, -1], [2, 16, 2])
    C, N = sp.lil_matrix((npv, nq)), sp.lil_matrix((npv, nq))
    for i in range(npv):
        for off, c, w in ((-2, -1, 0), (-1, -4, 1), (0, 0, 1), (1, 4, 1), (2, 1, 0)):
            if 0 <= 2 * i + off < nq:
                C[i, 2 * i + off], N[i, 2 * i + off] = c, w
    C, N = C.tocsr(), N.tocsr()
    inner = np.zeros(nq)
    inner[1:-1] = 1.0
    free = np.outer(inner, inner).ravel()
    D = sp.diags(free)
    L = D @ (sp.kron(M, K) + sp.kron(K, M)) @ D
    Bx, By = sp.kron(N, C) @ D, sp.kron(C, N) @ D
    _MAT[n] = tuple(m.tocsr() for m in (L, Bx, By)) + (1.0 - free,)
    return _MAT[n]


def apply_ref(n, nu, x):
    """A x and the rows' sum |a| |x|."""
    L, Bx, By, fixed = matrices(n)
    nv = (2 * n + 1) ** 2
    cl, cb = nu / 90.0, -1.0 / (18.0 * n)
    out = []
    for f, y in ((lambda m: m, x), (abs, np.abs(x))):
        u, v, p = y[:nv], y[nv:2 * nv], y[2 * nv:]
        c, d = (cl, cb) if y is x else (cl, abs(cb))
        out.append(np.concatenate([c * (f(L) @ u) + d * (f(Bx).T @ p) + fixed * u,
                                   c * (f(L) @ v) + d * (f(By).T @ p) + fixed * v,
                                   d * (f(Bx) @ u + f(By) @ v)]))
    return out


def field(n, form, rng):
    nq, npv = 2 * n + 1, n + 1
    j, i = np.mgrid[0:nq, 0:nq]
    u, v = rng.standard_normal((2, nq, nq))
    p = rng.standard_normal((npv, npv))
    if form in ("columns up", "columns down", "rows up", "rows down"):
        k = (i if form.startswith("columns") else j) * (0.625 if form.endswith("up") else -0.625)
        s = 2.0 ** k
        u, v, p = u * s, v * s, p * s[::2, ::2]
    elif form == "spikes":          # one node, one pressure far above the rest
        u[101, 90] = 2.0 ** 70
        v[40, 200] = -2.0 ** 30
        p[60, 70] = 2.0 ** 50
    elif form == "any size":
        u, v, p = (a * 2.0 ** rng.integers(-40, 41, a.shape) for a in (u, v, p))
    elif form == "u large":
        u *= 2.0 ** 60
    elif form == "v large":
        v *= 2.0 ** 60
    elif form == "p large":         # and nearly constant
        p = 2.0 ** 40 * (1.0 + 1e-3 * p)
    elif form == "tiny":
        u, v, p = (a * 2.0 ** -930 for a in (u, v, p))
    elif form == "wall":            # u x^2 and v x at the walls
        s = i / (nq - 1.0) * (1.0 - i / (nq - 1.0))
        u, v, p = s ** 2 * (1.0 + 0.1 * j / nq), s * (1.0 + 0.1 * j / nq), 0.01 * np.cos(np.arange(npv) / n)[:, None] + 0 * p
    elif form == "sparse":
        u, v, p = (np.where(rng.random(a.shape) < 0.01, a * 2.0 ** rng.integers(-60, 1, a.shape), 0.0) for a in (u, v, p))
    elif form == "u only":
        v, p = 0.0 * v, 0.0 * p
        u = u * 2.0 ** rng.integers(-60, 1, u.shape)
    return np.concatenate([np.ravel(u), np.ravel(v), np.ravel(p)])


FORMS = ["plain", "columns up", "columns down", "rows up", "rows down", "spikes", "any size", "u large", "v large",
         "p large", "tiny", "wall", "sparse", "u only"]


@pytest.mark.parametrize("nu", [1.0, 1e-6])
@pytest.mark.parametrize("form", FORMS)
def test_operator_keeps_every_entry(form, nu):
    import paper_2401_06277_gb300 as pkg
    n = 192
    H = pkg.Hierarchy(n, viscosity=nu, coarse_n=6, restart=1)
    rng = np.random.default_rng(FORMS.index(form))
    x = field(n, form, rng)
    want, size = apply_ref(n, nu, x)
    b = size * rng.standard_normal(len(x))
    xd, bd = torch.from_numpy(x).cuda(), torch.from_numpy(b).cuda()
    got = H.apply(xd).cpu().numpy()
    q = np.abs(got - want) / np.maximum(U * size, 1e-320)
    assert q.max() <= 66.0, (q.max(), int(q.argmax()))
    got = H.residual(bd, xd).cpu().numpy()
    err = np.abs(got - (b - want))
    assert (err <= U * (66.0 * size + 4.0 * np.abs(b))).all()
    # in place: r and b the same vector
    H.residual(bd, xd)
    from paper_2401_06277_gb300 import stokes
    stokes.stokes_residual(H.handle, H.levels - 1, bd, xd, bd)
    assert np.array_equal(bd.cpu().numpy(), got)
    H.close()


@pytest.mark.parametrize("n,coarse_n", [(128, 4), (144, 9), (160, 5), (176, 11), (192, 6), (208, 13), (224, 7)])
def test_operator_on_both_sides_of_the_size_rule(n, coarse_n):
    import paper_2401_06277_gb300 as pkg
    H = pkg.Hierarchy(n, coarse_n=coarse_n, restart=1)
    x = field(n, "plain", np.random.default_rng(n))
    want, size = apply_ref(n, 1.0, x)
    got = H.apply(torch.from_numpy(x).cuda()).cpu().numpy()
    assert (np.abs(got - want) <= 66.0 * U * size).all()
    H.close()
