"""The FP64 operator and residual of the levels on the tensor cores, and the transfers of
the larger levels, against the oracle's matrices.

Grids: the smallest that take these kernels and ragged ones (n + 1 one or a few more than
a multiple of the 128-column strip, and half a strip), odd row counts, all levels' kinds of
rows (Dirichlet, next to the boundary, pressure), non-finite entries.  Tolerance: 1e-13 of
the largest entry, the FP64 kernels' bar."""
import numpy as np
import pytest
import torch

import stokes_inputs as si
from oracle import stokes_oracle as O

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def close(got, want, tol=1e-13):
    return np.abs(got.cpu().numpy() - want).max() <= tol * np.abs(want).max()


@pytest.mark.parametrize("n,coarse_n", [(160, 5), (192, 6), (256, 4), (448, 7)])
def test_operator_and_transfers_match_the_matrices(n, coarse_n):
    import paper_2401_06277_gb300 as pkg
    from paper_2401_06277_gb300 import stokes
    H = pkg.Hierarchy(n, coarse_n=coarse_n, restart=1)
    lv = O.build_level(n, 1.0)
    x, b = si.random_vector(n, 1), si.random_vector(n, 2)
    Ax = lv.A @ x
    assert close(H.apply(dev(x)), Ax)
    assert close(H.residual(dev(b), dev(x)), b - Ax)
    # sizes falling by 2^-200 over the columns and rising by rows: each entry as its neighbours
    nq, nv = 2 * n + 1, (2 * n + 1) ** 2
    k = np.linspace(0, 200, nq)
    amp = 2.0 ** (k[:, None] + np.zeros(nq))
    y = x.copy()
    y[:nv] *= amp.ravel()
    y[nv: 2 * nv] *= amp.ravel()
    y[2 * nv:] *= amp[::2, ::2].ravel()
    got, want = H.apply(dev(y)).cpu().numpy(), lv.A @ y
    for c in range(2):
        g, w = (v[c * nv: (c + 1) * nv].reshape(nq, nq) for v in (got, want))
        assert (np.abs(g - w).max(axis=1) <= 1e-12 * np.abs(w).max(axis=1)).all()
    P = O.prolongation(O.Mesh(n), O.Mesh(n // 2))
    rc = torch.empty(P.shape[1], dtype=torch.float64, device="cuda")
    stokes.stokes_restrict(H.handle, H.levels - 1, dev(x), rc)
    assert close(rc, P.T @ x)
    e = si.random_vector(n // 2, 3)
    xf = dev(x)
    stokes.stokes_prolong_add(H.handle, H.levels - 1, dev(e), xf)
    assert close(xf, x + P @ e)
    H.close()


def test_operator_spreads_nonfinite_values_as_the_stencil_does():
    import paper_2401_06277_gb300 as pkg
    n = 192
    H = pkg.Hierarchy(n, coarse_n=6, restart=1)
    nq = 2 * n + 1
    x = dev(si.random_vector(n, 4))
    clean = H.apply(x).clone()
    x[100 * nq + 101] = float("nan")
    out = H.apply(x)
    bad = ~torch.isfinite(out[: nq * nq].view(nq, nq))
    rows, cols = torch.where(bad)
    assert rows.min() >= 98 and rows.max() <= 102 and cols.min() >= 99 and cols.max() <= 103
    ok = torch.isfinite(out)
    assert torch.allclose(out[ok], clean[ok], rtol=1e-12, atol=1e-12)
    H.close()


@pytest.mark.parametrize("n,coarse_n", [(640, 5), (704, 11)])
def test_prolongation_rows_per_thread(n, coarse_n):
    """The sizes on both sides of a change in the coarse rows a thread walks."""
    import paper_2401_06277_gb300 as pkg
    from paper_2401_06277_gb300 import stokes
    H = pkg.Hierarchy(n, coarse_n=coarse_n, restart=1)
    P = O.prolongation(O.Mesh(n), O.Mesh(n // 2))
    e, x = si.random_vector(n // 2, 3), si.random_vector(n, 4)
    xf = dev(x)
    stokes.stokes_prolong_add(H.handle, H.levels - 1, dev(e), xf)
    assert close(xf, x + P @ e)
    H.close()
