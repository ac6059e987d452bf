"""The tensor-core FP64 sweep (n >= 56) entry by entry, for residuals whose size changes
within a strip of 128 cells.

Bar: the a-priori bound of a sweep by FP64 patch solves, oracle.rounding's form of it (a
backward-stable solve per patch) with the FP64 unit roundoff 2^-53 in place of 2^-24."""
import numpy as np
import pytest
import torch

import stokes_inputs as si
from oracle import rounding as RB
from oracle import stokes_oracle as O

pytestmark = pytest.mark.gpu

N = 160
_LV = []


def level():
    if not _LV:
        _LV.append(O.build_hierarchy(N, coarse_n=5).levels[-1])
    return _LV[0]


def field(form, rng):
    n, nq = N, 2 * N + 1
    j, i = np.mgrid[0:nq, 0:nq]
    u, v = rng.standard_normal((2, nq, nq))
    p = rng.standard_normal((n + 1, n + 1)) / n          # pressure rows carry a factor h
    if form.startswith(("columns", "rows")):
        s = 2.0 ** ((i if form.startswith("columns") else j) * (0.75 if form.endswith("up") else -0.75))
        u, v, p = u * s, v * s, p * s[::2, ::2]
    elif form == "spikes":
        u[101, 90] = 2.0 ** 60
        p[60, 70] = 2.0 ** 40
    elif form == "any size":
        u, v, p = (a * 2.0 ** rng.integers(-40, 41, a.shape) for a in (u, v, p))
    elif form == "tiny":
        u, v, p = (a * 2.0 ** -930 for a in (u, v, p))
    elif form == "sparse":
        u, v, p = (np.where(rng.random(a.shape) < 0.001, a * 2.0 ** rng.integers(-60, 1, a.shape), 0.0) for a in (u, v, p))
    elif form == "p only":
        u, v = 0.0 * u, 0.0 * v
        p = p * 2.0 ** rng.integers(-30, 1, p.shape)
    return np.concatenate([np.ravel(u), np.ravel(v), np.ravel(p)])


FORMS = ["plain", "columns up", "columns down", "rows up", "rows down", "spikes", "any size", "tiny", "sparse", "p only"]


@pytest.mark.parametrize("form", FORMS)
def test_sweep_keeps_every_entry(form):
    import paper_2401_06277_gb300 as pkg
    from paper_2401_06277_gb300 import stokes
    H, lv = pkg.Hierarchy(N, coarse_n=5, restart=1), level()
    assert stokes.stokes_level_tile(H.handle, H.levels - 1) == 8
    b = field(form, np.random.default_rng(FORMS.index(form)))
    scale = 2.0 ** 900 if form == "tiny" else 1.0       # the reference in the normal range
    want = O.vanka_sweep(lv, np.zeros_like(b), b * scale, 0.7)
    bound = RB.sweep_error_bound(lv, None, b * scale, 0.7) * 2.0 ** -29
    got = H.sweep(None, torch.from_numpy(b).cuda()).cpu().numpy() * scale
    assert (np.abs(got - want) <= bound).all(), (np.abs(got - want) / np.maximum(bound, 1e-300)).max()
    H.close()


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("where", ["u", "p", "near the wall"])
def test_sweep_spreads_nonfinite_values_as_the_patches_do(where, bad):
    """Exactly the dofs of the patches that hold the bad residual are not finite; the others
    are what they are without it."""
    import paper_2401_06277_gb300 as pkg
    n, nq, lv = N, 2 * N + 1, level()
    H = pkg.Hierarchy(N, coarse_n=5, restart=1)
    b = si.random_vector(n, 9)
    k = {"u": 101 * nq + 101, "p": 2 * nq * nq + 50 * (n + 1) + 61, "near the wall": nq * nq + 101 * nq + 3}[where]
    clean = H.sweep(None, torch.from_numpy(b).cuda()).cpu().numpy()
    b[k] = bad
    out = H.sweep(None, torch.from_numpy(b).cuda()).cpu().numpy()
    hit = np.zeros(len(b), dtype=bool)
    for dofs in lv.patch_dofs[(lv.patch_dofs == k).any(axis=1)]:
        hit[dofs[dofs >= 0]] = True
    free = np.zeros((nq, nq), dtype=bool)
    free[1:-1, 1:-1] = True
    hit &= np.concatenate([free.ravel(), free.ravel(), np.ones((n + 1) ** 2, dtype=bool)])   # Dirichlet rows are identities
    assert not np.isfinite(out[hit]).any()
    assert np.isfinite(out[~hit]).all()
    assert np.abs(out - clean)[~hit].max() <= 1e-13 * np.abs(clean).max()
    H.close()
