"""The FP64 sweep as an exact digit contraction on the tensor cores, against the
oracle's patch-by-patch sweep.

Grids: the smallest it serves and ragged ones (strips of 128 cells, row pairs, an odd
number of interior rows on every grid), zero guess and a general iterate.  Residuals
whose size changes along the walk make it renew its common exponent; each dof must
then be as accurate as its own neighbourhood: within 2e-14 of the largest correction
that residuals of the size found within 12 nodes could cause (the contraction rounds
the residual at 2^-54 of the largest in reach, which is less than 1e-16; FP64 dot
products of 171 terms near the boundary and the oracle's own LU solves set the
rest).  Non-finite residuals and an expired wait are reported, not hidden."""
import numpy as np
import pytest
import torch
from scipy.ndimage import maximum_filter

import stokes_inputs as si
from oracle import stokes_oracle as O

pytestmark = pytest.mark.gpu

_LV = {}


def level(n, coarse_n):
    if (n, coarse_n) not in _LV:
        _LV[n, coarse_n] = O.build_hierarchy(n, coarse_n=coarse_n).levels[-1]
    return _LV[n, coarse_n]


def hierarchy(n, coarse_n):
    import paper_2401_06277_gb300 as pkg
    from paper_2401_06277_gb300 import stokes
    H = pkg.Hierarchy(n, coarse_n=coarse_n)
    assert stokes.stokes_level_tile(H.handle, H.levels - 1) == 8
    return H


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("n,coarse_n", [(56, 7), (64, 4), (96, 6), (128, 4), (160, 5), (256, 4)])
def test_tc64_sweep_matches_patch_sweep(n, coarse_n):
    H, lv = hierarchy(n, coarse_n), level(n, coarse_n)
    b, x = si.random_vector(n, 5 + n), si.random_vector(n, 6 + n)
    for guess in (None, x):
        want = O.vanka_sweep(lv, np.zeros_like(b) if guess is None else guess, b, 0.7)
        got = H.sweep(None if guess is None else dev(guess), dev(b)).cpu().numpy()
        err = np.abs(got - want).max() / np.abs(want).max()
        assert err <= 1e-12, (n, guess is None, err)
    H.close()


@pytest.mark.parametrize("slope", [-0.75, -0.25, 0.25, 0.75])
@pytest.mark.parametrize("axis", [0, 1])
def test_tc64_follows_the_size_of_the_residual(slope, axis):
    """Residuals growing or falling by 2^slope per node row (along the walk: 2^(2 x 254 x
    0.75) in all) or, gently, per column."""
    n = 128
    H, lv = hierarchy(n, 4), level(n, 4)
    nq, nv = 2 * n + 1, (2 * n + 1) ** 2
    b = si.random_vector(n, 77)
    k = np.arange(nq) * (slope if axis == 0 else slope / 128)
    amp = 2.0 ** (k[:, None] + np.zeros(nq) if axis == 0 else k[None, :] + np.zeros((nq, 1)))
    b[:nv] *= amp.ravel()
    b[nv: 2 * nv] *= amp.ravel()
    b[2 * nv:] *= amp[::2, ::2].ravel() / n       # pressure rows carry a factor h
    want = O.vanka_sweep(lv, np.zeros_like(b), b, 0.7)
    got = H.sweep(None, dev(b)).cpu().numpy()
    for block, m, size in ((slice(0, nv), nq, 25), (slice(nv, 2 * nv), nq, 25), (slice(2 * nv, None), n + 1, 13)):
        w, g = want[block].reshape(m, m), got[block].reshape(m, m)
        near = maximum_filter(np.abs(w), size=size)
        assert (np.abs(g - w) <= 2e-14 * near).all(), (np.abs(g - w) / near).max()
    H.close()


def test_tc64_reports_nonfinite_and_zero_residuals():
    n = 128
    H = hierarchy(n, 4)
    nq = 2 * n + 1
    assert float(H.sweep(None, torch.zeros(H.N, dtype=torch.float64, device="cuda")).abs().max()) == 0.0
    for bad in (float("nan"), float("inf")):
        b = dev(si.random_vector(n, 9))
        b[100 * nq + 101] = bad
        out = H.sweep(None, b)
        u = out[: nq * nq].view(nq, nq)
        assert not torch.isfinite(u[100, 101]) and torch.isfinite(u[10]).all()
    H.close()


def test_tc64_expired_wait_is_reported_and_recovered():
    from paper_2401_06277_gb300 import stokes
    n = 128
    H, lv = hierarchy(n, 4), level(n, 4)
    b = si.random_vector(n, 3)
    stokes.stokes_test_set_wait_limit(H.handle, 0)
    H.sweep(None, dev(b))
    assert stokes.stokes_device_status(H.handle, allow_timeout=True) == stokes.STOKES_ERR_TIMEOUT
    stokes.stokes_test_set_wait_limit(H.handle, -1)
    want = O.vanka_sweep(lv, np.zeros_like(b), b, 0.7)
    got = H.sweep(None, dev(b)).cpu().numpy()
    assert stokes.stokes_device_status(H.handle) == stokes.STOKES_OK
    assert np.abs(got - want).max() <= 1e-12 * np.abs(want).max()
    H.close()
