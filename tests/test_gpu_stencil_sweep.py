"""The FP64 sweep as one stencil (the composite of all patch solves) against the
oracle's patch-by-patch sweep.

Grids where it can go wrong: the smallest ones, on which every cell is within two
of a boundary or the interior is one cell wide; tile remainders (8 x 4 cells per
CTA); and the largest level the rule gives to it.  Iterates with a zero guess, and
with a residual on Dirichlet rows (identity rows).  The tolerance is the FP64
sweep's: 1e-12 of the largest entry."""
import numpy as np
import pytest
import torch

import stokes_inputs as si
from oracle import stokes_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,coarse_n", [(8, 4), (10, 5), (12, 6), (14, 7), (16, 4), (28, 7), (40, 5), (48, 6)])
def test_stencil_sweep_matches_patch_sweep(n, coarse_n):
    import paper_2401_06277_gb300 as pkg
    from paper_2401_06277_gb300 import stokes
    H = pkg.Hierarchy(n, coarse_n=coarse_n)
    assert stokes.stokes_level_tile(H.handle, H.levels - 1) == 7
    lv = O.build_hierarchy(n, coarse_n=coarse_n).levels[-1]
    b, x = si.random_vector(n, 5 + n), si.random_vector(n, 6 + n)
    for guess in (None, x):
        want = O.vanka_sweep(lv, np.zeros_like(b) if guess is None else guess, b, 0.7)
        got = H.sweep(None if guess is None else torch.from_numpy(guess).cuda(), torch.from_numpy(b).cuda())
        err = np.abs(got.cpu().numpy() - want).max() / np.abs(want).max()
        assert err <= 1e-12, (n, guess is None, err)
    H.close()
