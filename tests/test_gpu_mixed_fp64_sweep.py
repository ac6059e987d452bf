"""stokes_vanka_sweep is FP64 on every hierarchy: on a mixed one, with the split tile
configurations and with the Braess-Sarazin smoothers too, none of whose FP64 scratch a
mixed hierarchy holds.  Bar 1e-12, as for the FP64 form."""
import numpy as np
import pytest
import torch

import stokes_inputs as si
from oracle import stokes_oracle as O

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("kw", [{"tile": 4}, {"tile": 5}, {"smoother": 2}, {"smoother": 3}])
@pytest.mark.parametrize("n", [8, 32])
def test_fp64_sweep_of_a_mixed_hierarchy(n, kw):
    import paper_2401_06277_gb300 as pkg
    from paper_2401_06277_gb300 import stokes
    # with the shortest restart: the smallest workspace
    H = pkg.Hierarchy(n, prec=stokes.STOKES_MIXED_FP32, restart=1, **kw)
    for l in range(H.levels):
        nl = stokes.stokes_level_n(H.handle, l)
        lv = O.build_level(nl, 1.0)
        x, b = si.random_vector(nl, 30 + l), si.random_vector(nl, 40 + l)
        sm = kw.get("smoother", 0)
        sweep = {0: lambda x_: O.vanka_sweep(lv, x_, b, 0.7), 2: lambda x_: O.braess_sarazin_sweep(lv, x_, b, O.BSParams()),
                 3: lambda x_: O.schur_uzawa_sweep(lv, x_, b, O.BSParams())}[sm]
        for guess in (None, x):
            want = sweep(np.zeros_like(b) if guess is None else x)
            out = torch.empty(lv.mesh.ndof, dtype=torch.float64, device="cuda")
            stokes.stokes_vanka_sweep(H.handle, l, None if guess is None else dev(x), dev(b), out)
            assert np.abs(out.cpu().numpy() - want).max() <= 1e-12 * np.abs(want).max(), (l, guess is None)
    H.close()
