"""An expired wait of the tensor-core FP64 operator (n >= 192) is reported, by the direct
calls and by a mixed-precision hierarchy, and the next call is right again."""
import numpy as np
import pytest
import torch

import stokes_inputs as si
from oracle import stokes_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["STOKES_FP64", "STOKES_MIXED_FP32"])
@pytest.mark.parametrize("call", ["apply", "residual"])
def test_expired_operator_wait_is_reported_and_recovered(prec, call):
    import paper_2401_06277_gb300 as pkg
    from paper_2401_06277_gb300 import stokes
    n = 192
    H = pkg.Hierarchy(n, coarse_n=6, prec=getattr(stokes, prec), restart=1)
    x, b = si.random_vector(n, 1), si.random_vector(n, 2)
    xd, bd = torch.from_numpy(x).cuda(), torch.from_numpy(b).cuda()
    run = (lambda: H.apply(xd)) if call == "apply" else (lambda: H.residual(bd, xd))
    stokes.stokes_test_set_wait_limit(H.handle, 0)
    run()
    assert stokes.stokes_device_status(H.handle, allow_timeout=True) == stokes.STOKES_ERR_TIMEOUT
    stokes.stokes_test_set_wait_limit(H.handle, -1)
    got = run().cpu().numpy()
    assert stokes.stokes_device_status(H.handle) == stokes.STOKES_OK
    want = O.build_level(n, 1.0).A @ x
    want = want if call == "apply" else b - want
    assert np.abs(got - want).max() <= 1e-13 * np.abs(want).max()
    H.close()
