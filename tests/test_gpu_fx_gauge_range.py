"""The gauge force with couplings and coefficients near the small end of the double range: the factor that
turns fixed point into doubles must stay a normal number, or the FP64 kernels take the call."""

import numpy as np
import pytest

import synth
from gpu_common import requires_gpu
from test_gpu_fx_gauge_force import COEF, _check

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("beta", [0.0, 2.0**-40, 2.0**-51, -(2.0**-100), 2.0**59])
@pytest.mark.parametrize("e", [0, -400, -880])
def test_small_couplings(beta, e):
    dims = (4, 6, 4, 4)
    coef = tuple(c * 2.0**e for c in COEF)
    F, want = _check(dims, synth.gauge_field(dims, 0.3, 1074, return_thin=True)[2], beta, coef)
    assert beta != 0.0 or not F.any()
    # (norms of numbers this small underflow)
    if beta:
        unit = 2.0 ** (e - 3) * abs(beta)
        assert np.linalg.norm((F - want) / unit) <= 1e-14 * np.linalg.norm(want / unit)
