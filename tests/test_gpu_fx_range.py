"""The FP64 operator on link fields anywhere in the double range: uniformly scaled fields (the fixed-point
form's range check takes some and leaves the others in doubles), ordinary ones and ones whose every entry
is as large as the largest, through the small form, the one with a thread per site, and a group."""

import numpy as np
import pytest

import oracle
import synth
from gpu_common import requires_gpu
from test_gpu_fx_dslash import BOUND, _run, _vector

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("e", [-90, -70, -50, -40, 40, 50, 70, 90])
@pytest.mark.parametrize("rows", ["ordinary", "large"])
def test_scaled_fields(e, rows):
    dims = (4, 6, 8, 4)
    if rows == "ordinary":
        fat, lng = synth.gauge_field(dims, 0.3, 1086)
    else:  # entries of one size, row norms of sixteen hops up to 39 of it
        shape = synth.gauge_field(dims, 0.3, 1086)[0].shape
        fat, lng = np.full(shape, 1.0 + 1.0j), np.full(shape, 1.0 - 1.0j)
    fat, lng = fat * 2.0**e, lng * 2.0**e
    size = max(np.abs(fat).max(), np.abs(lng).max())
    psi = np.stack([_vector("plain", dims, r) for r in range(2)])
    for nrhs in (1, 2):
        got = _run(dims, fat, lng, psi if nrhs == 2 else psi[0], 0, nrhs).reshape(nrhs, -1, 3)
        for r in range(nrhs):
            want = oracle.dslash(fat, lng, psi[r], dims, 0)
            assert np.abs(got[r] - want).max() <= BOUND * np.abs(psi).max() * size * 2
