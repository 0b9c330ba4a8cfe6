"""The gauge force through the fixed-point kernels, at the sizes and inputs where they can go wrong:
volumes that are not a multiple of the 32-site tile, links near the unit matrix and matrices that are
not SU(3) (which take the FP64 kernels), single loop types and extreme coefficients."""

import numpy as np
import pytest
import torch

import oracle.gauge_force as ogf
import synth
from gpu_common import dev, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]

COEF = (1.0, -0.083, -0.008)


def _check(dims, thin, beta, coef, size=1.0):
    import paper_1712_00143_gb300 as stag

    F = stag.stag_gauge_force(dims, dev(thin), beta, *coef)
    torch.cuda.synchronize()
    want = ogf.force(thin, dims, beta, *coef)
    # 48 terms of up to six products: FP64 itself is off by up to 6 * 6 * 2^-53 = 4e-15 of the sum of their sizes
    terms = abs(beta) / 3 * (6 * abs(coef[0]) * size**4 + (18 * abs(coef[1]) + 24 * abs(coef[2])) * size**6)
    assert np.abs(F.cpu().numpy() - want).max() <= 4e-15 * terms
    return F.cpu().numpy(), want


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (6, 4, 8, 4), (4, 10, 4, 6), (6, 6, 6, 6)])
@pytest.mark.parametrize("eps", [0.3, 1.5])
def test_tiles(dims, eps):
    _check(dims, synth.gauge_field(dims, eps, 1070, return_thin=True)[2], 6.0, COEF)


@pytest.mark.parametrize("coef", [(1.0, 0.0, 0.0), (0.0, 1.0, 0.0), (0.0, 0.0, -1.0), (0.0, 0.0, 0.0),
                                  (1e-3, 2.0**60, 1.0), (1e290, 0.0, -1e289)])
def test_loop_types(coef):
    dims = (4, 6, 4, 6)
    _check(dims, synth.gauge_field(dims, 0.4, 1071, return_thin=True)[2], -2.5, coef)


@pytest.mark.parametrize("eps", [1e-6, 1e-3])
def test_small_fields_keep_relative_accuracy(eps):
    """Links near 1: the force is of the order of eps and still known to FP64's relative accuracy."""
    dims = (4, 4, 6, 4)
    F, want = _check(dims, synth.gauge_field(dims, eps, 1072, return_thin=True)[2], 6.0, COEF)
    assert np.linalg.norm(F - want) <= 1e-13 * np.linalg.norm(want)


def test_other_matrices():
    """Links scaled away from SU(3): the table's parallelograms pair a link with its adjoint, so only plaquettes
    and rectangles have a definition to compare with."""
    dims = (4, 6, 4, 4)
    thin = 1.25 * synth.gauge_field(dims, 0.3, 1073, return_thin=True)[2]
    _check(dims, thin, 6.0, (1.0, 0.0, 0.0), 1.25)
