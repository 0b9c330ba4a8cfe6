"""Link construction through the fixed-point kernels, at the sizes and inputs where they can go wrong:
lattices whose volume is not a multiple of the 32-site tile, links at and beyond the edges of the
integer range (which take the FP64 kernel), and unusual coefficients."""

import numpy as np
import pytest
import torch

import oracle.links as olk
import synth
from gpu_common import dev, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]

# an entry of F is a sum of 13 terms of up to 3 products each: FP64 itself is off by about
# 13 * 6 * 2^-53 = 9e-15 of the largest term in the worst case; the same bound holds here
BOUND = 9e-15


def _build(dims, thin, **kw):
    import paper_1712_00143_gb300 as stag

    fat, lng = stag.stag_build_links(dims, dev(thin), **kw)
    torch.cuda.synchronize()
    return fat.cpu().numpy(), lng.cpu().numpy()


def _check(dims, thin, c1=1.0, c_staple=0.125, c3=-1.0 / 24.0):
    fat, lng = _build(dims, thin, c1=c1, c_staple=c_staple, c3=c3)
    fo, lo = olk.fat_links(thin, dims, c1=c1, c_st=c_staple), olk.naik_links(thin, dims, c3=c3)
    scale = np.abs(thin).max()
    assert np.abs(fat - fo).max() <= BOUND * (abs(c1) * scale + 6 * abs(c_staple) * scale**3)
    assert np.abs(lng - lo).max() <= BOUND * abs(c3) * scale**3


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (4, 6, 10, 6), (6, 6, 6, 6), (10, 4, 14, 4)])
@pytest.mark.parametrize("eps", [1e-9, 0.01, 0.05, 0.3, 2.0])
def test_tiles_and_distance_from_unity(dims, eps):
    _check(dims, synth.gauge_field(dims, eps, 1060, return_thin=True)[2])


@pytest.mark.parametrize("coef", [(0.0, 0.0, 0.0), (0.0, -3.0, 1e-200), (1e300, 1e250, -1e299), (-2.0**-20, 1.0, 7.0)])
def test_coefficients(coef):
    dims = (4, 6, 10, 6)
    _check(dims, synth.gauge_field(dims, 0.3, 1061, return_thin=True)[2], *coef)


@pytest.mark.parametrize("kind", ["scaled", "one_link", "zero", "large"])
def test_other_matrices(kind):
    """Links that are not SU(3) matrices are multiplied as they are."""
    dims = (6, 6, 6, 6)
    thin = synth.gauge_field(dims, 0.3, 1062, return_thin=True)[2].copy()
    if kind == "scaled":
        thin *= 1.7
    elif kind == "one_link":
        thin[777, 2] *= 1.001
    elif kind == "zero":
        thin[:] = 0.0
    else:
        thin[5, 1, 0, 0] = 1e30
    _check(dims, thin)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_not_finite(bad):
    """A bad entry reaches every link whose definition holds it, and no other."""
    dims = (6, 4, 4, 6)
    thin = synth.gauge_field(dims, 0.3, 1063, return_thin=True)[2].copy()
    ref_fat, ref_lng = _build(dims, thin)
    thin[100, 3, 1, 2] = bad
    fat, lng = _build(dims, thin)
    with np.errstate(invalid="ignore"):
        fo, lo = olk.fat_links(thin, dims), olk.naik_links(thin, dims)
    for got, want, ref in ((fat, fo, ref_fat), (lng, lo, ref_lng)):
        ok = np.isfinite(want).all(axis=(2, 3))
        assert (np.isfinite(got).all(axis=(2, 3)) == ok).all()
        assert np.abs(got[ok] - ref[ok]).max() <= BOUND
