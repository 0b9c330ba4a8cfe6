"""The fermion force through the fixed-point kernels, at the sizes and inputs where they can go wrong:
volumes that are not a multiple of the 32-site tile, solution pairs whose sites differ by many orders of
magnitude, zeros, one and the largest number of terms, unusual weights and coefficients, and inputs
(links that are not SU(3) or all close to 1, vectors out of range or not finite) that take the FP64 kernels."""

import numpy as np
import pytest
import torch

import oracle.fermion_force as ff
import synth
from gpu_common import dev, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]

FULL = (1.0, 0.125, -1.0 / 24.0)


def _force(dims, thin, xs, ys, alphas, coef):
    import paper_1712_00143_gb300 as stag

    F = stag.stag_fermion_force(dims, dev(thin), dev(xs), dev(ys), alphas, *coef)
    torch.cuda.synchronize()
    return F.cpu().numpy()


def _check(dims, thin, xs, ys, alphas, coef=FULL, link_size=1.0):
    got = _force(dims, thin, xs, ys, alphas, coef)
    want = ff.fermion_force(thin, list(xs), list(ys), alphas, dims, *coef)
    # a link's force sums 22 outer products through up to four links each: FP64 is off by at most some
    # 6 * 5 * 2^-53 = 3.4e-15 of the sum of their sizes, taken with the largest outer product anywhere
    g = sum(abs(a) * np.abs(x).max() * np.abs(y).max() for a, x, y in zip(alphas, xs, ys)) * 3
    size = (abs(coef[0]) + 18 * abs(coef[1]) * link_size**2 + 3 * abs(coef[2]) * link_size**2) * link_size * g
    assert np.abs(got - want).max() <= 3.4e-15 * size
    return got, want


def _pairs(dims, n, seed=0):
    xs = np.stack([synth.random_spinor(dims, 90 + seed + i) for i in range(n)])
    ys = np.stack([synth.random_spinor(dims, 190 + seed + i) for i in range(n)])
    return xs, ys


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (4, 6, 10, 6), (6, 6, 6, 6), (10, 4, 14, 4)])
@pytest.mark.parametrize("n", [1, 5, 32])
def test_tiles_and_terms(dims, n):
    thin = synth.gauge_field(dims, 0.3, 1090, return_thin=True)[2]
    xs, ys = _pairs(dims, n)
    _check(dims, thin, xs, ys, [0.3 - 0.02 * i for i in range(n)])


@pytest.mark.parametrize("coef", [(1.0, 0.0, 0.0), (0.0, 1.0, 0.0), (0.0, 0.0, 1.0), (0.0, 0.0, 0.0), (1e-3, 2.0**40, -7.0),
                                  (1e-250, 0.0, 0.0)])
def test_coefficients(coef):
    dims = (4, 6, 4, 6)
    thin = synth.gauge_field(dims, 0.4, 1091, return_thin=True)[2]
    _check(dims, thin, *_pairs(dims, 2), [1.0, -2.0], coef)


@pytest.mark.parametrize("kind", ["wide", "point", "zero_term", "zero", "weights", "large"])
def test_vectors(kind):
    dims = (6, 4, 6, 8)
    thin = synth.gauge_field(dims, 0.3, 1092, return_thin=True)[2]
    xs, ys = _pairs(dims, 3)
    alphas = [0.5, 0.25, -1.0]
    rng = np.random.default_rng(2)
    if kind == "wide":
        xs *= 10.0 ** rng.uniform(-9, 9, size=(3, xs.shape[1], 1))
        ys *= 10.0 ** rng.uniform(-9, 9, size=(3, ys.shape[1], 1))
    elif kind == "point":
        keep = xs[:, 7].copy()
        xs[:] = 0.0
        xs[:, 7] = keep
    elif kind == "zero_term":
        xs[1] = 0.0
        alphas[2] = 0.0
    elif kind == "zero":
        xs[:] = 0.0
    elif kind == "weights":
        alphas = [1e30, -1e-30, 1e10]
    else:  # beyond the integer kernels' exponents
        xs *= 1e100
        ys *= 1e-90
    got, want = _check(dims, thin, xs, ys, alphas)
    if kind in ("wide", "point"):  # a site's own size: links far from the large values keep their accuracy
        size = np.abs(want).max(axis=(2, 3))
        far = size < 1e-6 * size.max()
        assert np.isfinite(got).all() and (np.abs(got - want).max(axis=(2, 3))[far] <= 1e-6 * size.max()).all()
    if kind == "zero":
        assert (got == 0.0).all()


@pytest.mark.parametrize("kind", ["near_one", "scaled"])
def test_other_links(kind):
    dims = (4, 6, 4, 4)
    thin = synth.gauge_field(dims, 1e-4 if kind == "near_one" else 0.3, 1093, return_thin=True)[2]
    size = 1.25 if kind == "scaled" else 1.0
    _check(dims, size * thin, *_pairs(dims, 2), [1.0, 0.5], FULL, size)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_not_finite(bad):
    dims = (6, 4, 6, 8)
    thin = synth.gauge_field(dims, 0.3, 1094, return_thin=True)[2]
    xs, ys = _pairs(dims, 2)
    xs[1, 11, 2] = bad
    got = _force(dims, thin, xs, ys, [1.0, 0.5], FULL)
    with np.errstate(invalid="ignore"):
        want = ff.fermion_force(thin, list(xs), list(ys), [1.0, 0.5], dims, *FULL)
    ok = np.isfinite(want).all(axis=(2, 3))
    assert not ok.all() and (np.isfinite(got).all(axis=(2, 3)) == ok).all()
    assert np.abs(got[ok] - want[ok]).max() <= 1e-13 * np.abs(want[ok]).max()
