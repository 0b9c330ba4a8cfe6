"""The FP64 operator's fixed-point sums at the largest values its range check admits, through the form with
a thread per hop, the one with a thread per site, and a group: one site whose sixteen hops all point the
same way, in a field whose other links are nearly as large."""

import math

import numpy as np
import pytest

import oracle
import synth
from gpu_common import requires_gpu
from test_gpu_fx_dslash import _run

pytestmark = [pytest.mark.gpu, requires_gpu]

# 48 products per sum: FP64 rounds to within 96 * 2^-53 of (sum over hops of the row's norm) x (largest vector's norm)
BOUND = 1.1e-14

# (lattice, vectors): a thread per hop, a group (a thread per site), a thread per site
FORMS = [((8, 8, 8, 8), 1), ((8, 8, 8, 8), 2), ((16, 16, 16, 18), 1)]


def _hops(dims, site, parity):
    """For the hops t = 4 mu + {+1, -1, +3, -3} of one output site: (field, link's site, mu, sign, adjoint,
    neighbour's index), so that the hop's matrix is sign / 2 times that link (or its adjoint)."""
    lex = oracle.parity_sites(dims, parity)
    c = oracle.site_coords(dims, lex)
    here = int(lex[site])
    x = np.unravel_index(here, dims[::-1])[::-1]
    out = []
    for mu in range(4):
        eta = -1.0 if sum(x[:mu]) % 2 else 1.0
        for which, k in ((0, 1), (0, -1), (1, 3), (1, -3)):
            n = int(oracle.neighbour_lex(dims, c, mu, k)[site])
            out.append((which, here if k > 0 else n, mu, eta if k > 0 else -eta, k < 0, n // 2))
    return out


def _field(dims, site, parity, matrices, others):
    """A field whose hop matrices are (1 + i) others, up to signs, except the site's, which are given."""
    links = [np.full((math.prod(dims), 4, 3, 3), (1 + 1j) * 2 * others) for _ in range(2)]
    for (which, lk, mu, sign, adj, _), m in zip(_hops(dims, site, parity), matrices):
        links[which][lk, mu] = (2 * sign * m).conj().T if adj else 2 * sign * m
    return links


def _compare(dims, nrhs, site, fat, lng, psi):
    got = _run(dims, fat, lng, np.stack([psi] * nrhs) if nrhs > 1 else psi, 0, nrhs).reshape(nrhs, -1, 3)
    want = oracle.dslash(fat, lng, psi, dims, 0)
    row = 8 * 0.5 * np.sqrt((np.abs(fat) ** 2).sum(-1)).max() + 8 * 0.5 * np.sqrt((np.abs(lng) ** 2).sum(-1)).max()
    size = row * np.sqrt((np.abs(psi) ** 2).sum(-1)).max()
    for g in got:
        assert np.abs(g - want).max() <= BOUND * size, (site, g[site], want[site])


@pytest.mark.parametrize("dims,nrhs", FORMS)
@pytest.mark.parametrize("phase", [1, -1, 1j])
def test_sums_before_a_larger_neighbour(dims, nrhs, phase):
    site = 37
    z, c = 5e-3, 0.5238  # the site's row norms add up to 8.99 x 2, the other sites' to at most 7.7 x 2
    matrices = [np.full((3, 3), (1 + 1j) * (z if t in (0, 15) else c) * (1 if t in (0, 15) else phase)) for t in range(16)]
    fat, lng = _field(dims, site, 0, matrices, 0.3)
    psi = synth.random_spinor(dims, 77) * 0.1
    for t, h in enumerate(_hops(dims, site, 0)):
        psi[h[5]] = (1 + 1j) * (1.99 if t == 0 else 7.99 if t == 15 else 3.999)
    _compare(dims, nrhs, site, fat, lng, psi)


@pytest.mark.parametrize("dims,nrhs", FORMS)
@pytest.mark.parametrize("c", [1 - 2.0**-40, 0.95])
def test_one_hop_of_large_rows(dims, nrhs, c):
    """One hop's entries (1 + i) c beside small ones, and vectors whose low words are nearly full."""
    site = 37
    low = 1.0 + (2.0**52 - 1) * 2.0**-52
    matrices = [np.full((3, 3), (1 + 1j) * (c if t == 4 else 0.02)) for t in range(16)]
    fat, lng = _field(dims, site, 0, matrices, 0.02)
    psi = synth.random_spinor(dims, 78) * 0.1
    for h in _hops(dims, site, 0):
        psi[h[5]] = (1 + 1j) * low
    _compare(dims, nrhs, site, fat, lng, psi)


def _sizes(dims, fat, lng, psi, parity):
    """Per output site and row, the sum over hops of (row norm) x (vector norm)."""
    Vh = len(psi)
    lex = oracle.parity_sites(dims, parity)
    c = oracle.site_coords(dims, lex)
    norm = np.sqrt((np.abs(psi) ** 2).sum(-1))
    out = np.zeros((Vh, 3))
    for mu in range(4):
        for links, k in ((fat, 1), (lng, 3)):
            fwd, back = oracle.neighbour_lex(dims, c, mu, k), oracle.neighbour_lex(dims, c, mu, -k)
            out += 0.5 * np.sqrt((np.abs(links[lex, mu]) ** 2).sum(-1)) * norm[fwd // 2][:, None]
            out += 0.5 * np.sqrt((np.abs(links[back, mu]) ** 2).sum(-2)) * norm[back // 2][:, None]
    return out


@pytest.mark.parametrize("dims,nrhs", FORMS)
@pytest.mark.parametrize("kind", ["zero_naik", "zero_matrices", "small_direction", "small_matrices"])
def test_accuracy_is_that_of_each_matrix(dims, nrhs, kind):
    """Vectors far larger behind zero matrices, or seen through matrices far smaller than the others: every row
    is known to within 96 * 2^-53 of the sizes of its own products (twice, with the reference's own rounding)."""
    fat, lng = synth.gauge_field(dims, 0.3, 1087)
    rng = np.random.default_rng(4)
    psi = synth.random_spinor(dims, 79)
    if kind == "zero_naik":  # a third of the sites far larger: three sites away they must not count
        lng[:] = 0.0
        psi *= np.where(rng.uniform(size=(len(psi), 1)) < 0.3, 2.0**40, 1.0)
    elif kind == "zero_matrices":  # the links that leave every third site
        lex = np.arange(len(fat))
        fat[lex % 3 == 0] = 0.0
        lng[lex % 3 == 0] = 0.0
        psi *= 2.0 ** rng.integers(-30, 30, size=(len(psi), 1))
    elif kind == "small_direction":
        fat[:, 2] *= 2.0**-30
        lng[:, 2] *= 2.0**-30
        psi *= np.where(rng.uniform(size=(len(psi), 1)) < 0.01, 1.0, 0.0)
    else:
        scale = 2.0 ** rng.integers(-45, 45, size=(len(fat), 4, 1, 1))
        fat, lng = fat * scale, lng * scale
    got = _run(dims, fat, lng, np.stack([psi] * nrhs) if nrhs > 1 else psi, 0, nrhs).reshape(nrhs, -1, 3)
    want = oracle.dslash(fat, lng, psi, dims, 0)
    size = _sizes(dims, fat, lng, psi, 0)
    for g in got:
        assert (np.abs(g - want) <= 2 * BOUND * size).all(), (np.abs(g - want) / np.maximum(size, 1e-300)).max()
