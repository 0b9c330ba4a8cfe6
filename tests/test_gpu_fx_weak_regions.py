"""Lattices that are ordinary in one part and near the unit matrix (or minus it) in another: the small gauge
force there, and the small off-diagonal entries of the fat and Naik links, keep FP64's relative accuracy,
whether the part is most of the lattice (the FP64 kernels then do all of it) or a few links (done one by one)."""

import numpy as np
import pytest
import torch

import oracle.gauge_force as ogf
import oracle.links as olk
import synth
from gpu_common import dev, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]

COEF = (1.0, -0.083, -0.008)


def _mixed(dims, eps, inside, seed):
    """Thin links, near 1 where `inside` (a mask of sites) holds."""
    thin = synth.gauge_field(dims, 0.3, seed, return_thin=True)[2].copy()
    thin[inside] = synth.gauge_field(dims, eps, seed + 1, return_thin=True)[2][inside]
    return thin


def _coords(dims):
    lex = np.arange(np.prod(dims))
    return np.stack(np.unravel_index(lex, dims[::-1])[::-1], axis=-1)


def _interior(dims, inside):
    """Sites all of whose loops' links lie inside: every site within two steps (and their links' far ends)."""
    grid = inside.reshape(dims[::-1])
    for axis in range(4):
        grid = np.all([np.roll(grid, k, axis) for k in range(-3, 3)], axis=0)
    return grid.reshape(-1)


@pytest.mark.parametrize("eps", [1e-6, 1e-3, 0.02])
@pytest.mark.parametrize("shape", ["slab", "box"])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_small_forces_in_part_of_a_lattice(eps, shape, sign):
    import paper_1712_00143_gb300 as stag

    dims = (4, 4, 4, 12) if shape == "slab" else (8, 8, 10, 10)
    c = _coords(dims)
    inside = c[:, 3] >= 3 if shape == "slab" else (c < 6).all(axis=1)
    thin = _mixed(dims, eps, inside, 1100)
    if sign < 0:  # antiperiodic in t
        thin[c[:, 3] == (7 if shape == "slab" else 3), 3] *= -1.0
    F = stag.stag_gauge_force(dims, dev(thin), 6.0, *COEF)
    torch.cuda.synchronize()
    F, want = F.cpu().numpy(), ogf.force(thin, dims, 6.0, *COEF)
    terms = 2.0 * (6 + 18 * 0.083 + 24 * 0.008)
    assert np.abs(F - want).max() <= 4e-15 * terms
    deep = _interior(dims, inside)
    assert deep.any() and np.abs(want[deep]).max() < 10 * terms * eps
    # FP64 sums of such links are off by a few 2^-53 of the largest of their own terms, which are of the force's size
    assert np.linalg.norm((F - want)[deep]) <= 1e-14 * np.linalg.norm(want[deep])


@pytest.mark.parametrize("eps", [1e-6, 1e-3, 0.01])
@pytest.mark.parametrize("shape", ["slab", "box"])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_small_entries_of_built_links(eps, shape, sign):
    import paper_1712_00143_gb300 as stag

    dims = (4, 4, 4, 12) if shape == "slab" else (8, 8, 10, 10)
    c = _coords(dims)
    inside = c[:, 3] >= 3 if shape == "slab" else (c < 6).all(axis=1)
    thin = _mixed(dims, eps, inside, 1102)
    if sign < 0:
        thin[c[:, 3] == (7 if shape == "slab" else 3), 3] *= -1.0
    fat, lng = stag.stag_build_links(dims, dev(thin))
    torch.cuda.synchronize()
    deep, off = _interior(dims, inside), ~np.eye(3, dtype=bool)
    for got, want in ((fat.cpu().numpy(), olk.fat_links(thin, dims)), (lng.cpu().numpy(), olk.naik_links(thin, dims))):
        assert np.linalg.norm(got - want) <= 1e-15 * np.linalg.norm(want)
        got, want = got[deep][..., off], want[deep][..., off]
        assert np.linalg.norm(got - want) <= 1e-14 * np.linalg.norm(want)


@pytest.mark.parametrize("eps", [0.02, 0.05, 0.08, 0.1, 0.15])
def test_weak_fields_on_every_route(eps):
    """Whole lattices from all links near 1 (FP64 at once) through a share of them (marked, done one by one) to
    none; a force's error against the reference's own, 4e-15 of the sum of its terms, and its own size."""
    import paper_1712_00143_gb300 as stag

    dims = (4, 6, 10, 6)
    thin = synth.gauge_field(dims, eps, 1104, return_thin=True)[2]
    F = stag.stag_gauge_force(dims, dev(thin), 6.0, *COEF)
    fat, lng = stag.stag_build_links(dims, dev(thin))
    torch.cuda.synchronize()
    want = ogf.force(thin, dims, 6.0, *COEF)
    assert np.linalg.norm(F.cpu().numpy() - want) <= 5e-16 * np.linalg.norm(want)
    off = ~np.eye(3, dtype=bool)
    for got, ref in ((fat.cpu().numpy(), olk.fat_links(thin, dims)), (lng.cpu().numpy(), olk.naik_links(thin, dims))):
        assert np.linalg.norm(got - ref) <= 4e-16 * np.linalg.norm(ref)
        assert np.linalg.norm((got - ref)[..., off]) <= 6e-16 * np.linalg.norm(ref[..., off])
