"""The FP64 operator's fixed-point form at the sizes and values where it can go wrong: both kernel forms
(few sites: one thread per hop; many: one thread per site) and every group size, vectors whose
neighbours differ by many orders of magnitude, exact zeros, the ends of the double range, infinities and
NaN, and links whose range keeps them in doubles."""

import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_common import dev, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]

# A site's sum has 48 products of complex numbers; FP64 rounds it to within 96 * 2^-53 = 1.1e-14 of
# (largest link row norm) x (largest neighbour), whatever the order.
BOUND = 1.1e-14


def _stag():
    import paper_1712_00143_gb300 as stag

    return stag


def _largest_neighbour(psi, dims, out_parity):
    """Largest |component| among the sixteen neighbours of every output site."""
    lex = oracle.parity_sites(dims, out_parity)
    c = oracle.site_coords(dims, lex)
    m = np.abs(psi).max(axis=-1)
    out = np.zeros(len(lex))
    for mu in range(4):
        for k in (1, -1, 3, -3):
            out = np.maximum(out, m[oracle.neighbour_lex(dims, c, mu, k) // 2])
    return out


def _run(dims, fat, lng, psi, out_parity, nrhs=1):
    stag = _stag()
    h = stag.stag_load_links(dims, dev(fat), dev(lng), prec_mask=1 << stag.STAG_FP64)
    out = torch.empty(psi.shape, dtype=torch.complex128, device="cuda")
    stag.stag_dslash(h, out, dev(psi), out_parity, "fp64", nrhs=nrhs)
    got = out.cpu().numpy()
    h.free()
    return got


def _check(dims, fat, lng, psi, out_parity, got):
    want = oracle.dslash(fat, lng, psi, dims, out_parity)
    size = _largest_neighbour(psi, dims, out_parity)[:, None]
    assert (np.abs(got - want) <= BOUND * size).all(), (np.abs(got - want) / np.maximum(size, 1e-300)).max()


def _vector(kind, dims, seed=0):
    psi = synth.random_spinor(dims, 70 + seed)
    rng = np.random.default_rng(seed)
    if kind == "wide":  # sites twenty orders of magnitude apart
        psi *= 10.0 ** rng.uniform(-10, 10, size=(len(psi), 1))
    elif kind == "components":
        psi *= 2.0 ** rng.integers(-60, 60, size=psi.shape)
    elif kind == "point":
        keep = psi[5].copy()
        psi[:] = 0.0
        psi[5] = keep
    elif kind == "zero":
        psi[:] = 0.0
    elif kind == "large":
        psi *= 1e290
    elif kind == "small":
        psi *= 1e-290
    elif kind == "sparse":  # zero sites beside huge and tiny ones
        psi *= rng.choice([0.0, 1e-300, 1.0, 1e150], size=(len(psi), 1))
    return psi


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (4, 6, 8, 10), (6, 10, 4, 14)])
@pytest.mark.parametrize("kind", ["plain", "wide", "components", "point", "zero", "large", "small", "sparse"])
def test_values(dims, kind):
    fat, lng = synth.gauge_field(dims, 0.3, 1080)
    for p in (0, 1):
        psi = _vector(kind, dims, p)
        _check(dims, fat, lng, psi, p, _run(dims, fat, lng, psi, p))


@pytest.mark.parametrize("dims", [(16, 16, 16, 16), (16, 16, 16, 18)])
def test_both_sides_of_the_size_rule(dims):
    """2^15 sites per parity (the last of the small form) and just above it."""
    fat, lng = synth.gauge_field(dims, 0.3, 1081)
    for kind in ("plain", "sparse"):
        psi = _vector(kind, dims, 3)
        _check(dims, fat, lng, psi, 1, _run(dims, fat, lng, psi, 1))


@pytest.mark.parametrize("nrhs", [2, 3, 4, 5, 8])
def test_groups(nrhs):
    dims = (6, 10, 4, 14)
    fat, lng = synth.gauge_field(dims, 0.3, 1082)
    kinds = ["plain", "wide", "point", "sparse", "zero", "components", "large", "small"]
    psi = np.stack([_vector(kinds[r], dims, r) for r in range(nrhs)])
    got = _run(dims, fat, lng, psi, 0, nrhs)
    for r in range(nrhs):
        _check(dims, fat, lng, psi[r], 0, got[r])


@pytest.mark.parametrize("kind", ["scaled_direction", "one_small_matrix", "zero_naik", "large_rows", "huge"])
def test_other_links(kind):
    """Links that keep their doubles (a range too wide, a unit out of range), and others that need not."""
    dims = (4, 6, 8, 4)
    fat, lng = synth.gauge_field(dims, 0.3, 1083)
    if kind == "scaled_direction":
        fat[:, 3] *= 1e-7
        lng[:, 3] *= 1e-7
    elif kind == "one_small_matrix":
        fat[17, 2] *= 1e-12
    elif kind == "zero_naik":
        lng[:] = 0.0
    elif kind == "large_rows":  # every entry as large as the largest
        fat[:] = 1.0 + 1.0j
        lng[:] = 1.0 - 1.0j
    else:
        fat *= 1e200
        lng *= 1e200
    psi = _vector("plain", dims)
    want = oracle.dslash(fat, lng, psi, dims, 0)
    got = _run(dims, fat, lng, psi, 0)
    assert np.abs(got - want).max() <= BOUND * np.abs(psi).max() * max(np.abs(fat).max(), np.abs(lng).max()) * 2


def test_not_finite():
    """A NaN or an infinity reaches the sixteen neighbours' sums and no other."""
    dims = (8, 8, 8, 8)
    fat, lng = synth.gauge_field(dims, 0.3, 1084)
    psi = _vector("plain", dims)
    ref = _run(dims, fat, lng, psi, 1)
    for bad in (np.nan, np.inf, -np.inf):
        q = psi.copy()
        q[100, 1] = bad
        got = _run(dims, fat, lng, q, 1)
        with np.errstate(invalid="ignore"):
            ok = np.isfinite(oracle.dslash(fat, lng, q, dims, 1)).all(axis=1)
        assert (~ok).sum() == 16
        assert (np.isfinite(got).all(axis=1) == ok).all()
        assert (got[ok] == ref[ok]).all()


def test_solve_takes_the_same_result_with_either_form():
    """A point source to 1e-12 with links in fixed point, and with one matrix small enough to keep the doubles."""
    stag = _stag()
    dims = (6, 6, 8, 4)
    fat, lng = synth.gauge_field(dims, 0.3, 1085)
    b = _vector("point", dims)
    for small in (1.0, 1e-9):
        fat[40, 1] *= small
        h = stag.stag_load_links(dims, dev(fat), dev(lng))
        x = torch.zeros((h.Vh, 3), dtype=torch.complex128, device="cuda")
        for mode in ("plain64", "mixed32"):
            info = stag.stag_cg(h, x, dev(b), 0.1, mode=mode, tol=1e-12)
            assert info["converged"]
            assert oracle.true_residual(fat, lng, x.cpu().numpy(), b, 0.1, dims) <= 1.01e-12
        h.free()
