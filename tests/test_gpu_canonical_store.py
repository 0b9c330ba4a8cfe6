"""stag_dslash and stag_apply_m with the result stored as doubles by the operator kernel: whole and
partial warps (sites per parity on both sides of multiples of 32), every vector count, the output
aliasing the input, and values a float cannot hold as a normal number."""

import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_common import TOL_DSLASH, dev, rel_l2, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]

PRECS = ["fp64", "fp32", "fp16", "fx16", "fx16l"]


def _handle(dims, recon=12, seed=1100):
    import paper_1712_00143_gb300 as stag

    fat, lng = synth.gauge_field(dims, 0.3, seed)
    return stag, stag.stag_load_links(dims, dev(fat), dev(lng), recon_long=recon), fat, lng


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (4, 6, 6, 6), (6, 6, 6, 10)])
@pytest.mark.parametrize("prec", PRECS)
def test_every_vector_count(dims, prec):
    """128, 432 = 13.5 warps and 1080 = 33.75 warps of sites; 1 to 9 vectors, 11 and 13."""
    stag, h, fat, lng = _handle(dims)
    psi = np.stack([synth.random_spinor(dims, 110 + k) for k in range(13)])
    want = np.stack([oracle.dslash(fat, lng, p, dims, 1) for p in psi])
    for n in list(range(1, 10)) + [11, 13]:
        out = torch.full((n, h.Vh, 3), 7.0, dtype=torch.complex128, device="cuda")
        stag.stag_dslash(h, out, dev(psi[:n]), 1, prec, nrhs=n)
        got = out.cpu().numpy()
        for k in range(n):
            assert rel_l2(got[k], want[k]) < TOL_DSLASH[prec], (n, k)
    h.free()


@pytest.mark.parametrize("prec", PRECS)
def test_output_over_input(prec):
    """The output may be the input's memory: the same values as with two fields."""
    dims = (6, 6, 6, 10)
    stag, h, _, _ = _handle(dims)
    for n in (1, 2, 3, 6):
        psi = dev(np.stack([synth.random_spinor(dims, 130 + k) for k in range(n)]))
        apart, over = torch.empty_like(psi), psi.clone()
        stag.stag_dslash(h, apart, psi, 0, prec, nrhs=n)
        stag.stag_dslash(h, over, over, 0, prec, nrhs=n)
        assert torch.equal(apart, over)
    one = dev(synth.random_spinor(dims, 140))
    apart, over = torch.empty_like(one), one.clone()
    stag.stag_apply_m(h, apart, one, 0.1, prec=prec)
    stag.stag_apply_m(h, over, over, 0.1, prec=prec)
    assert torch.equal(apart, over)
    h.free()


def test_floats_at_the_ends():
    """FP32 results that are subnormal, zero, infinite or NaN widen to the same doubles."""
    dims = (4, 4, 4, 4)
    stag, h, fat, lng = _handle(dims, recon=18)
    base = synth.random_spinor(dims, 150)
    for scale in (1e-39, 1e-44, 0.0, 1e37):
        psi = base * scale
        out = torch.empty(psi.shape, dtype=torch.complex128, device="cuda")
        stag.stag_dslash(h, out, dev(psi), 1, "fp32")
        got = out.cpu().numpy()
        assert (got.real == got.real.astype(np.float32)).all() and (got.imag == got.imag.astype(np.float32)).all()
        want = oracle.dslash(fat, lng, psi, dims, 1)
        # subnormal terms are rounded to multiples of 2^-149, forty-eight of them per sum
        assert np.abs(got - want).max() <= 1e-5 * np.abs(want).max() + 96 * 2.0**-149
    psi = base.copy()
    psi[3, 1] = np.nan
    psi[40, 2] = np.inf
    out = torch.empty(psi.shape, dtype=torch.complex128, device="cuda")
    stag.stag_dslash(h, out, dev(psi), 1, "fp32")
    with np.errstate(invalid="ignore"):
        ok = np.isfinite(oracle.dslash(fat, lng, psi, dims, 1)).all(axis=1)
    assert (np.isfinite(out.cpu().numpy()).all(axis=1) == ok).all() and not ok.all()
    h.free()
