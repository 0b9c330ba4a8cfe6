"""Mixed-precision CG with the iterations of a reliable-update cycle in one cooperative kernel: lattices
whose sites fill their warps and blocks unevenly, one and several groups of sites per warp, both sides of
the size rule, every sloppy format, iteration caps, an initial guess, and sources that end it at once."""

import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_common import dev, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]

MODES = ["mixed32", "mixed16l", "mixedfx16", "mixed16"]


def _setup(dims, recon=18, seed=1110):
    import paper_1712_00143_gb300 as stag

    fat, lng = synth.gauge_field(dims, 0.3, seed)
    return stag, stag.stag_load_links(dims, dev(fat), dev(lng), recon_long=recon), fat, lng


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (4, 6, 6, 6), (10, 4, 6, 14), (8, 8, 8, 18), (8, 12, 10, 14)])
@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("recon", [12, 18])
def test_solves(dims, mode, recon):
    stag, h, fat, lng = _setup(dims, recon)
    b = synth.gaussian_source(dims, 5100)
    x = torch.zeros((h.Vh, 3), dtype=torch.complex128, device="cuda")
    info = stag.stag_cg(h, x, dev(b), 0.2, mode=mode, tol=1e-10)
    assert info["converged"] and info["reliable_updates"] >= 1
    assert oracle.true_residual(fat, lng, x.cpu().numpy(), b, 0.2, dims) <= 1.001e-10
    y = torch.zeros_like(x)  # the same again, bit for bit
    again = stag.stag_cg(h, y, dev(b), 0.2, mode=mode, tol=1e-10)
    assert torch.equal(x, y) and again["iters"] == info["iters"]
    h.free()


def test_iterations_are_those_of_plain_cg():
    """The count follows the FP64 oracle's, within the last update cycle."""
    dims = (8, 8, 8, 8)
    stag, h, fat, lng = _setup(dims)
    b = synth.gaussian_source(dims, 5101)
    _, want = oracle.cg(fat, lng, b, 0.1, dims, tol=1e-10)
    x = torch.zeros((h.Vh, 3), dtype=torch.complex128, device="cuda")
    info = stag.stag_cg(h, x, dev(b), 0.1, mode="mixed32", tol=1e-10)
    assert abs(info["iters"] - want["iters"]) <= 6, (info["iters"], want["iters"])
    h.free()


@pytest.mark.parametrize("cap", [0, 1, 2, 7, 16, 17])
@pytest.mark.parametrize("mode", ["mixed32", "mixedfx16"])
def test_iteration_cap(cap, mode):
    """A solve stopped after `cap` iterations returns that iterate, whose residual the oracle confirms."""
    dims = (6, 8, 6, 4)
    stag, h, fat, lng = _setup(dims)
    b = synth.gaussian_source(dims, 5102)
    x = torch.zeros((h.Vh, 3), dtype=torch.complex128, device="cuda")
    info = stag.stag_cg(h, x, dev(b), 0.05, mode=mode, tol=1e-12, max_iter=cap, raise_on_error=False)
    assert not info["converged"] and info["iters"] == cap
    res = oracle.true_residual(fat, lng, x.cpu().numpy(), b, 0.05, dims)
    assert abs(res - info["true_rel_resid"]) <= 1e-12 * max(1.0, res)
    h.free()


def test_segments_and_special_sources():
    """A chain of short segments from where the last stopped; a zero and a point source; a finished guess."""
    dims = (6, 6, 4, 10)
    stag, h, fat, lng = _setup(dims, 12)
    b = synth.gaussian_source(dims, 5103)
    x = torch.zeros((h.Vh, 3), dtype=torch.complex128, device="cuda")
    last = np.inf
    for _ in range(6):
        stag.stag_cg(h, x, dev(b), 0.1, mode="mixed32", tol=1e-12, max_iter=9, check_interval=1, use_initial_guess=1,
                     raise_on_error=False)
        res = oracle.true_residual(fat, lng, x.cpu().numpy(), b, 0.1, dims)
        assert res < last
        last = res
    stag.stag_cg(h, x, dev(b), 0.1, mode="mixed32", tol=1e-11, use_initial_guess=1)
    done = stag.stag_cg(h, x, dev(b), 0.1, mode="mixed32", tol=1e-10, use_initial_guess=1)
    assert done["iters"] == 0 and done["converged"]
    zero = stag.stag_cg(h, x, dev(np.zeros_like(b)), 0.1, mode="mixed32")
    assert zero["converged"] and not x.any()
    point = np.zeros_like(b)
    point[17, 1] = 1.0j
    info = stag.stag_cg(h, x, dev(point), 0.1, mode="mixed32", tol=1e-11)
    assert info["converged"] and oracle.true_residual(fat, lng, x.cpu().numpy(), point, 0.1, dims) <= 1.01e-11
    h.free()


@pytest.mark.parametrize("dims", [(16, 16, 16, 16), (16, 16, 16, 18)])
def test_both_sides_of_the_size_rule(dims):
    stag, h, fat, lng = _setup(dims, 12)
    b = synth.gaussian_source(dims, 5104)
    x = torch.zeros((h.Vh, 3), dtype=torch.complex128, device="cuda")
    info = stag.stag_cg(h, x, dev(b), 0.2, mode="mixed32", tol=1e-10)
    assert info["converged"] and oracle.true_residual(fat, lng, x.cpu().numpy(), b, 0.2, dims) <= 1.001e-10
    h.free()


def test_not_finite_source_breaks_down():
    dims = (4, 4, 4, 6)
    stag, h, _, _ = _setup(dims)
    b = synth.gaussian_source(dims, 5105)
    b[3, 0] = np.nan
    x = torch.zeros((h.Vh, 3), dtype=torch.complex128, device="cuda")
    info = stag.stag_cg(h, x, dev(b), 0.1, mode="mixed32", raise_on_error=False)
    want = stag.stag_cg(h, torch.zeros_like(x), dev(b), 0.1, mode="plain64", raise_on_error=False)
    assert info["return"] == want["return"] and info["iters"] == want["iters"]
    h.free()
