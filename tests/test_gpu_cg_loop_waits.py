"""The small-lattice CG kernel when a grid barrier's wait runs out (a bounded wait that nothing satisfies; no
fault, no hang): every block leaves, and the solve is done with queued launches instead."""

import pytest
import torch

import oracle
import synth
from gpu_common import dev, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (8, 8, 8, 8), (8, 12, 10, 14)])
@pytest.mark.parametrize("mode", ["mixed32", "mixedfx16"])
def test_a_wait_that_gives_up_costs_the_solve_nothing(dims, mode):
    import paper_1712_00143_gb300 as stag

    fat, lng = synth.gauge_field(dims, 0.3, 1111)
    h = stag.stag_load_links(dims, dev(fat), dev(lng))
    b = synth.gaussian_source(dims, 5200)
    runs = []
    for polls, what in ((0, 0), (300, 1), (300, 1), (0, 0)):
        stag.stag_cg_loop_test(h, polls, what)
        x = torch.zeros((h.Vh, 3), dtype=torch.complex128, device="cuda")
        info = stag.stag_cg(h, x, dev(b), 0.2, mode=mode, tol=1e-10)
        assert info["return"] == stag.STAG_OK and info["converged"]
        assert oracle.true_residual(fat, lng, x.cpu().numpy(), b, 0.2, dims) <= 1.001e-10
        runs.append((x, info["iters"]))
    assert torch.equal(runs[1][0], runs[2][0]) and runs[1][1] == runs[2][1]  # queued launches, both times
    assert torch.equal(runs[0][0], runs[3][0]) and runs[0][1] == runs[3][1]  # the loop kernel, before and after
    h.free()


def test_an_initial_guess_survives():
    import paper_1712_00143_gb300 as stag

    dims = (6, 6, 8, 4)
    fat, lng = synth.gauge_field(dims, 0.3, 1112)
    h = stag.stag_load_links(dims, dev(fat), dev(lng))
    b = synth.gaussian_source(dims, 5201)
    x = torch.zeros((h.Vh, 3), dtype=torch.complex128, device="cuda")
    stag.stag_cg(h, x, dev(b), 0.1, mode="mixed32", tol=1e-6)
    stag.stag_cg_loop_test(h, 300, 1)
    info = stag.stag_cg(h, x, dev(b), 0.1, mode="mixed32", tol=1e-11, use_initial_guess=1)
    assert info["converged"] and oracle.true_residual(fat, lng, x.cpu().numpy(), b, 0.1, dims) <= 1.01e-11
    h.free()


@pytest.mark.parametrize("mode", ["mixed32", "mixedfx16"])
def test_without_scratch_the_launches_are_queued(mode):
    import paper_1712_00143_gb300 as stag

    dims = (6, 6, 8, 4)
    fat, lng = synth.gauge_field(dims, 0.3, 1113)
    h = stag.stag_load_links(dims, dev(fat), dev(lng))
    b = synth.gaussian_source(dims, 5202)
    runs = []
    for polls, what in ((300, 1), (0, 2), (0, 0), (0, 2)):
        stag.stag_cg_loop_test(h, polls, what)
        x = torch.zeros((h.Vh, 3), dtype=torch.complex128, device="cuda")
        info = stag.stag_cg(h, x, dev(b), 0.2, mode=mode, tol=1e-10)
        assert info["converged"] and oracle.true_residual(fat, lng, x.cpu().numpy(), b, 0.2, dims) <= 1.001e-10
        runs.append(x)
    assert torch.equal(runs[0], runs[1]) and torch.equal(runs[1], runs[3])
    h.free()
