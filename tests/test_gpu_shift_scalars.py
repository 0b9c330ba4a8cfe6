"""Multi-shift CG and batched CG with one lane per shift or system in the scalar recurrences: one shift, two,
one less than a warp and a full warp of 32; one to eight systems of which some end long before the others."""

import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_common import dev, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]

DIMS = (4, 4, 6, 8)


def _residual(fat, lng, x, b, mass, shift):
    sites = np.arange(b.shape[0])
    r = b - oracle.apply_m_at_sites(fat, lng, x, mass, DIMS, sites, shift=shift)
    return np.linalg.norm(r) / np.linalg.norm(b)


@pytest.mark.parametrize("nshift", [1, 2, 31, 32])
@pytest.mark.parametrize("mode", ["plain64", "mixed32"])
def test_shifts(nshift, mode):
    """tol 1e-9; the iterated residual leaves the true one by about 2^-53 times the condition number
    (8 / 0.01): far below the 1 % allowed here."""
    import paper_1712_00143_gb300 as stag

    fat, lng = synth.gauge_field(DIMS, 0.3, 1020)
    h = stag.stag_load_links(DIMS, dev(fat), dev(lng), recon_long=18)
    mass, shifts = 0.1, [10.0 ** (-4.0 + 0.125 * k) for k in range(nshift)]
    b = synth.gaussian_source(DIMS, 5200)
    xs = [torch.zeros((h.Vh, 3), dtype=torch.complex128, device="cuda") for _ in shifts]
    infos = stag.stag_multishift_cg(h, xs, dev(b), mass, shifts, mode=mode, tol=1e-9)
    assert all(i["converged"] for i in infos)
    its = [i["iters"] for i in infos]
    assert mode != "plain64" or its == sorted(its, reverse=True)
    for s, x in zip(shifts, xs):
        assert _residual(fat, lng, x.cpu().numpy(), b, mass, s) < 1.01e-9
    h.free()


@pytest.mark.parametrize("n", [1, 2, 3, 5, 8])
@pytest.mark.parametrize("mode", ["plain64", "mixed32"])
def test_batched_systems(n, mode):
    """Sources M^k b (k = 0, 1, ...) have ever less of the small modes and take fewer iterations."""
    import paper_1712_00143_gb300 as stag

    fat, lng = synth.gauge_field(DIMS, 0.3, 1020)
    h = stag.stag_load_links(DIMS, dev(fat), dev(lng), recon_long=18)
    mass = 0.1
    bs, sites = [synth.gaussian_source(DIMS, 5300)], np.arange(h.Vh)
    for _ in range(1, n):
        v = oracle.apply_m_at_sites(fat, lng, bs[-1], mass, DIMS, sites, shift=0.0)
        bs.append(v / np.linalg.norm(v))
    b = torch.stack([dev(v) for v in bs])
    x = torch.zeros_like(b)
    info = stag.stag_batch_solve([(h, x, b, n, mass)], mode=mode, tol=1e-9)
    assert all(i["converged"] for i in info)
    assert all(info[i]["iters"] <= info[0]["iters"] for i in range(n))
    for i in range(n):
        assert _residual(fat, lng, x[i].cpu().numpy(), bs[i], mass, 0.0) < 1.01e-9
    h.free()
