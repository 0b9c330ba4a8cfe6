"""The preconditioner network on register fragments: every kernel of the forward pass and of the gradient
against the FP64 network oracle, for networks of two to three layers and of one, on lattices whose sites
fill the warps' groups of 32 unevenly, with fewer groups than warps and with more than one per warp."""

import numpy as np
import pytest
import torch

import oracle
import oracle.network as onet
import synth
from gpu_common import dev, rel_l2, requires_gpu
from test_gpu_net import _flat_grads, _oracle_params

pytestmark = [pytest.mark.gpu, requires_gpu]

CASES = [
    ((4, 4, 4, 4), (1, 1), 12),
    ((4, 4, 6, 10), (1, 1), 18),
    ((4, 4, 4, 4), (1, 16, 1), 18),
    ((6, 6, 6, 10), (1, 16, 1), 12),
    ((4, 4, 4, 4), (1, 16, 16, 1), 12),
    ((10, 4, 6, 6), (1, 16, 16, 1), 18),
    ((12, 12, 12, 14), (1, 16, 16, 1), 12),
]


@pytest.mark.parametrize("dims,channels,recon", CASES)
def test_forward_and_gradients(dims, channels, recon):
    """A transport enters the 16 -> 16 products as two bfloat16 parts (error <= 2^-18 of each value, at
    random), the gradients' factors as three (2^-26), all sums are FP32: per layer some 2e-6 forward,
    doubled in the backward pass; 5e-5, 1e-4 and 1e-5 bound the result, its gradient and the loss."""
    import paper_1712_00143_gb300 as stag

    fat, lng = synth.gauge_field(dims, 0.3, 1020)
    h = stag.stag_load_links(dims, dev(fat), dev(lng), recon_long=recon)
    net = stag.stag_net_create(channels, seed=5)
    p = stag.stag_net_get_params(net)
    rng = np.random.default_rng(7)
    off = 0
    for l in range(len(channels) - 1):
        off += 9 * channels[l] * channels[l + 1]
        if l < len(channels) - 2:
            p[off : off + channels[l + 1]] = rng.normal(0.0, 0.5, channels[l + 1])
            off += channels[l + 1]
    stag.stag_net_set_params(net, p)
    params = _oracle_params(stag.stag_net_get_params(net, rounded=True), channels)
    even = oracle.parity_sites(dims, 0)
    r, e = synth.random_spinor(dims, 61), synth.random_spinor(dims, 62)

    z = torch.empty((h.Vh, 3), dtype=torch.complex128, device="cuda")
    stag.stag_net_apply(net, h, z, dev(r))
    zo, _ = onet.forward(fat, params, r, dims, even)
    assert rel_l2(z.cpu().numpy(), zo) < 5e-5

    mass = 0.05
    for kind in ("error", "residual"):
        loss, g = stag.stag_net_loss_grad(net, h, dev(r), dev(e), loss=kind, mass=mass)
        if kind == "error":
            lo, go = onet.backward(fat, params, r, e, dims, even)
        else:
            lo, go = onet.backward_residual(fat, lng, params, r, mass, dims, even)
        go = _flat_grads(go)
        assert abs(loss - lo) < 1e-5 * abs(lo)
        assert np.linalg.norm(g - go) < 1e-4 * np.linalg.norm(go)
    net.free()
    h.free()
