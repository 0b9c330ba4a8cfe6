"""The network's tensor-core sums are added with rounding: a gradient, which is a sum over all sites, is then
known better than the values at single sites, whose errors average out."""

import numpy as np
import pytest

import oracle
import oracle.network as onet
import synth
from gpu_common import dev, requires_gpu
from test_gpu_net import _flat_grads, _oracle_params

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("dims,channels", [((8, 8, 8, 8), (1, 16, 16, 1)), ((6, 8, 10, 10), (1, 16, 16, 16, 1))])
@pytest.mark.parametrize("seed", [1, 2])
def test_gradients_have_no_error_in_common(dims, channels, seed):
    """Single values carry some 2e-6 per layer at random (two bfloat16 parts); over thousands of sites and six
    components that leaves well below 1e-6 of the gradient, and below 5e-7 along the gradient itself, where a
    truncated chain of 18 sums per layer (each down by a quarter to a half of 2^-23) would put some 3e-6."""
    import paper_1712_00143_gb300 as stag

    fat, lng = synth.gauge_field(dims, 0.3, 1021)
    h = stag.stag_load_links(dims, dev(fat), dev(lng))
    net = stag.stag_net_create(channels, seed=seed)
    params = _oracle_params(stag.stag_net_get_params(net, rounded=True), channels)
    r, e = synth.random_spinor(dims, 61 + seed), synth.random_spinor(dims, 71 + seed)
    _, g = stag.stag_net_loss_grad(net, h, dev(r), dev(e), loss="residual", mass=0.05)
    _, go = onet.backward_residual(fat, lng, params, r, 0.05, dims, oracle.parity_sites(dims, 0))
    go = _flat_grads(go)
    assert np.linalg.norm(g - go) < 1e-6 * np.linalg.norm(go)
    assert abs(np.dot(g - go, go)) < 5e-7 * np.dot(go, go)
    net.free()
    h.free()
