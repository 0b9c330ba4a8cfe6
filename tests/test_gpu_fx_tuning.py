"""Loading FP64 links times the launch shapes there are: four on a large lattice, one on a small one, whose
fixed-point operator runs in a shape of its own."""

import pytest

import synth
from gpu_common import dev, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("dims,shapes", [((4, 4, 4, 4), 1), ((8, 8, 8, 8), 1), ((16, 16, 16, 18), 4)])
def test_launches_of_a_load(dims, shapes):
    import paper_1712_00143_gb300 as stag

    fat, lng = synth.gauge_field(dims, 0.3, 1120)
    fat, lng = dev(fat), dev(lng)
    stag.stag_profile_reset()
    h = stag.stag_load_links(dims, fat, lng, prec_mask=1 << stag.STAG_FP64)
    # per kernel (plain and epilogue) and shape two warm-up and five timed launches, and the remap, the units
    # and the conversion of the links
    assert stag.stag_launch_count() == 2 * shapes * 7 + 3
    block, min_blocks, us = stag.stag_tuned_shape(h, "fp64", 0)
    assert us > 0.0
    h.free()
