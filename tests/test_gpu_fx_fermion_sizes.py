"""The fermion force of fields whose sites differ by many orders of magnitude, link by link: each link's error
is bounded by the sizes of the terms that enter it with their coefficients, so that a part with a small or
zero coefficient (the Naik products at c3 = 0, say) costs the others nothing, however large it is."""

import numpy as np
import pytest

import oracle.fermion_force as ff
import synth
from gpu_common import requires_gpu
from oracle.staggered import lex_of, site_coords
from test_gpu_fx_fermion_force import _force

pytestmark = [pytest.mark.gpu, requires_gpu]

DIMS = (6, 4, 6, 8)


def _sizes(xs, ys, alphas, coef):
    """Per link, the sum of |coefficient| x norm over its 1 + 18 + 3 outer products, all terms' norms added."""
    c = site_coords(DIMS, np.arange(np.prod(DIMS)))
    nf, nl = np.zeros((len(c), 4)), np.zeros((len(c), 4))
    for x, y, a in zip(xs, ys, alphas):
        gf, gl = ff.outer_products([x], [y], [a], DIMS)
        nf += np.sqrt((np.abs(gf) ** 2).sum((2, 3)))
        nl += np.sqrt((np.abs(gl) ** 2).sum((2, 3)))

    def at(*steps):
        q = c.copy()
        for mu, k in steps:
            q[:, mu] = (q[:, mu] + k) % DIMS[mu]
        return lex_of(DIMS, q)

    out = np.zeros((len(c), 4))
    for r in range(4):
        out[:, r] += abs(coef[0]) * nf[at(), r]
        for n in range(4):
            if n != r:
                for pn, q, far in ((at((n, 1)), at(), at((r, 1))), (at((n, -1)), at((n, -1)), at((r, 1), (n, -1)))):
                    out[:, r] += abs(coef[1]) * (nf[pn, r] + nf[q, n] + nf[far, n])
        out[:, r] += abs(coef[2]) * (nl[at(), r] + nl[at((r, -1)), r] + nl[at((r, -2)), r])
    return out


@pytest.mark.parametrize("coef", [(1.0, 0.125, -1.0 / 24.0), (1.0, 0.0, 0.0), (0.0, 1.0, 0.0), (0.0, 0.0, 1.0),
                                  (1.0, 1e-12, 0.0), (1e-14, 0.0, 1.0), (1.0, 1e-9, 1e-13)])
@pytest.mark.parametrize("decades", [0, 3, 9])
def test_every_link_by_its_own_terms(coef, decades):
    thin = synth.gauge_field(DIMS, 0.3, 1096, return_thin=True)[2]
    rng = np.random.default_rng(decades)
    xs = np.stack([synth.random_spinor(DIMS, 95 + i) for i in range(2)])
    ys = np.stack([synth.random_spinor(DIMS, 195 + i) for i in range(2)])
    xs *= 10.0 ** rng.uniform(-decades, decades, size=(1, xs.shape[1], 1))
    ys *= 10.0 ** rng.uniform(-decades, decades, size=(1, ys.shape[1], 1))
    alphas = [1.0, -0.5]
    got = _force(DIMS, thin, xs, ys, alphas, coef)
    want = ff.fermion_force(thin, list(xs), list(ys), alphas, DIMS, *coef)
    # FP64 is off by at most some 6 * 5 * 2^-53 = 3.4e-15 of these sizes, and so may the reference be
    err = np.abs(got - want).max(axis=(2, 3))
    assert (err <= 2 * 3.4e-15 * _sizes(xs, ys, alphas, coef)).all()
