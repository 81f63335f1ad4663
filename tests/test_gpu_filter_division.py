"""The FP32 mode's filter takes the ordinary division in SiLU(a) = a / (1 +
exp(-a)). An approximate one (``__fdividef``) is 0 where the divisor is above
2^126, that is for a below -87.4, where the quotient is still a number: a
filter whose activations lie there and whose second matrix is as large as its
values are small would vanish.

Here every activation is -88 (W1 = 0, b1 = -88) and W2 is of the order of
1e36, without the pair repulsion: with a vanishing filter the forces are zero.
Tolerance: ``__expf(88)`` is off by at most 2 + 1.173 x 88 ulp, 1.3e-5, common
to all pairs; through at most two layers, amplified less than tenfold in each,
1.3e-3 of the forces' norm.
"""
import dataclasses

import numpy as np
import pytest

from oracle import model as M
from paper_2510_06562_gb300 import dmts as D
from paper_2510_06562_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _params(arch, seed):
    F, K, S = arch.n_feat, arch.n_radial, arch.n_species
    p = I.init_params(arch, seed).copy()
    layer = F * F + K * F + F + F * F + F + 2 * (F * F + F)
    for l in range(arch.n_layers):
        o = S * F + l * layer + F * F
        p[o:o + K * F] = 0.0                                   # W1
        p[o + K * F:o + K * F + F] = -88.0                     # b1
        o += K * F + F
        p[o:o + F * F] *= 1.0 / 5e-37                          # W2 (SiLU(-88) = -5.3e-37)
    return p


@pytest.mark.parametrize("n_side,arch", [(4, I.small_arch()), (4, I.big_arch()), (7, I.big_arch())],
                         ids=["one_layer", "two_layers", "two_layers_by_species"])
def test_activations_below_the_approximate_division(n_side, arch):
    arch = dataclasses.replace(arch, rep_a=0.0)
    s = I.make_water(n_side, round(3.105 * n_side, 2), 0)
    p = _params(arch, 3)
    _, ref = M.energy_forces(M.spec_of(arch), p, s.x, s.species, s.atom_offset, s.box)
    assert np.sqrt(np.mean(ref ** 2)) > 1e-4                   # the filter does not vanish
    with D.Context(s, arch, p) as ctx:
        ctx.set_state(s.x)
        f = ctx.forces(D.BIG)[1]
    assert np.linalg.norm(f - ref) <= 1.3e-3 * np.linalg.norm(ref)
