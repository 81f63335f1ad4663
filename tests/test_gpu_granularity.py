"""The most CTAs per SM that a model's BF16 edge passes may be given: what the
kernels of its own layers fit, whatever other variants need. For the one-tile
backward pass at F = 32 that is five: 95 or 96 registers of 65,536 / (5 x 128),
40 of 227 KB of shared memory, 64 of 512 tensor-memory columns. Below and above
the size from which layer 0 reads a species table, in a one-layer and in a
two-layer model; forces at five CTAs have the bits of forces at one."""
import dataclasses

import numpy as np
import pytest

from paper_2510_06562_gb300 import dmts as D
from paper_2510_06562_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers", [1, 2])
@pytest.mark.parametrize("n_side", [4, 12])
def test_five_ctas_of_the_one_tile_backward_pass(layers, n_side):
    s = I.make_water(n_side, round(3.105 * n_side, 2), 0)
    arch = dataclasses.replace(I.small_arch(), n_layers=layers)
    with D.Context(s, arch, I.init_params(arch, 2), precision=D.BF16_MLP) as ctx:
        ctx.set_state(s.x)
        forces = {}
        for k in (1, 99):
            ctx.set_tuning(D.BIG, k, k, 1)
            assert ctx.tuning(D.BIG)["atoms_bwd"] == (5 if k == 99 else 1)
            forces[k] = ctx.forces(D.BIG)[1]
    np.testing.assert_array_equal(forces[1], forces[99])
