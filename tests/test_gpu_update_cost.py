"""A parameter update writes the embeddings of all atoms and of each species
with one kernel, and the evaluations that read either see the new weights."""
import numpy as np
import pytest

from paper_2510_06562_gb300 import dmts as D
from paper_2510_06562_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [D.FP32, D.BF16_MLP])
@pytest.mark.parametrize("n_side", [4, 12])
def test_one_launch_per_update(prec, n_side):
    # 192 atoms: u^0 per atom; 5,184 atoms: sums by species (FP32), the species table (BF16)
    s = I.make_water(n_side, round(3.105 * n_side, 2), 0)
    ba = I.big_arch()
    p = I.init_params(ba, 3)
    g = np.random.default_rng(2).normal(size=p.size)
    with D.Context(s, ba, p, precision=prec) as ctx:
        ctx.set_state(s.x)
        ctx.forces(D.BIG)
        n = ctx.launch_count
        ctx.adam_step(D.BIG, g, np.zeros_like(p), np.zeros_like(p), 1, 1e-2)
        assert ctx.launch_count - n == 1
        got = ctx.forces(D.BIG)
        new = ctx.get_params(D.BIG)
    with D.Context(s, ba, new, precision=prec) as ctx:
        ctx.set_state(s.x)
        ref = ctx.forces(D.BIG)
    for a, b in zip(got, ref):
        np.testing.assert_array_equal(a, b)
