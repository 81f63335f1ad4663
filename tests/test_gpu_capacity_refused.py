"""Neighbour rows beyond what the kernels hold (6,591 atoms at one point) are an
error that leaves the context as usable as before: the capacities are what they
were, a captured step has no stale buffers, candidate rows that the overflow
truncated are built again, and a distillation call puts the state back. A later
evaluation, step or gradient gives the bits of a context that never failed."""
import json

import numpy as np
import pytest

from paper_2510_06562_gb300 import dmts as D
from paper_2510_06562_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("skin", [0.0, 1.0])
@pytest.mark.parametrize("prec", [D.FP32, D.BF16_MLP])
def test_the_context_stays_usable(prec, skin):
    s = I.make_water(13, round(3.105 * 13, 2), 0)
    assert s.n_atoms > 6000
    sa, ba = I.small_arch(), I.big_arch()
    v = I.maxwell_boltzmann(s.mass, 300.0, 1)
    g = np.random.default_rng(3)
    frame = s.x[None] + 0.03 * g.standard_normal((1,) + s.x.shape)
    labels = g.normal(size=frame.shape), g.normal(size=1)
    one_point = np.full_like(s.x, 7.0)

    def run(fails):
        opts = json.dumps({"skin": skin, "autotune": 0})
        with D.Context(s, ba, I.init_params(ba, 3), sa, I.init_params(sa, 2), precision=prec, options=opts) as ctx:
            ctx.set_state(s.x, v)
            ctx.respa_step(1, 2.0, 2)                          # a captured step
            if fails:
                for call in (lambda: ctx.forces(D.BIG), lambda: ctx.neighbors(D.SMALL),
                             lambda: ctx.respa_step(1, 2.0, 2)):
                    ctx.set_state(one_point, v)
                    with pytest.raises(D.DmtsError) as e:
                        call()
                    assert e.value.code == -4
            ctx.set_state(s.x, v)
            out = [*ctx.forces(D.SMALL), *ctx.forces(D.BIG)]
            if fails:
                with pytest.raises(D.DmtsError) as e:
                    ctx.distill_grad(one_point[None], *labels, 1.0)
                assert e.value.code == -4
            out += [ctx.respa_step(2, 2.0, 2), *ctx.get_state()]
            return out + [np.asarray(a) for a in ctx.distill_grad(frame, *labels, 1.0)]

    for a, b in zip(run(True), run(False)):
        np.testing.assert_array_equal(a, b)
