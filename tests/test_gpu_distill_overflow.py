"""A neighbour overflow inside a batch of distillation frames: the capacity
options of the context are those of its batches too, so small ones make the
first call grow rows, pairs or cells and run again, for whole batches and with
a last batch of fewer frames. A later call on the grown capacities gives the
same bits, and both equal the mean of one frame at a time (tolerance: the order
of FP32 sums, 1e-5 of the gradient's norm and 1e-6 of the loss, as for any
batch)."""
import numpy as np
import pytest

from paper_2510_06562_gb300 import dmts as D
from paper_2510_06562_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_side,frames", [(4, 3), (7, 129)], ids=["one_batch", "a_shorter_last_batch"])
@pytest.mark.parametrize("options", ['{"row_capacity": 4}', '{"edge_capacity_factor": 0.05}', '{"cell_capacity": 2}',
                                     '{"row_capacity": 4, "edge_capacity_factor": 0.05, "cell_capacity": 2}'])
def test_capacities_grow_inside_a_batch(n_side, frames, options):
    s = I.make_water(n_side, round(3.105 * n_side, 2), 0)
    sa, ba = I.small_arch(), I.big_arch()
    sp, bp = I.init_params(sa, 2), I.init_params(ba, 3)
    g = np.random.default_rng(7)
    x = np.stack([s.x + 0.03 * g.standard_normal(s.x.shape) for _ in range(frames)])
    f, e = g.normal(scale=0.8, size=x.shape), g.normal(scale=5.0, size=frames)
    with D.Context(s, ba, bp, sa, sp) as ref:
        ref.set_state(s.x)
        one = [ref.distill_grad(x[k:k + 1], f[k:k + 1], e[k:k + 1], 0.5) for k in range(frames)]
    loss, grad = np.mean([o[0] for o in one]), np.mean([o[1] for o in one], axis=0)
    with D.Context(s, ba, bp, sa, sp, options=options) as ctx:
        ctx.set_state(s.x)
        first, again = ctx.distill_grad(x, f, e, 0.5), ctx.distill_grad(x, f, e, 0.5)
    assert first[0] == again[0]
    np.testing.assert_array_equal(first[1], again[1])
    assert abs(first[0] - loss) <= 1e-6 * abs(loss)
    assert np.linalg.norm(first[1] - grad) <= 1e-5 * np.linalg.norm(grad)
