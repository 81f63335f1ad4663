"""Distillation on the context's stream: a caller that fills the frames, the
reference forces and the energies with work queued on that stream, and has
not waited for it, gets the gradient of what that work writes, from one frame
a call and from a batch. The call's arithmetic is the same either way, so its
results are the same bits."""
import numpy as np
import pytest

from paper_2510_06562_gb300 import dmts as D
from paper_2510_06562_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 3])
def test_frames_written_on_the_contexts_stream(m):
    import torch
    s = I.water_192(0)
    sa, ba = I.small_arch(), I.big_arch()
    g = np.random.default_rng(3)
    data = (np.stack([s.x + 0.03 * g.standard_normal(s.x.shape) for _ in range(m)]),
            g.normal(scale=0.8, size=(m,) + s.x.shape), g.normal(scale=5.0, size=m))
    with D.Context(s, ba, I.init_params(ba, 3), sa, I.init_params(sa, 2)) as ctx:
        ctx.set_state(s.x)
        ref = ctx.distill_grad(*data, 0.5)
        src = [torch.as_tensor(a, device="cuda") for a in data]
        dst = [torch.as_tensor(a, device="cuda") for a in (np.broadcast_to(s.x, data[0].shape).copy(),
                                                           np.zeros_like(data[1]), np.zeros_like(data[2]))]
        torch.cuda.synchronize()
        with torch.cuda.stream(torch.cuda.ExternalStream(ctx.stream)):
            torch.cuda._sleep(100_000_000)           # some 50 ms
            for a, b in zip(dst, src):
                a.copy_(b)
        got = ctx.distill_grad(*dst, 0.5)
    assert got[0] == ref[0]
    np.testing.assert_array_equal(got[1], ref[1])
