"""Buffers are cleared on the context's stream. That stream does not follow
the default stream, so a clear there (``cudaMemset``, asynchronous to the host)
may run after the kernels that count on it: behind whatever the caller has
queued on the default stream. The source has no such clear, and a context
created, grown and used for distillation while the default stream is busy gives
the results of an idle one, bit for bit."""
import glob
import os
import re

import numpy as np
import pytest

from paper_2510_06562_gb300 import dmts as D
from paper_2510_06562_gb300 import inputs as I

CSRC = os.path.join(os.path.dirname(os.path.abspath(D.__file__)), "csrc")


def test_no_clear_names_the_default_stream():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        assert not re.search(r"\bcudaMemset\s*\(", open(path).read()), path


@pytest.mark.gpu
@pytest.mark.parametrize("frames", [1, 3])
def test_results_do_not_depend_on_the_default_stream(frames):
    import torch
    s = I.water_192(0)
    sa, ba = I.small_arch(), I.big_arch()
    sp, bp = I.init_params(sa, 2), I.init_params(ba, 3)
    g = np.random.default_rng(4)
    x = np.stack([s.x + 0.03 * g.standard_normal(s.x.shape) for _ in range(frames)])
    f, e = g.normal(scale=0.8, size=x.shape), g.normal(scale=5.0, size=frames)

    def results(busy):
        if busy:
            torch.cuda._sleep(200_000_000)           # some 100 ms on the default stream
        # a row capacity below the rows' lengths: the first evaluation grows it
        with D.Context(s, ba, bp, sa, sp, options='{"row_capacity": 16, "autotune": 0}') as ctx:
            ctx.set_state(s.x)
            if busy:
                torch.cuda._sleep(200_000_000)
            out = [*ctx.distill_grad(x, f, e, 0.5)]
            for which in (D.SMALL, D.BIG):
                out += [*ctx.forces(which, virial=True)]
        torch.cuda.synchronize()
        return out

    for a, b in zip(results(False), results(True)):
        np.testing.assert_array_equal(a, b)
