"""Contexts on a GPU with little free memory: the FP32 mode's stored filter
rows take what the other buffers leave, never the memory those need, and a
distillation call whose batch does not fit runs its frames one at a time and
gives the batch's memory back.

Tolerance: both forms of the filter rows evaluate the same formulas in FP32;
their sums run in other orders (1e-5 of the norm, as one frame at a time
against a batch).
"""
import contextlib

import numpy as np
import pytest

from paper_2510_06562_gb300 import dmts as D
from paper_2510_06562_gb300 import inputs as I

pytestmark = pytest.mark.gpu
MB = 1 << 20


@contextlib.contextmanager
def _free_memory(megabytes):
    """All but so much of the GPU's memory held, in one allocation."""
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    held = torch.empty(torch.cuda.mem_get_info()[0] - megabytes * MB, dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        del held
        torch.cuda.empty_cache()


def _close(a, b):
    assert np.linalg.norm(np.asarray(a) - np.asarray(b)) <= 1e-5 * np.linalg.norm(np.asarray(b))


def _models():
    sa, ba = I.small_arch(), I.big_arch()
    return ba, I.init_params(ba, 3), sa, I.init_params(sa, 2)


def _evaluate(s):
    with D.Context(s, *_models(), options='{"autotune": 0}') as ctx:
        ctx.set_state(s.x)
        return [a for which in (D.SMALL, D.BIG) for a in ctx.forces(which, virial=True)]


@pytest.fixture(scope="module")
def water():
    return I.water_12288(0)


@pytest.fixture(scope="module")
def reference(water):
    return _evaluate(water)


@pytest.mark.parametrize("megabytes", [256, 400, 640])
def test_filter_rows_leave_room_for_the_rest(water, reference, megabytes):
    # the rows of both models take 0.6 GB, everything else 0.15 GB
    with _free_memory(megabytes):
        for a, b in zip(_evaluate(water), reference):
            _close(a, b)


@pytest.mark.parametrize("megabytes", [160, 320, 640])
def test_a_batch_that_does_not_fit(water, megabytes):
    import torch
    g = np.random.default_rng(6)
    x = np.stack([water.x + 0.03 * g.standard_normal(water.x.shape) for _ in range(8)])
    f, e = g.normal(scale=0.8, size=x.shape), g.normal(scale=5.0, size=8)
    with D.Context(water, *_models()) as ctx:
        ctx.set_state(water.x)
        one = [ctx.distill_grad(x[k:k + 1], f[k:k + 1], e[k:k + 1], 0.5) for k in range(8)]
        with _free_memory(megabytes):
            before = torch.cuda.mem_get_info()[0]
            loss, grad = ctx.distill_grad(x, f, e, 0.5)
            # a batch of 98,304 atoms takes 0.6 GB; one frame's buffers 30 MB
            if megabytes < 600:
                assert torch.cuda.mem_get_info()[0] >= before - 48 * MB
        assert abs(loss - np.mean([o[0] for o in one])) <= 1e-6 * loss
        _close(grad, np.mean([o[1] for o in one], axis=0))
        energies = ctx.respa_step(2, 3.0, 3)                    # the context is as usable as before
    assert np.all(np.isfinite(energies))
