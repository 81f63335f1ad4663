"""Distillation gradients over batches of frames: a call over M frames runs
them as the systems of one batch (several batches, the last one shorter, when
M frames exceed the batch size), and equals the mean of M one-frame calls, also
after the weights changed; the state is left as it was.

Tolerance (FP32): the two differ in the order of FP32 sums of up to 1e5 terms
per gradient entry, 1e-5 of the gradient's norm at most. In the BF16 mode
another order can also round a single operand the other way (2^-8 of one of a
frame's few thousand features), so a batch is compared with the FP64 oracle at
that mode's bounds (2e-2 of the norm, 5e-3 of the loss).
"""
import numpy as np
import pytest

from oracle import model as M
from paper_2510_06562_gb300 import dmts as D
from paper_2510_06562_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _frames(s, m, seed=5):
    g = np.random.default_rng(seed)
    x = np.stack([s.x + 0.03 * g.standard_normal(s.x.shape) for _ in range(m)])
    return x, g.normal(scale=0.8, size=x.shape), g.normal(scale=5.0, size=m)


def _same(got, ref):
    assert abs(got[0] - ref[0]) <= 1e-6 * abs(ref[0])
    assert np.linalg.norm(got[1] - ref[1]) <= 1e-5 * np.linalg.norm(ref[1])


@pytest.mark.parametrize("system,m", [("water", 2), ("water", 3), ("water", 701), ("vacuum", 5), ("replicas", 4)])
def test_a_batch_is_the_mean_of_its_frames(system, m):
    s = {"water": I.water_192, "vacuum": lambda k: I.make_vacuum_batch(3, 10, 60, k),
         "replicas": lambda k: I.replicas([I.water_192(k), I.water_192(k + 1)])}[system](0)
    sa, ba = I.small_arch(s.n_species), I.big_arch(s.n_species)
    sp, bp = I.init_params(sa, 2), I.init_params(ba, 3)
    x, f, e = _frames(s, m)
    v = I.maxwell_boltzmann(s.mass, 300.0, 1, s.atom_offset)
    with D.Context(s, ba, bp, sa, sp) as ctx:
        ctx.set_state(s.x, v)
        before = ctx.get_state()
        for params in (sp, I.init_params(sa, 9)):
            ctx.set_params(D.SMALL, params)
            got = ctx.distill_grad(x, f, e, 0.5)
            one = [ctx.distill_grad(x[k:k + 1], f[k:k + 1], e[k:k + 1], 0.5) for k in range(m)]
            _same(got, (np.mean([o[0] for o in one]), np.mean([o[1] for o in one], axis=0)))
            got = ctx.force_matching_grad(x, f)
            one = [ctx.force_matching_grad(x[k:k + 1], f[k:k + 1]) for k in range(min(m, 5))]
            if m <= 5:
                _same(got, (np.mean([o[0] for o in one]), np.mean([o[1] for o in one], axis=0)))
        after = ctx.get_state()
    for a, b in zip(before, after):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("m", [2, 3])
def test_a_bf16_batch_matches_the_oracle(m):
    s = I.water_192(0)
    sa, ba = I.small_arch(), I.big_arch()
    sp, bp = I.init_params(sa, 2), I.init_params(ba, 3)
    x, f, e = _frames(s, m)
    L, g = M.distill_grad(M.spec_of(sa), sp, x, s.species, s.atom_offset, s.box, f, e, 0.5)
    with D.Context(s, ba, bp, sa, sp, precision=D.BF16_MLP) as ctx:
        ctx.set_state(s.x)
        got = ctx.distill_grad(x, f, e, 0.5)
    assert abs(got[0] - L) <= 5e-3 * L
    assert np.linalg.norm(got[1] - g) <= 2e-2 * np.linalg.norm(g)
