"""The bounds-checked build against the ordinary one where its paths differ or
its indices are of another kind: forces and virials of both models, in the FP32
mode with the filter rows chunked by atoms (the checked build's limit of 16 MB
makes it so for the two-layer model from 1,029 atoms of water and for the
one-layer model at 12,288; the ordinary build keeps all rows), and distillation
batches, whole and with a last batch of fewer frames. Every call must succeed
without an index outside its array.

Tolerances: FP32, other orders of FP32 sums, 1e-5 of an array's norm (1e-6 of
a loss). BF16 mode: the same kernels, but one operand rounded the other way
would already be 2^-9 of a feature: that mode's bounds against the oracle, 5e-3
of forces, virials and losses and 2e-2 of gradients."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2510_06562_gb300 import build as B

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys
import numpy as np
sys.path.insert(0, ROOT)
from paper_2510_06562_gb300 import dmts as D, inputs as I
out = {}
systems = {"vacuum64": I.make_vacuum_batch(64, 10, 60, seed=0), "water192": I.water_192(0),
           "water1029": I.make_water(7, 21.735, 0), "water12288": I.water_12288(0),
           "replicas3": I.replicas([I.water_192(k) for k in range(3)])}
frames = {"vacuum64": 3, "water192": 5, "water1029": 129, "replicas3": 4}
for name, s in systems.items():
    sa, ba = I.small_arch(s.n_species), I.big_arch(s.n_species)
    for prec in (D.FP32, D.BF16_MLP):
        with D.Context(s, ba, I.init_params(ba, 3), sa, I.init_params(sa, 2), precision=prec) as ctx:
            ctx.set_state(s.x)
            for which in (D.SMALL, D.BIG):
                for key, a in zip(("energy", "forces", "virial"), ctx.forces(which, virial=True)):
                    out[f"{name}/{prec}/{which}/{key}"] = a
            if name in frames:
                g, m = np.random.default_rng(9), frames[name]
                x = np.stack([s.x + 0.03 * g.standard_normal(s.x.shape) for _ in range(m)])
                loss, grad = ctx.distill_grad(x, g.normal(scale=0.8, size=x.shape), g.normal(scale=5.0, size=m), 0.5)
                out[f"{name}/{prec}/0/loss"], out[f"{name}/{prec}/0/grad"] = np.array([loss]), grad
np.savez(sys.argv[1], **out)
"""


def _run(lib, path):
    r = subprocess.run([sys.executable, "-c", CHILD.replace("ROOT", repr(ROOT)), path], capture_output=True, text=True,
                       env=dict(os.environ, DMTS_LIBRARY=lib), timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    return np.load(path)


def test_the_checked_build_gives_the_ordinary_results(tmp_path):
    got = _run(B.build(check=True), str(tmp_path / "check.npz"))
    ref = _run(B.build(), str(tmp_path / "plain.npz"))
    assert sorted(got.files) == sorted(ref.files)
    for key in ref.files:
        _, prec, _, kind = key.split("/")
        bound = {"loss": 1e-6}.get(kind, 1e-5) if prec == "0" else {"grad": 2e-2}.get(kind, 5e-3)
        assert np.linalg.norm(got[key] - ref[key]) <= bound * np.linalg.norm(ref[key]), key
