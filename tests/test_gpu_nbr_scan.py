"""Pair list: candidates numbered 64 at a time through the non-empty cells (or
the molecule's atoms), rows of 8 atoms per block placed by a scan over blocks
and chunks of 32 blocks. Sizes around whole blocks and chunks, dense rows (one
key per lane, two per lane, beyond), empty rows, replicas with their own
cells; the same list again at moved and restored positions, against the FP64
pair oracle (exact).
"""
import numpy as np
import pytest

from oracle import model as M
from paper_2510_06562_gb300 import dmts as D
from paper_2510_06562_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _same(ctx, s, x):
    for which, rc in ((D.SMALL, 3.5), (D.BIG, 5.0)):
        rp, col = ctx.neighbors(which)
        oi, oj = M.pair_list(x, s.atom_offset, s.box, rc)
        np.testing.assert_array_equal(np.repeat(np.arange(s.n_atoms), np.diff(rp)), oi)
        np.testing.assert_array_equal(col, oj)


def _check(s):
    sa, ba = I.small_arch(s.n_species), I.big_arch(s.n_species)
    moved = s.x + 0.2 * np.random.default_rng(1).standard_normal(s.x.shape)
    if s.box[0] > 0:
        moved -= s.box[0] * np.floor(moved / s.box[0])
    with D.Context(s, ba, I.init_params(ba, 3), sa, I.init_params(sa, 2)) as ctx:
        for x in (s.x, moved, s.x):
            ctx.set_state(x)
            _same(ctx, s, x)


def _gas(sizes, spacing, seed=0):
    rng = np.random.default_rng(seed)
    xs = []
    for n in sizes:
        k = int(np.ceil(n ** (1 / 3)))
        g = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n]
        xs.append(spacing * (g + 0.2 * rng.uniform(-1, 1, g.shape)))
    x = np.concatenate(xs)
    return I.System(x=x, species=np.zeros(len(x), np.int32), mass=np.full(len(x), 12.0),
                    atom_offset=np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32), box=np.zeros(len(sizes)),
                    n_species=2, name="gas")


# 255 .. 257 atoms: a chunk of 32 blocks less one row, whole, and one more
@pytest.mark.parametrize("sizes", [(1,), (7,), (8,), (9,), (255, 8), (256, 8), (257, 8), (260, 261), (3,) * 100])
@pytest.mark.parametrize("spacing", [0.9, 1.9, 40.0])
def test_molecules(sizes, spacing):
    _check(_gas(sizes, spacing))


@pytest.mark.parametrize("n_side,stretch", [(4, 1.0), (5, 1.03), (7, 1.0), (11, 1.0)])
def test_periodic(n_side, stretch):
    _check(I.make_water(n_side, 3.105 * n_side * stretch, 3))


def test_replicas():
    _check(I.replicas([I.make_water(5, 15.53, 10 + k) for k in range(3)]))
