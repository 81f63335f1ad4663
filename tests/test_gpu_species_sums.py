"""FP32 mode, layer 0 summed by neighbour species before the filter's second
product (models of two layers and more, periodic systems of at least 1,024
atoms, up to four species; others take the general passes): forces, energies
and virial of one to five species, both widths, one to three layers, atom counts that are not multiples
of the 32-atom blocks, species that no atom has, and the distillation
gradient, against the FP64 oracle. Tolerances as in test_gpu_pair_filter.py,
and of test_gpu_distill.py for the gradient.
"""
import numpy as np
import pytest

from oracle import model as M
from paper_2510_06562_gb300 import dmts as D
from paper_2510_06562_gb300 import inputs as I
from test_gpu_pair_filter import _check

pytestmark = pytest.mark.gpu


def _of_species(n, n_species, used, seed):
    """The first n atoms of a 1,029-atom water box, with elements drawn from used."""
    s = I.make_water(7, 21.74, seed)
    s.x, s.mass = s.x[:n], s.mass[:n]
    s.species = np.random.default_rng(seed + 1).choice(used, n).astype(np.int32)
    s.atom_offset = np.array([0, n], dtype=np.int32)
    s.n_species = n_species
    return s


@pytest.mark.parametrize("S,used", [(1, [0]), (2, [1]), (3, [0, 2]), (3, [0, 1, 2]), (4, [0, 1, 2, 3]),
                                    (5, [0, 1, 2, 3, 4])])
@pytest.mark.parametrize("F,L", [(32, 1), (64, 1), (64, 2), (32, 3)])
def test_species_counts(S, used, F, L):
    _check(_of_species(1029, S, used, S), I.Arch(3.5, 8, L, F, S))


@pytest.mark.parametrize("n", [1023, 1024, 1025])
@pytest.mark.parametrize("F", [32, 64])
def test_block_edges(n, F):
    _check(_of_species(n, 3, [0, 1, 2], 5), I.Arch(3.5, 8, 2, F, 3))


@pytest.mark.parametrize("S", [1, 3, 5])
def test_distillation_gradient(S):
    s = _of_species(1029, S, list(range(S)), 7)
    arch = I.Arch(3.5, 8, 1, 32, S)
    p = I.init_params(arch, 2)
    rng = np.random.default_rng(0)
    frames = s.x[None] + 0.02 * rng.standard_normal((2,) + s.x.shape)
    f_ref = 0.5 * rng.standard_normal(frames.shape)
    e_ref = rng.standard_normal(2)
    L_ref, g_ref = M.distill_grad(M.spec_of(arch), p, frames, s.species, s.atom_offset, s.box, f_ref, e_ref, 1.0)
    big = I.Arch(5.0, 16, 2, 64, S)
    with D.Context(s, big, I.init_params(big, 3), arch, p) as ctx:
        L, g = ctx.distill_grad(frames, f_ref, e_ref, 1.0)
    assert abs(L - L_ref) <= 1e-5 * abs(L_ref)
    assert np.abs(g - g_ref).max() <= 1e-5 * np.abs(g_ref).max()
