"""FP32 mode: filters once per unordered pair (tiles of 128 pairs), gathers by
row (chunks of 32 pairs). Sizes where the tiling can go wrong, against the
FP64 oracle: no pair, one pair, a tile less one, whole and one more, rows of
31 to 33 pairs; radial functions below, at and above the padded counts of 8
and 16; one to three layers; both widths; a row capacity that overflows.

Tolerances: the FP32 bounds of the parity tests (1e-6 eV per atom, 1e-5 eV/A
RMSE) per unit of the largest |E_i| or RMS force beyond 1, since FP32 rounding
scales with the summed magnitudes.
"""
import numpy as np
import pytest

from oracle import model as M
from paper_2510_06562_gb300 import dmts as D
from paper_2510_06562_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _cluster(n, rng, radius, d_min=0.75):
    pts = []
    while len(pts) < n:
        p = rng.uniform(-radius, radius, 3)
        if np.linalg.norm(p) <= radius and all(np.linalg.norm(p - q) >= d_min for q in pts):
            pts.append(p)
    return np.array(pts)


def _system(sizes, seed=0, radius=1.7):
    rng = np.random.default_rng(seed)
    x = np.concatenate([_cluster(n, rng, radius) for n in sizes])
    z = rng.integers(0, 2, len(x)).astype(np.int32)
    return I.System(x=x, species=z, mass=np.where(z == 1, 15.999, 1.008),
                    atom_offset=np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32), box=np.zeros(len(sizes)),
                    n_species=2, name="clusters")


def _check(s, arch, seed=3, options=None):
    p = I.init_params(arch, seed)
    Er, Fr = M.energy_forces(M.spec_of(arch), p, s.x, s.species, s.atom_offset, s.box)
    Wr = M.virial(M.spec_of(arch), p, s.x, s.species, s.atom_offset, s.box)
    with D.Context(s, arch, p, options=options) as ctx:
        ctx.set_state(s.x)
        E, F, W = ctx.forces(D.BIG, virial=True)
        E2, F2 = ctx.forces(D.BIG)
    np.testing.assert_array_equal(E, E2)
    np.testing.assert_array_equal(F, F2)
    rms = float(np.sqrt(np.mean(Fr ** 2)))
    n = np.diff(s.atom_offset)
    assert np.all(np.abs(E - Er) <= 1e-6 * np.maximum(n, np.abs(Er)))
    assert float(np.sqrt(np.mean((F - Fr) ** 2))) <= 1e-5 * max(1.0, rms)
    assert np.abs(W - Wr).max() <= 1e-4 * max(1.0, np.abs(Wr).max())


# all atoms of a cluster lie within 3.4 A of each other: n (n - 1) / 2 unordered pairs
@pytest.mark.parametrize("sizes", [(1,), (2,), (1, 1, 2), (16, 4, 2, 2), (16, 4, 2), (16, 5), (32,), (33,), (34,),
                                   (23, 3), (34, 1, 33, 2)])
def test_tile_and_row_edges(sizes):
    _check(_system(sizes), I.Arch(3.5, 8, 2, 64, 2))


@pytest.mark.parametrize("K,L,F", [(1, 1, 32), (7, 1, 64), (8, 3, 32), (9, 1, 32), (15, 2, 64), (16, 3, 64)])
def test_radial_counts_layers_and_widths(K, L, F):
    _check(_system((20, 7, 12), seed=1), I.Arch(3.5, K, L, F, 2))


def test_row_overflow_is_redone():
    s = I.make_water(4, 12.42, 2)
    arch = I.big_arch()
    p = I.init_params(arch, 3)
    with D.Context(s, arch, p) as a, D.Context(s, arch, p, options='{"row_capacity": 8, "autotune": 0}') as b:
        v = I.maxwell_boltzmann(s.mass, 300.0, 1)
        for ctx in (a, b):
            ctx.set_state(s.x, v)
        np.testing.assert_array_equal(a.respa_step(4, 1.0, 1), b.respa_step(4, 1.0, 1))
        np.testing.assert_array_equal(a.get_state()[0], b.get_state()[0])
