"""BF16 mode, layer 0 of more than 4,864 atoms: u of each species from a table
in shared memory (up to eight species), otherwise gathered rows. Both give the
same bits (the same weights in a model of eight species and in one of nine
whose last is unused); against the FP64 oracle within the BF16 bound of the
parity tests (5e-3 eV/A RMSE per unit of RMS force beyond 1), on both sides
of the atom count where the passes change.
"""
import numpy as np
import pytest

from oracle import model as M
from paper_2510_06562_gb300 import dmts as D
from paper_2510_06562_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _system(n, used, n_species, seed=4):
    s = I.make_water(12, 37.26, seed)
    s.x, s.mass = s.x[:n], s.mass[:n]
    s.species = np.random.default_rng(seed).choice(used, n).astype(np.int32)
    s.atom_offset = np.array([0, n], dtype=np.int32)
    s.n_species = n_species
    return s


def _forces(s, sa, sp, ba, bp):
    with D.Context(s, ba, bp, sa, sp, precision=D.BF16_MLP, options='{"autotune": 0}') as ctx:
        ctx.set_state(s.x)
        return [np.concatenate([np.ravel(a) for a in ctx.forces(w, virial=True)]) for w in (D.SMALL, D.BIG)]


def _with_unused(p, F, S):
    return np.concatenate([p[:S * F], np.full(F, 0.3), p[S * F:], [0.7]])


@pytest.mark.parametrize("n", [4865, 5184])
@pytest.mark.parametrize("used", [[0], [0, 1, 2, 3, 4, 5, 6, 7]])
def test_table_and_gathered_rows_agree_bit_for_bit(n, used):
    sa, ba = I.small_arch(8), I.big_arch(8)
    sp, bp = I.init_params(sa, 2), I.init_params(ba, 3)
    got = _forces(_system(n, used, 8), sa, sp, ba, bp)
    sa9, ba9 = I.small_arch(9), I.big_arch(9)
    ref = _forces(_system(n, used, 9), sa9, _with_unused(sp, 32, 8), ba9, _with_unused(bp, 64, 8))
    for a, b in zip(got, ref):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("n", [4864, 4865])
@pytest.mark.parametrize("S", [2, 9])
def test_forces_against_the_oracle(n, S):
    s = _system(n, list(range(S)), S)
    sa, ba = I.small_arch(S), I.big_arch(S)
    sp, bp = I.init_params(sa, 2), I.init_params(ba, 3)
    with D.Context(s, ba, bp, sa, sp, precision=D.BF16_MLP) as ctx:
        ctx.set_state(s.x)
        for which, arch, par in ((D.SMALL, sa, sp), (D.BIG, ba, bp)):
            F = ctx.forces(which)[1]
            Fr = M.energy_forces(M.spec_of(arch), par, s.x, s.species, s.atom_offset, s.box)[1]
            assert np.sqrt(np.mean((F - Fr) ** 2)) <= 5e-3 * max(1.0, np.sqrt(np.mean(Fr ** 2)))
