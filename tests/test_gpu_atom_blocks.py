"""Per-atom kernels at the atom counts where their blocks change: part of a
block of 8, whole, one more; the most atoms in blocks of 8 and of 16 (at F = 32
and 64) and one more; both models and both precisions against the FP64 oracle.
Tolerances: those of the parity tests (1e-6 eV per atom and 1e-5 eV/A RMSE in
FP32, 5e-3 eV per atom and eV/A in BF16) per unit of the largest |E| per atom
or RMS force beyond 1.
"""
import numpy as np
import pytest

from oracle import model as M
from paper_2510_06562_gb300 import dmts as D
from paper_2510_06562_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol_e,tol_f", [(D.FP32, 1e-6, 1e-5), (D.BF16_MLP, 5e-3, 5e-3)])
@pytest.mark.parametrize("n", [3, 8, 9, 1215, 1216, 1217, 1824, 1825, 2432, 2433])
def test_block_sizes(n, prec, tol_e, tol_f):
    s = I.make_water(10, 31.05, n)
    s.x, s.mass, s.species = s.x[:n], s.mass[:n], s.species[:n]
    s.atom_offset = np.array([0, n], dtype=np.int32)
    sa, ba = I.small_arch(2), I.big_arch(2)
    sp, bp = I.init_params(sa, 2), I.init_params(ba, 3)
    with D.Context(s, ba, bp, sa, sp, precision=prec) as ctx:
        ctx.set_state(s.x)
        for which, arch, par in ((D.SMALL, sa, sp), (D.BIG, ba, bp)):
            E, F, W = ctx.forces(which, virial=True)
            Er, Fr = M.energy_forces(M.spec_of(arch), par, s.x, s.species, s.atom_offset, s.box)
            Wr = M.virial(M.spec_of(arch), par, s.x, s.species, s.atom_offset, s.box)
            assert abs(E[0] - Er[0]) <= tol_e * max(n, abs(Er[0]))
            assert np.sqrt(np.mean((F - Fr) ** 2)) <= tol_f * max(1.0, np.sqrt(np.mean(Fr ** 2)))
            assert np.abs(W - Wr).max() <= 10 * tol_f * max(1.0, np.abs(Wr).max())
