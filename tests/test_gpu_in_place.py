"""Device buffers of the caller: on an 8-byte boundary the kernels read and
write them in place, at any other address they go through the staging copy;
either gives the bits of host buffers."""
import ctypes as C

import numpy as np
import pytest

from paper_2510_06562_gb300 import dmts as D
from paper_2510_06562_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [0, 4, 8])
def test_device_buffers_at_any_address(shift):
    import torch
    s = I.water_192(0)
    ba = I.big_arch()
    v = I.maxwell_boltzmann(s.mass, 300.0, 1)
    nb = 8 * s.x.size
    lib = D.load_library()

    def buf(a=None):
        t = torch.zeros(nb + 16, dtype=torch.uint8, device="cuda")
        if a is not None:
            t[shift:shift + nb] = torch.from_numpy(np.ascontiguousarray(a).view(np.uint8).reshape(-1)).cuda()
        torch.cuda.synchronize()
        return t

    def at(t):
        return C.c_void_p(t.data_ptr() + shift)

    def host(t):
        return t[shift:shift + nb].cpu().numpy().copy().view(np.float64).reshape(s.x.shape)

    with D.Context(s, ba, I.init_params(ba, 3)) as ref, D.Context(s, ba, I.init_params(ba, 3)) as ctx:
        ref.set_state(s.x, v)
        x_in, v_in, x_out, v_out, f_out = buf(s.x), buf(v), buf(), buf(), buf()
        assert lib.dmts_set_state(ctx._h, at(x_in), at(v_in), s.n_atoms) == 0
        assert lib.dmts_get_state(ctx._h, at(x_out), at(v_out)) == 0
        assert lib.dmts_forces(ctx._h, D.BIG, at(f_out), None, None) == 0
        x, vv = ref.get_state()
        np.testing.assert_array_equal(host(x_out), x)
        np.testing.assert_array_equal(host(v_out), vv)
        np.testing.assert_array_equal(host(f_out), ref.forces(D.BIG)[1])
