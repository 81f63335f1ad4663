"""Device buffers of the caller that are too small for what a call reads or
writes in place: refused on the host, before any work, as the copy that went
through a staging buffer refused them; a buffer that ends exactly at the end of
its allocation is used. Nothing is written to a refused one."""
import ctypes as C

import numpy as np
import pytest

from paper_2510_06562_gb300 import dmts as D
from paper_2510_06562_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_short_device_buffers_are_refused():
    import torch
    torch.zeros(1, device="cuda")                            # the device's primary context
    cu = C.CDLL("libcuda.so.1")
    s = I.water_192(0)
    ba = I.big_arch()
    lib = D.load_library()
    n = 8 * s.x.size
    slack = 1 << 21                                          # beyond any rounding of an allocation's size
    with D.Context(s, ba, I.init_params(ba, 3)) as ctx:
        ctx.set_state(s.x, np.ones_like(s.x))
        forces = ctx.forces(D.BIG)[1]
        base = C.c_uint64(0)
        assert cu.cuMemAlloc_v2(C.byref(base), C.c_size_t(n + slack)) == 0
        host = np.ascontiguousarray(s.x)
        assert cu.cuMemcpyHtoD_v2(base, host.ctypes.data_as(C.c_void_p), C.c_size_t(n)) == 0

        def at(offset):
            return C.c_void_p(base.value + offset)

        def read(offset):
            out = np.empty_like(s.x)
            assert cu.cuMemcpyDtoH_v2(out.ctypes.data_as(C.c_void_p), C.c_uint64(base.value + offset), C.c_size_t(n)) == 0
            return out

        short = at(slack + n - 8)                            # one double is left of the allocation
        assert lib.dmts_set_state(ctx._h, short, None, s.n_atoms) == -1
        assert lib.dmts_set_state(ctx._h, at(0), short, s.n_atoms) == -1
        assert lib.dmts_get_state(ctx._h, short, None) == -1
        assert lib.dmts_get_state(ctx._h, None, short) == -1
        assert lib.dmts_forces(ctx._h, D.BIG, short, None, None) == -1
        x, v = ctx.get_state()                               # the state is what it was
        np.testing.assert_array_equal(v, np.ones_like(s.x))
        # the last n bytes of the allocation, in place
        assert lib.dmts_forces(ctx._h, D.BIG, at(slack), None, None) == 0
        np.testing.assert_array_equal(read(slack), forces)
        assert lib.dmts_get_state(ctx._h, at(slack), None) == 0
        np.testing.assert_array_equal(read(slack), x)
        assert lib.dmts_set_state(ctx._h, at(0), at(slack), s.n_atoms) == 0
        np.testing.assert_array_equal(ctx.get_state()[1], x)
        assert cu.cuMemFree_v2(base) == 0
