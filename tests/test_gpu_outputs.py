"""Host outputs in every state of their pages: fresh, there already, half and half, and
arrays that begin and end inside a page."""
import ctypes
import mmap

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N = 48  # 16.8 MB of populations, 2.7 MB of velocity


@pytest.mark.parametrize("state", ["fresh", "there", "half"])
@pytest.mark.parametrize("offset", [0, 8, 4096 - 8])
def test_outputs(gpu_lib, state, offset):
    lbm = gpu_lib
    D = ctypes.POINTER(ctypes.c_double)
    with lbm.Lattice(lbm.make_params(N, nu0=0.01, cs=0.1)) as L:
        L.init_random(seed=4)
        L.step(3)
        for want, call in ((L.populations(), lambda p: lbm.load().lbm_get_populations(L.h, 0, p, 1)),
                           (L.fields()["u"], lambda p: lbm.load().lbm_get_velocity(L.h, 0, p))):
            m = mmap.mmap(-1, want.nbytes + 2 * 65536)
            whole = np.frombuffer(m, dtype=np.uint8)
            if state != "fresh":
                whole[:whole.size // (2 if state == "half" else 1)] = 0xAB
            got = whole[offset:offset + want.nbytes].view(np.float64)
            for _ in range(2):  # and once more into the same pages
                assert call(got.ctypes.data_as(D)) == lbm.LBM_OK
                assert np.array_equal(got, want.ravel())
            edge = 0 if state == "fresh" else 0xAB
            assert np.all(whole[:offset] == edge)
            tail = whole[offset + want.nbytes:]
            assert np.all(tail == (0xAB if state == "there" else 0))
