"""Read-outs large enough for their pages to be touched by several threads
(32 MB and more): the values are those of kin_sample_f, in fresh, reused and
unaligned result arrays, and nothing beyond the array is written."""
import ctypes

import numpy as np
import pytest

import kin_inputs as ki

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,storage", [(64, 0), (65, 3)])
def test_large_readouts(N, storage):
    import paper_1601_03815_gb300 as kin

    kin.load()
    sim = kin.Sim(N, kin.LBE_MRT, 0.013, 0.1, 1.0, storage)
    sim.set_velocity(ki.random_velocity(N, N, N, 8, 0.03))
    sim.step(1)
    cells = np.random.default_rng(3).integers(0, N ** 3, 20000)
    want = sim.sample_f(cells)
    fresh = sim.get_f()
    np.testing.assert_array_equal(fresh.reshape(19, -1)[:, cells].T, want)
    raw = np.full(19 * N ** 3 * 8 + 24, 7, np.uint8)  # resident, offset by 8 bytes
    for _ in range(2):
        view = raw[8:-16].view(np.float64)
        view[:] = -1.0
        kin._check(kin.lib().kin_get_f(sim.handle, view.ctypes.data_as(ctypes.c_void_p)), "kin_get_f")
        np.testing.assert_array_equal(view, fresh.reshape(-1))
        assert (raw[:8] == 7).all() and (raw[-16:] == 7).all()
    sim.close()


def test_large_velocity():
    import paper_1601_03815_gb300 as kin

    kin.load()
    N = 116  # 37 MB
    u = ki.random_velocity(N, N, N, 9, 0.03)
    sim = kin.Sim(N, kin.DUGKS, 0.013, 0.1, 0.5, kin.F64)
    sim.set_velocity(u)
    np.testing.assert_allclose(sim.get_velocity(), u, rtol=0, atol=1e-15)
    sim.close()
