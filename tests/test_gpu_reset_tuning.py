"""After any tuning the library's own choices can be had back: the same launches, the
same work items and the same bits as where nothing was set."""
import numpy as np
import pytest

import kin_inputs as ki

pytestmark = pytest.mark.gpu


def _sim(kin, scheme, N, storage=0):
    sim = kin.Sim(N, scheme, 0.013, 0.1, 1.0 if scheme == kin.LBE_MRT else 0.5, storage)
    sim.set_velocity(ki.random_velocity(N, N, N, 40 + N, 0.03))
    return sim


def _launches(sim, steps):
    before = sim.kernel_launches
    sim.step(steps)
    return sim.kernel_launches - before


@pytest.mark.parametrize("N", [24, 96])
def test_lbe_steps_go_in_pairs_again(kin, N):
    sim, fresh = _sim(kin, kin.LBE_MRT, N), _sim(kin, kin.LBE_MRT, N)
    sim.set_tuning(block_x=128)
    assert _launches(sim, 4) == 4
    sim.reset_tuning()
    assert _launches(sim, 4) == _launches(fresh, 4) == 2
    fresh.step(4)
    np.testing.assert_array_equal(sim.get_f(), fresh.get_f())
    sim.close()
    fresh.close()


def test_dugks_goes_back_to_the_fused_step(kin):
    sim, fresh = _sim(kin, kin.DUGKS, 33), _sim(kin, kin.DUGKS, 33)
    f = sim.get_f()
    sim.set_tuning(tile_y=4, zchunk=3, variant=1)
    assert _launches(sim, 3) == 6
    sim.reset_tuning()
    sim.set_f(f)
    assert _launches(sim, 3) == _launches(fresh, 3) == 3
    np.testing.assert_array_equal(sim.get_f(), fresh.get_f())
    sim.close()
    fresh.close()


@pytest.mark.parametrize("storages", [(0, 0), (1, 1), (0, 2)])
def test_ensemble_goes_back_to_its_defaults(kin, storages):
    sims = [_sim(kin, kin.DUGKS, N, st) for N, st in zip((34, 16), storages)] + [_sim(kin, kin.LBE_MRT, 12)]
    untuned = kin.Ensemble(sims)
    want = untuned.info()
    untuned.close()
    ens = kin.Ensemble(sims)
    ens.set_tuning(8 if storages[0] != storages[1] else 6, 32, 32)
    assert ens.info()["items"] != want["items"]
    ens.step(2)
    ens.reset_tuning()
    got = ens.info()
    assert (got["items"], got["grid"]) == (want["items"], want["grid"])
    ens.step(2)
    ens.close()
    for s in sims:
        s.close()


def test_null_handles_are_rejected(kin):
    assert kin.lib().kin_reset_tuning(None) == kin.KIN_EINVAL
    assert kin.lib().kin_ensemble_reset_tuning(None) == kin.KIN_EINVAL
