"""The DUGKS step that holds whole periodic rows in a warp (N = 31 and 32, at 31 with an
idle lane) against the FP64 oracle, beside the sizes next to them, which take tiles of
30 columns.  The state is random in every population, so a wrong periodic neighbour
shows at once.  Bounds: the one-step parity tolerances of the storage types."""
import numpy as np
import pytest

import kin_inputs as ki

pytestmark = pytest.mark.gpu

TOL = {3: 1e-12, 0: 1e-5}  # keyed by storage code


@pytest.mark.parametrize("zchunk", [0, 5])
@pytest.mark.parametrize("storage", [3, 0])
@pytest.mark.parametrize("N", [30, 31, 32, 33])
def test_whole_rows_match_the_oracle(kin, orc, N, storage, zchunk):
    u = ki.random_velocity(N, N, N, 310 + N, 0.03)
    sim = kin.Sim(N, kin.DUGKS, 0.013, 0.1, 0.5, storage)
    if zchunk:
        sim.set_tuning(zchunk=zchunk)
    sim.set_f(orc.equilibrium_field(u) + ki.random_populations(N, N, N, 311 + N, 2e-5))
    f = sim.get_f()
    sim.step(1)
    got, ref = sim.get_f(), orc.step("dugks", f, 0.013, 0.5)
    scale = np.abs(ref).reshape(19, -1).max(axis=1)
    assert (np.abs(got - ref).reshape(19, -1).max(axis=1) / scale).max() < TOL[storage]
    sim.check_guards()
    sim.close()
