"""Ensembles by the storage types of their DUGKS members (a kernel for each of FP32,
FP16 and BF16 and one for mixtures), as the library shapes them and with every tile
height: each member is bitwise its solo kin_step run."""
import numpy as np
import pytest

import kin_inputs as ki

pytestmark = pytest.mark.gpu

F32, F16, BF16 = 0, 1, 2
MIXES = {
    "f32": [("dugks", 33, F32), ("dugks", 12, F32), ("lbe", 9, F32)],
    "f16": [("dugks", 34, F16), ("dugks", 10, F16), ("lbe", 12, F16)],
    "bf16": [("dugks", 34, BF16), ("dugks", 4, BF16)],
    "f16 and bf16": [("dugks", 18, F16), ("dugks", 32, BF16)],
    "all": [("dugks", 33, F32), ("dugks", 34, F16), ("dugks", 14, BF16), ("lbe", 18, BF16), ("lbe", 9, F32)],
}


@pytest.mark.parametrize("tuning", [(0, 0), (4, 0), (4, 5), (6, 3), (8, 0), (8, 7)])
@pytest.mark.parametrize("mix", MIXES)
def test_members_are_bitwise_their_solo_runs(kin, mix, tuning):
    members, solo = [], []
    for k, (scheme, N, storage) in enumerate(MIXES[mix]):
        u = ki.random_velocity(N, N, N, 700 + k, 0.03)
        for group in (members, solo):
            sim = kin.Sim(N, kin.LBE_MRT if scheme == "lbe" else kin.DUGKS, 0.012 + 0.001 * k, 0.1,
                          1.0 if scheme == "lbe" else 0.45, storage)
            sim.set_velocity(u)
            group.append(sim)
    ens = kin.Ensemble(members)
    if any(tuning):
        ens.set_tuning(*tuning)
    ens.step(2)
    ens.step(3)
    for a, b in zip(members, solo):
        b.step(5)
        a.check_guards()
        np.testing.assert_array_equal(a.get_f(), b.get_f())
    ens.close()
    for s in members + solo:
        s.close()
