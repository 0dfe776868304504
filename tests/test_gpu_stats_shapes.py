"""E and eps of every storage, layout and box remainder against the stored
populations.

The statistics kernels have a vector form (N a multiple of 4), two-byte vector
gathers for both layouts, and a reduction whose last block forms the total, so
boxes below, at and above those limits are compared with the FP64 sums over
kin_get_f (which returns the stored values exactly).

Tolerance: FP64 storage 1e-12.  Otherwise a velocity component is ten stored
values added in FP32, an error of at most 10 * 2^-24 of their absolute sum,
which is at most ~3 times the velocity here: 2e-6; E doubles it, a squared
difference of two velocities quadruples it, and the FP32 products and sums of
up to 32 cells add 2e-6: 2e-5 covers both.
"""
import numpy as np
import pytest

import kin_inputs as ki

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kin():
    import paper_1601_03815_gb300 as k

    k.load()
    return k


def _reference(kin, sim):
    xi, _ = kin.lattice()
    u = np.einsum("ic,izyx->czyx", xi.astype(float), sim.get_f())
    g = [[(np.roll(u[b], -1, 2 - a) - np.roll(u[b], 1, 2 - a)) / 2 for b in range(3)] for a in range(3)]
    ss = sum(((g[a][b] + g[b][a]) / 2) ** 2 for a in range(3) for b in range(3))
    return 0.5 * np.mean((u * u).sum(0)), 2 * sim.nu * np.mean(ss)


@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("storage", [0, 1, 2, 3])
@pytest.mark.parametrize("N", [2, 4, 5, 6, 12, 33, 36, 68])
def test_energy_and_dissipation(kin, N, storage, scheme):
    sim = kin.Sim(N, scheme, 0.013, 0.1, 1.0 if scheme == kin.LBE_MRT else 0.5, storage)
    sim.set_velocity(ki.random_velocity(N, N, N, 300 + N, 0.03))
    sim.step(1)
    tol = 1e-12 if storage == 3 else 2e-5
    for _ in range(2):  # the counter of the reduction is ready for the next call
        got = sim.stats()
        np.testing.assert_allclose(got, _reference(kin, sim), rtol=tol)
        sim.step(1)
    sim.close()


def test_asynchronous_results_reach_any_host_memory(kin):
    torch = pytest.importorskip("torch")
    N = 12
    sim = kin.Sim(N, kin.DUGKS, 0.013, 0.1, 0.5, kin.F32)
    sim.set_velocity(ki.random_velocity(N, N, N, 5, 0.03))
    want = np.array(sim.stats())
    pinned = torch.zeros(5, dtype=torch.float64, pin_memory=True).numpy()
    raw = torch.zeros(64, dtype=torch.uint8, pin_memory=True).numpy()
    odd = np.frombuffer(raw.data, dtype=np.float64, count=2, offset=4)  # page-locked, not 8-byte aligned
    pageable = np.zeros(2)
    for out in (pinned[1:3], pageable, odd):
        sim.stats_async(out)
        sim.sync()
        np.testing.assert_array_equal(out, want)
    assert pinned[0] == 0 and pinned[3] == 0 and pinned[4] == 0
    sim.close()
