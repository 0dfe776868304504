"""Steps captured in a CUDA graph: every replay advances the state by the captured
number of steps, whatever number of launches they were made of (LBE steps go in
pairs up to 32^3 and, in FP32, from 88^3 on)."""
import numpy as np
import pytest

import kin_inputs as ki

pytestmark = pytest.mark.gpu

REPLAYS = 3


@pytest.mark.parametrize("n", [2, 4, 6, 10])
@pytest.mark.parametrize("scheme,storage,N", [(0, 0, 24), (0, 1, 24), (0, 2, 9), (0, 0, 96), (0, 0, 48), (1, 0, 24)])
def test_replays_of_an_even_number_of_steps_advance(kin, scheme, storage, N, n):
    torch = pytest.importorskip("torch")
    dt = 1.0 if scheme == kin.LBE_MRT else 0.5
    stream = torch.cuda.Stream()
    u = ki.random_velocity(N, N, N, 177, 0.03)
    captured, alone = (kin.Sim(N, scheme, 0.013, 0.1, dt, storage, stream=s) for s in (stream, None))
    for s in (captured, alone):
        s.set_velocity(u)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        captured.step(n)
    for _ in range(REPLAYS):
        g.replay()
    torch.cuda.synchronize()
    # after the graph the simulation's own calls find the state where the replays left it
    captured.step(3)
    alone.step(REPLAYS * n + 3)
    np.testing.assert_array_equal(captured.get_f(), alone.get_f())
    del g
    captured.close()
    alone.close()
