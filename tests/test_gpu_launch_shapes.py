"""Launch shapes chosen by the library give the bits of the explicit ones.

The fused DUGKS step picks its tile height (5, 8 or 11 rows; FP64 3 or 7) and z
chunk, and for N = 31 and 32 may hold whole rows in a warp; the LBE step puts two rows in a block for boxes of 33 to 64; a cell's arithmetic
does not depend on either, so every choice is compared bitwise with 4-row tiles
of three planes, or with one-warp LBE blocks.  Odd and ragged sizes leave
partial tiles, chunks and blocks on every side.
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


def _run(kin, N, scheme, storage, steps, **tuning):
    sim = kin.Sim(N, scheme, 0.013, 0.1, 1.0 if scheme == kin.LBE_MRT else 0.5, storage)
    if tuning:
        sim.set_tuning(**tuning)
    sim.set_velocity(ki.random_velocity(N, N, N, 900 + N, 0.03))
    sim.step(steps)
    f = sim.get_f()
    sim.check_guards()
    sim.close()
    return f


@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("N", [2, 11, 30, 31, 32, 45, 61, 64, 97])
def test_dugks_default_shape_is_bitwise_the_small_tiles(kin, N, storage):
    ref = _run(kin, N, kin.DUGKS, storage, 2, tile_y=4, zchunk=3)
    np.testing.assert_array_equal(_run(kin, N, kin.DUGKS, storage, 2), ref)


@pytest.mark.parametrize("N", [3, 30, 31, 32, 33, 45])
def test_dugks_fp64_shapes_agree_bitwise(kin, N):
    """Chunks of 1, 5 and 16 planes take 3- or 7-row tiles and, at 31 and 32,
    whole-row warps or 30-column tiles."""
    ref = _run(kin, N, kin.DUGKS, kin.F64, 2)
    for zc in (1, 5, 16):
        np.testing.assert_array_equal(_run(kin, N, kin.DUGKS, kin.F64, 2, zchunk=zc), ref)


@pytest.mark.parametrize("storage", [0, 1, 2, 3])
@pytest.mark.parametrize("N", [5, 32, 33, 34, 49, 63, 64, 65])
def test_lbe_default_blocks_are_bitwise_the_one_warp_blocks(kin, N, storage):
    ref = _run(kin, N, kin.LBE_MRT, storage, 3, block_x=32)
    np.testing.assert_array_equal(_run(kin, N, kin.LBE_MRT, storage, 3), ref)
    np.testing.assert_array_equal(_run(kin, N, kin.LBE_MRT, storage, 3, block_x=256), ref)


@pytest.mark.parametrize("steps", [2, 5])
@pytest.mark.parametrize("N", [87, 88, 89, 97, 121])
def test_lbe_step_pairs_are_bitwise_single_steps(kin, N, steps):
    """From 88^3 on FP32 steps go in pairs (one pass over memory); an explicit
    block size keeps the single-step kernel.  Edges: tiles of 30 x 6 cells and z
    chunks with remainders, an odd step left over."""
    ref = _run(kin, N, kin.LBE_MRT, kin.F32, steps, block_x=128)
    np.testing.assert_array_equal(_run(kin, N, kin.LBE_MRT, kin.F32, steps), ref)


@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("N", [2, 3, 4, 5, 17, 31, 32])
def test_lbe_small_step_pairs_are_bitwise_single_steps(kin, N, storage):
    """Up to 32^3 steps go in pairs of one launch (4 rows x 2 planes a block)."""
    ref = _run(kin, N, kin.LBE_MRT, storage, 5, block_x=32)
    np.testing.assert_array_equal(_run(kin, N, kin.LBE_MRT, storage, 5), ref)


@pytest.mark.parametrize("scheme", [0, 1])
def test_steps_captured_in_a_graph(kin, scheme):
    """Steps launched to overlap the one before them, replayed from a graph."""
    torch = pytest.importorskip("torch")
    N, dt = 24, (1.0 if scheme == kin.LBE_MRT else 0.5)
    stream = torch.cuda.Stream()
    u = ki.random_velocity(N, N, N, 77, 0.03)
    sims = [kin.Sim(N, scheme, 0.013, 0.1, dt, kin.F32, stream=s) for s in (stream, None)]
    for s in sims:
        s.set_velocity(u)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        sims[0].step(4)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    sims[1].step(12)
    np.testing.assert_array_equal(sims[0].get_f(), sims[1].get_f())
    del g
    for s in sims:
        s.close()
