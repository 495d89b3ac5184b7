"""Lanes per walker of the polymer sweep: with a bead a lane at most, every grouping gives the same bits
(further lanes add zeros), and short chains in small groupings keep the SMs full."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("moves", [0, 1])
@pytest.mark.parametrize("N,lanes", [(2, (2, 4, 8, 16, 32)), (3, (4, 8, 16, 32)), (4, (4, 8, 16, 32)), (5, (8, 16, 32)),
                                     (8, (8, 16, 32)), (9, (16, 32)), (16, (16, 32))])
def test_groupings_with_a_bead_a_lane_agree(N, lanes, moves):
    import paper_1312_2213_gb300 as m

    states = []
    for g_ in lanes:
        g = m.Muca(m.POLYMER3D, N, 0, 77, 3, window=(2.0 * N, 6.0 * N))
        g.set_param("moves", moves)
        g.set_param("lanes", g_)
        for sweeps in (30, 7, 8):
            g.iterate(sweeps)
            g.merge_and_update()
        states.append(g.get_state())
        g.close()
    for s in states[1:]:
        assert np.array_equal(s, states[0])


@pytest.mark.parametrize("N", [3, 5, 13])
def test_a_lane_a_walker_fills_the_gpu(N):
    """32768 short chains, one lane each: about a quarter of the time of 16 lanes each (it took longer
    when a warp's slots left room for two warps an SM)."""
    import torch

    import paper_1312_2213_gb300 as m

    times = {}
    for lanes in (1, 16):
        g = m.Muca(m.POLYMER3D, N, 0, 32768, 3, window=(2.0 * N, 6.0 * N))
        g.set_param("lanes", lanes)
        best = None
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            g.iterate(40)
            b.record()
            torch.cuda.synchronize()
            t = a.elapsed_time(b)
            best = t if best is None else min(best, t)
        times[lanes] = best
        g.close()
    assert times[1] < 0.7 * times[16], times
