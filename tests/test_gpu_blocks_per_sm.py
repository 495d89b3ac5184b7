"""Many walkers at small L: blocks small enough to share an SM do, so that no launch shape falls behind
for want of registers."""
import pytest

pytestmark = pytest.mark.gpu


def _ms(system, L, q, p, block, sweeps):
    import torch

    import paper_1312_2213_gb300 as m

    g = m.Muca(system, L, q, p, 7, beta=0.4407 if system == 2 else None, block=block)
    for _ in range(6):
        g.iterate(20)
        g.merge_and_update()
    best = None
    for _ in range(4):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        g.iterate(sweeps)
        b.record()
        torch.cuda.synchronize()
        t = a.elapsed_time(b)
        best = t if best is None else min(best, t)
    g.close()
    return best


@pytest.mark.parametrize("L,sweeps", [(8, 1200), (16, 300)])
def test_potts_blocks_of_32_and_64_walkers(L, sweeps):
    """16384 walkers: blocks of 32 keep up with blocks of 64 (they took a fifth longer with two of
    them an SM)."""
    t32, t64 = (_ms(1, L, 8, 16384, b, sweeps) for b in (32, 64))
    assert t32 < 1.1 * t64, (t32, t64)


@pytest.mark.parametrize("system", [0, 2])
def test_ising_and_muma_L8_with_many_walkers(system):
    """131072 walkers at L = 8 take less than 6.3 times as long as 16384 (8 times the work in blocks that
    share the SMs; with two blocks an SM it took 6.7)."""
    t16, t128 = (_ms(system, 8, 2, p, None, 300) for p in (16384, 131072))
    assert t128 < 6.3 * t16, (t16, t128)


@pytest.mark.parametrize("system,L,q,p,block", [(0, 8, 2, 19457, None), (2, 8, 2, 19457, None), (2, 8, 2, 19470, 32),
                                                (1, 8, 3, 4865, 32), (1, 16, 10, 4890, 32), (1, 24, 7, 4865, 32)])
def test_forms_for_many_walkers_equal_the_one_warp_form(system, L, q, p, block):
    """The launches that put more blocks on an SM, just above the walker counts where they begin."""
    import numpy as np

    import paper_1312_2213_gb300 as m

    gs = []
    for pipeline in (2, 0):
        g = m.Muca(system, L, q, p, 21, beta=0.4407 if system == 2 else None, block=block)
        g.set_param("pipeline", pipeline)
        for sweeps, flush in ((1, 0), (7, 3), (4, 1)):
            g.set_param("flush_every", flush)
            g.iterate(sweeps)
            g.merge_and_update()
        gs.append((g.histogram(), g.spins(), g.bins(), g.lnW(), tuple(sorted(g.metrics().items()))))
        g.close()
    for x, y in zip(gs[0][:4], gs[1][:4]):
        assert np.array_equal(x, y)
    assert gs[0][4] == gs[1][4]
