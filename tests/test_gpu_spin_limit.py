"""Waits that give up at once: with a limit of a few tries the code form either runs as it should or
reports MUCA_ERR_TIMEOUT, its bins stay inside the table, and the context goes on from a checkpoint."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("system,L,q", [(0, 8, 2), (0, 64, 2), (2, 8, 2), (2, 32, 2), (1, 8, 3), (1, 32, 8), (1, 48, 10),
                                        (1, 64, 10)])
@pytest.mark.parametrize("p,limit", [(64, 1), (100, 1), (100, 2)])
def test_waits_that_give_up_early(system, L, q, p, limit):
    import paper_1312_2213_gb300 as m

    make = lambda: m.Muca(system, L, q, p, 5, beta=0.4407 if system == 2 else None, block=32 if L == 48 else 64)
    g, ref = make(), make()
    ref.set_param("pipeline", 0)
    for c in (g, ref):
        c.iterate(2)
        c.merge_and_update()
    blob = g.get_state()
    g.set_param("spin_limit", limit)
    g.set_param("flush_every", 3)
    g.iterate(10)
    timed_out = False
    try:
        g.synchronize()
    except m.MucaError as e:
        assert e.code == -4
        timed_out = True
    bins = np.zeros(p, dtype=np.int32)
    try:
        m.muca_get_walker_bins(g.h, bins)
    except m.MucaError as e:
        assert timed_out and e.code == -4
    assert np.all((bins >= 0) & (bins < g.B))
    if timed_out:
        g.set_state(blob)
        g.set_param("spin_limit", 0)
        g.iterate(10)
    g.merge_and_update()
    g.synchronize()
    ref.iterate(10)
    ref.merge_and_update()
    for a, b in ((g.histogram(), ref.histogram()), (g.bins(), ref.bins()), (g.spins(), ref.spins())):
        assert np.array_equal(a, b)
