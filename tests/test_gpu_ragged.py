"""The code form's lanes without a walker and its joined sweeps: walker counts around warps and
blocks, with one sweep, a few, and flushes in between, against the one-warp form."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("system,L,q", [(0, 8, 2), (0, 12, 2), (0, 64, 2), (2, 8, 2), (2, 32, 2), (2, 48, 2), (1, 8, 3),
                                        (1, 24, 7)])
@pytest.mark.parametrize("p", [1, 31, 33, 64, 97])
def test_code_form_equals_one_warp_form(system, L, q, p):
    import paper_1312_2213_gb300 as m

    gs = []
    for pipeline in (2, 0):
        g = m.Muca(system, L, q, p, 21, beta=0.4407 if system == 2 else None, block=64)
        g.set_param("pipeline", pipeline)
        for it, (sweeps, flush) in enumerate(((1, 0), (7, 3), (4, 1))):
            g.set_param("flush_every", flush)
            g.iterate(sweeps)
            g.merge_and_update()
        gs.append((g.histogram(), g.spins(), g.bins(), g.lnW(), tuple(sorted(g.metrics().items()))))
        g.close()
    a, b = gs
    for x, y in zip(a[:4], b[:4]):
        assert np.array_equal(x, y)
    assert a[4] == b[4]
