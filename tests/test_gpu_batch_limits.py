"""Kernels are shared by all contexts and batches of the process: a batch made for small systems
beside one of large systems leaves the large one runnable, in both forms, with and without a graph."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# form 1: q-Potts at L = 64 (the recursion's 65 KB of terms); form 0: the largest table of the tiles
LARGE = {1: [(1, 64, 10, 40), (0, 16, 2, 33)], 0: [(1, 48, 10, 40), (0, 16, 2, 33)]}


@pytest.mark.parametrize("form", [1, 0])
@pytest.mark.parametrize("use_graph", [False, True])
def test_small_batch_leaves_the_large_one_runnable(form, use_graph):
    import paper_1312_2213_gb300 as m

    make = lambda specs: [m.Muca(s, L, q, p, 50 + i) for i, (s, L, q, p) in enumerate(specs)]
    alone, large, small = make(LARGE[form]), make(LARGE[form]), make([(0, 8, 2, 32), (0, 4, 2, 32)])
    a = m.Batch(large, form=form)
    b = m.Batch(small, form=form)
    a.run(2, 3, use_graph=use_graph)
    b.run(2, 3, use_graph=use_graph)
    for c, d in zip(alone, large):
        for _ in range(2):
            c.iterate(3)
            c.merge_and_update()
        assert np.array_equal(c.get_state(), d.get_state())
    for x in (a, b, *alone, *large, *small):
        x.close()
