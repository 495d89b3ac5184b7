"""The polymer sweep's unrolled loop (16 lanes, shifts, every walker of the warp inside its window)
against its general loop, which a traced iterate always takes: the same chains, energies, bins,
counts and metrics bit for bit, at the edges of a lane's partners (N = 16, 32, 64, 96, 128), of the
chunks of 16 beads and of the warps."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _context(m, N, p, model, record, bin_width=None):
    window = (2.0 * N, 6.0 * N) if model == 0 else (-3.6 * N, 3.0 * N)
    g = m.Muca(m.POLYMER3D, N, 0, p, 77, window=window, record=record)
    g.set_param("model", model)
    if bin_width:
        g.set_param("bin_width", bin_width)
    return g


@pytest.mark.parametrize("model,record", [(0, 0), (1, 1)])
@pytest.mark.parametrize("N,p", [(2, 33), (3, 64), (13, 70), (15, 31), (16, 70), (17, 70), (31, 33), (32, 70), (33, 70),
                                 (48, 33), (63, 33), (64, 70), (65, 33), (96, 33), (97, 33), (127, 33), (128, 70)])
def test_unrolled_loop_equals_the_general_loop(N, p, model, record):
    import paper_1312_2213_gb300 as m

    a, b = (_context(m, N, p, model, record) for _ in range(2))
    for it, sweeps in enumerate((40, 12, 12)):
        a.iterate(sweeps)
        r = b.iterate_traced(sweeps)
        a.merge_and_update()
        b.merge_and_update()
        inside = (r["b"][:, -1, -1] >= 0) & (r["b"][:, -1, -1] < a.B)
    assert inside.mean() > 0.5, "the walkers never reached the window"
    assert np.array_equal(a.histogram(), b.histogram())
    assert np.array_equal(a.get_state(), b.get_state())
    a.close()
    b.close()


def test_bin_of_energies_beyond_the_product():
    """The bin is the upper half of (E - e_lo) k modulo 2^64, clamped to [-1, B], also for energies
    (beads on top of each other) whose product with k leaves 64 bits."""
    import paper_1312_2213_gb300 as m

    p, N, k = 96, 5, 10
    g = m.Muca(m.POLYMER3D, N, 0, p, 4, window=(10.0, 30.0))
    buf = g.get_state()
    off = buf.size - p - 64 - 56 * g.B - 8 * p  # the energies lie before seven arrays of B words
    rng = np.random.default_rng(1)
    E0 = (rng.integers(-2 ** 62, 2 ** 62, p) >> rng.integers(0, 60, p)).astype(np.int64)
    buf[off: off + 8 * p] = E0.view(np.uint8)
    g.set_state(buf)
    r = g.iterate_traced(1)[:, 0, :]
    elo = np.int64(10 * 2 ** 32)
    with np.errstate(over="ignore"):
        before = np.concatenate([E0[:, None], r["E"][:, :-1]], axis=1)
        want = np.clip(((before + r["dq"] - elo) * np.int64(k)) >> np.int64(32), -1, g.B)
    assert np.array_equal(r["bn"], want)
    g.close()
