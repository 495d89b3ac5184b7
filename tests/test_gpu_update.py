"""The weight update's ordered sum, ln W(r_{k+1}) = ln W(r_k) + lnR_k, against the same additions
made one after the other in binary64: every bit has to agree, for terms that tie, cross binades,
change the sum's sign, vanish, are subnormal or not finite."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _terms(kind, n, rng):
    if kind == "normal":
        return rng.normal(0.0, 0.3, n)
    if kind == "drift":  # as a converged run: down to -hundreds and back
        return np.where(np.arange(n) < n // 2, -0.9, 0.9) + rng.normal(0.0, 1e-3, n)
    if kind == "ties":  # odd multiples of half a unit in the last place of sums in [64, 128)
        r = (2 * rng.integers(-2000, 2000, n) + 1) * 2.0 ** -47
        r[0] = 80.0
        return r
    if kind == "crossing":  # noise about a power of two
        r = rng.normal(0.0, 2.0 ** -44, n)
        r[0] = 64.0
        return r
    if kind == "zeros":
        r = np.where(rng.random(n) < 0.5, 0.0, rng.normal(0.0, 1.0, n))
        r[: n // 3] = 0.0
        r[1] = -0.0
        return r
    if kind == "scales":
        return rng.choice([-1.0, 1.0], n) * 2.0 ** rng.uniform(-70, 20, n)
    if kind == "subnormal":
        return rng.integers(-1000, 1000, n) * 5e-324
    assert kind == "nonfinite"
    r = rng.normal(0.0, 1.0, n)
    r[n // 2] = np.inf
    r[3 * n // 4] = -np.inf
    return r


@pytest.mark.parametrize("system,L,q", [(0, 4, 2), (0, 8, 2), (1, 16, 5), (1, 64, 10)])
@pytest.mark.parametrize("kind", ["normal", "drift", "ties", "crossing", "zeros", "scales", "subnormal", "nonfinite"])
def test_ordered_sum_is_bit_exact(system, L, q, kind):
    import paper_1312_2213_gb300 as m

    p = 32
    g = m.Muca(system, L, q, p, 3)
    rl = np.flatnonzero(np.isfinite(g.lnW()))
    r = _terms(kind, rl.size - 1, np.random.default_rng(L))
    buf = g.get_state()
    # behind lnR: merged H, open histogram, thresholds, observable sums, metrics, tunnelling states
    off = buf.size - p - 64 - 48 * g.B - 4 * g.B * g.C - 16 * g.B - 8 * g.B
    lnR = np.zeros(g.B)
    lnR[: r.size] = r
    buf[off: off + 8 * g.B] = lnR.view(np.uint8)
    g.set_state(buf)
    g.merge_and_update()  # nothing counted: the terms are summed as they are
    want = np.zeros(rl.size)
    with np.errstate(all="ignore"):
        for k in range(r.size):
            want[k + 1] = want[k] + r[k]
    got = g.lnW()[rl]
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(got), nan)
    assert np.array_equal(got[~nan].view(np.uint64), want[~nan].view(np.uint64))
    g.close()


@pytest.mark.parametrize("recursion", [0, 1])
@pytest.mark.parametrize("p,block", [(70, 32), (1000, 32), (64, 64)])
def test_merge_and_flatness_over_blocks(recursion, p, block):
    """Merge rows and pair blocks at their edges: counts conserved, statistics of the reachable bins."""
    import paper_1312_2213_gb300 as m

    g = m.Muca(m.ISING2D, 16, 2, p, 9, block=block)
    g.set_param("recursion", recursion)
    for it in range(2):
        g.iterate(3)
        g.merge_and_update()
        h = g.histogram()
        assert int(h.sum()) == p * 256 * 3
        rl = np.flatnonzero(np.isfinite(g.lnW()))
        st = g.flatness()
        assert (st[0], st[2]) == (float(h[rl].min()), float(h[rl].max()))
        assert st[1] == float(h[rl].sum()) / rl.size
    g.close()
