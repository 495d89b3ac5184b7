"""The polymer's energy change from the lanes' sums at its largest: a lane's sum may reach 2^22, so a
walker's reaches 2^22 times its lanes, and its fixed-point form must be right up to there, in both
signs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
Q = 2.0 ** -32


def _lj(r):
    """4 (r^-12 - r^-6), cut at 2.5 and shifted, and |v| + |r v'|, the scale of its binary32 error."""
    v = 4.0 * (r ** -12 - r ** -6)
    return v - 4.0 * (2.5 ** -12 - 2.5 ** -6), np.abs(v) + np.abs(24.0 * r ** -6 - 48.0 * r ** -12)


@pytest.mark.parametrize("lanes", [16, 32])
@pytest.mark.parametrize("rising", [False, True])
def test_largest_sums_over_the_lanes(lanes, rising):
    """Bead 0 beside a cluster of all others: it leaves (the sum is negative, the walker above its
    window) or comes closer (positive, below the window).  The change of the first attempt against
    binary64 within 1e-6 of the pair terms' scale, as everywhere for the binary32 sums."""
    import paper_1312_2213_gb300 as m

    N, p = 128, 2048
    g = m.Muca(m.POLYMER3D, N, 0, p, 9, window=(226.0, 748.4))
    g.set_param("bin_width", 1.0)  # (E - e_lo) k stays far inside 64 bits
    g.set_param("lanes", lanes)
    buf = g.get_state()
    e_off = buf.size - p - 64 - 56 * g.B - 8 * p  # energies; before them bins and coordinates
    x_off = e_off - 4 * p - 24 * N * p
    # at distance r0 the lanes hold `each` apiece: 4 r0^-12 of 126 partners
    each = 2.0e5 if rising else 3.6e6
    r0 = (each * lanes / 126 / 4) ** (-1.0 / 12.0)
    X = np.zeros((p, 3, N), dtype=np.int64)
    X[:, 0, 1:] = int(r0 * 2.0 ** 44)
    E = np.full(p, int((-1.5e8 if rising else 1.5e8) * 2 ** 32), dtype=np.int64)
    buf[x_off: e_off - 4 * p] = X.reshape(-1).view(np.uint8)
    buf[e_off: e_off + 8 * p] = E.view(np.uint8)
    g.set_state(buf)
    r = g.iterate_traced(1)[:, 0, 0]
    moved = (r["flags"] & 7) == 1  # accepted, no bond broken, no lane's sum refused
    after = np.linalg.norm(g.coords()[moved][:, 2:], axis=2)  # bead 0 is the origin again
    new, s_new = _lj(after)
    old, s_old = _lj(np.full_like(after, int(r0 * 2.0 ** 44) * 2.0 ** -44))
    bond = lambda d: -0.5 * 40.0 * 1.5 ** 2 * np.log1p(-(d / 1.5) ** 2)
    want = (new - old).sum(1) + bond(after[:, 0]) - bond(r0)
    scale = (s_new + s_old).sum(1)
    got = r["dq"][moved] * Q
    big = np.abs(want) > lanes * 2.0 ** 21  # in the upper binade of what the lanes can hold
    assert big.sum() >= 10
    assert np.all((got > 0) == rising)
    assert np.all(np.abs(got - want) <= 1e-6 * scale), np.abs(got - want).max()
    g.close()
