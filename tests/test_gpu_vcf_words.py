"""The velocity correlation's sums where its histogram words fill to their last
bit: agents that move alike (every product has the same limbs) and slow opposed
streams beside one fast agent (small negative products, whose low limbs are all
ones), in one and two shells that take most pairs, with cells and without; and
the accuracy of single products, in shells of few pairs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _state(D, L, na, seed):
    """Agents with both beads at one place, on the grid L 2^-16."""
    c = np.random.default_rng(seed).integers(0, 1 << 16, (na, D)) * (L / 65536.0)
    return c, np.repeat(c, 2, axis=0)


def _run(D, L, x, v, dr, nbins, dt=1e-6):
    from paper_1310_0998_gb300 import Sim, Sim3
    if D == 2:
        with Sim(L, len(x), dt=dt) as s:
            s.set_state(x, v, np.zeros_like(v))
            return s.velocity_correlation(dr, nbins)
    with Sim3(L, len(x), dt=dt, a=0.0, gamma=0.0, kBT=0.0, k_bond=0.0, f_p=0.0, zeta=0.0) as s:
        s.set_positions(x, v)
        return s.velocity_correlation(dr, nbins)


def _pair_sums(c, v, L, dr, nbins):
    """Counts and sums of v_a . v_b by shell, pair by pair (FP64, 80-bit sums)."""
    num, cnt = np.zeros(nbins, np.longdouble), np.zeros(nbins, np.int64)
    for a in range(len(c) - 1):
        d = c[a] - c[a + 1:]
        d -= L * np.rint(d / L)
        b = np.floor(np.sqrt((d * d).sum(1)) / dr).astype(np.int64)
        w = (v[a].astype(np.longdouble) * v[a + 1:]).sum(1)
        for k in range(nbins):
            m = b == k
            cnt[k] += m.sum()
            num[k] += w[m].sum()
    return num, cnt


@pytest.mark.parametrize("D,L,na,dr,nbins", [
    (2, 32.0, 10000, 40.0, 1), (2, 32.0, 10000, 13.0, 2), (2, 32.0, 4096, 10.0, 1), (2, 32.0, 6000, 5.0, 2),
    (3, 12.0, 10000, 16.0, 1), (3, 12.0, 4096, 4.0, 1)])
def test_one_velocity(D, L, na, dr, nbins):
    c, x = _state(D, L, na, na)
    cnt0 = None
    for u in ((0.3, 0.0, 0.1), (0.6, 0.8, 0.0), (1.1, 0.3, 0.7), (0.33, 0.81, 0.25), (-0.5, 0.0, 0.0)):
        u = np.array(u[:D], np.float32)
        v = np.tile(u, (2 * na, 1))
        _, _, num, cnt = _run(D, L, x, v, dr, nbins)
        if cnt0 is None:
            cnt0 = cnt
            if nbins == 1 and dr > L:
                assert cnt[0] == na * (na - 1) // 2
        np.testing.assert_array_equal(cnt, cnt0)
        want = cnt * float((u.astype(np.float64) ** 2).sum())
        # a product is good to 2^-48 of the largest, which it is here; a word that
        # loses its top bit is off by 3e-5
        np.testing.assert_allclose(num, want, rtol=2.0**-48)


@pytest.mark.parametrize("D,L,na,dr,nbins", [(2, 32.0, 4096, 40.0, 1), (2, 32.0, 4096, 10.0, 1), (3, 12.0, 4096, 4.0, 1)])
def test_crossing_streams(D, L, na, dr, nbins):
    """Half of the products just below zero: a high limb of -1 over ones."""
    c, x = _state(D, L, na, na + 2)
    vc = np.zeros((na, D), np.float32)
    vc[::2, 0] = 1.0
    vc[1::2, :2] = (-2.0**-33, 1.0)
    _, _, num, cnt = _run(D, L, x, np.repeat(vc, 2, axis=0), dr, nbins)
    want, wcnt = _pair_sums(c, vc.astype(np.float64), L, dr, nbins)
    np.testing.assert_array_equal(cnt, wcnt)
    np.testing.assert_allclose(num, want.astype(np.float64), rtol=2.0**-48)


@pytest.mark.parametrize("D,L,na,dr,nbins", [(2, 32.0, 4096, 40.0, 1), (2, 32.0, 4096, 10.0, 1), (3, 12.0, 4096, 4.0, 1)])
def test_slow_opposed_streams_and_one_fast_agent(D, L, na, dr, nbins):
    c, x = _state(D, L, na, na + 1)
    vc = np.zeros((na, D), np.float32)
    vc[:, 0] = np.where(np.arange(na) % 64 == 0, -2.0**-9, 2.0**-13)
    vc[7] = 1.0
    _, _, num, cnt = _run(D, L, x, np.repeat(vc, 2, axis=0), dr, nbins)
    want, wcnt = _pair_sums(c, vc.astype(np.float64), L, dr, nbins)
    np.testing.assert_array_equal(cnt, wcnt)
    # the products are whole multiples of 2^-26, their sums below 2^53 of them: exact
    np.testing.assert_array_equal(num, want.astype(np.float64))


@pytest.mark.parametrize("D,L,na,dr,nbins", [(2, 32.0, 300, 16.0 / 4000, 4000), (2, 32.0, 1000, 8.0 / 2500, 2500), (2, 48.0, 40, 0.02, 600),
                                             (3, 12.0, 300, 0.002, 3000), (3, 12.0, 700, 4.0 / 2000, 2000)])
@pytest.mark.parametrize("kind", ["alike", "head"])
def test_products(D, L, na, dr, nbins, kind):
    """Shells of a pair or two.  kind "head": the tail's velocity 2^-1 to 2^-24 of
    the head's, so that their sum needs more bits than FP32 has."""
    c, x = _state(D, L, na, na + 3)
    rng = np.random.default_rng(na)
    v = rng.standard_normal((2 * na, D)).astype(np.float32)
    if kind == "head":
        v[1::2] *= np.exp2(-rng.integers(1, 25, (na, 1))).astype(np.float32)
    _, _, num, cnt = _run(D, L, x, v, dr, nbins)
    vc = 0.5 * (v[0::2].astype(np.longdouble) + v[1::2].astype(np.longdouble))
    want, wcnt = _pair_sums(c, vc, L, dr, nbins)
    np.testing.assert_array_equal(cnt, wcnt)
    assert (cnt == 1).any()
    # a product is good to 2^-55 of the largest |v|^2 at least; the result is rounded to FP64
    v2 = (vc * vc).sum(1).max()
    err = np.abs(num - want)
    assert np.all(err <= cnt * 2.0**-55 * v2 + 2.0**-53 * np.abs(want)), float(err.max())


@pytest.mark.parametrize("D,L,na,dr,nbins", [(2, 32.0, 500, 16.0 / 100, 100), (2, 32.0, 2000, 8.0 / 30, 30), (3, 12.0, 500, 0.06, 100),
                                             (3, 12.0, 2000, 4.0 / 20, 20), (2, 32.0, 2000, 40.0, 1)])
@pytest.mark.parametrize("scale", [1.0, 1e-30, 1e25])
def test_wide_speeds(D, L, na, dr, nbins, scale):
    """One agent 2^12 times faster than the rest, and speeds whose squares are no
    FP32 numbers: every product, the mean and the mean square to FP64."""
    c, x = _state(D, L, na, na + 4)
    v = np.random.default_rng(na).standard_normal((2 * na, D))
    v[10:12] *= 4096.0
    v = (v * scale).astype(np.float32)
    g, _, num, cnt = _run(D, L, x, v, dr, nbins, dt=1e-35)
    vc = 0.5 * (v[0::2].astype(np.longdouble) + v[1::2].astype(np.longdouble))
    want, wcnt = _pair_sums(c, vc, L, dr, nbins)
    size, _ = _pair_sums(c, np.abs(vc), L, dr, nbins)   # sum of |v_a . v_b| component by component
    np.testing.assert_array_equal(cnt, wcnt)
    # FP64 products (three roundings each) added one by one: a sum of n terms
    # is off by n 2^-53 of their magnitudes at most
    assert np.all(np.abs(num - want) <= (cnt + 3) * 2.0**-53 * size)
    m2, v2 = (vc.mean(0) ** 2).sum(), (vc * vc).sum(1).mean()
    on = cnt > 0
    wg = (want[on] / cnt[on] - m2) / (v2 - m2)
    tol = ((cnt + 3) * 2.0**-53 * size)[on] / cnt[on] / (v2 - m2) + na * 2.0**-51 * (1.0 + np.abs(wg))
    assert np.all(np.abs(g[on] - wg) <= tol)


@pytest.mark.parametrize("D,L,na,dr,nbins", [(2, 32.0, 31, 5.0, 2), (2, 32.0, 290, 5.0, 2), (2, 32.0, 1200, 2.5, 4), (2, 32.0, 600, 0.02, 500),
                                             (3, 12.0, 33, 1.0, 4), (3, 12.0, 1500, 1.9, 2)])
def test_shares_of_few_cells(D, L, na, dr, nbins):
    """Grids of 9 to 27 cells, whose agents are shared out by 32."""
    c, x = _state(D, L, na, na + 9)
    v = np.random.default_rng(na).standard_normal((2 * na, D)).astype(np.float32)
    _, _, num, cnt = _run(D, L, x, v, dr, nbins)
    vc = 0.5 * (v[0::2].astype(np.longdouble) + v[1::2].astype(np.longdouble))
    want, wcnt = _pair_sums(c, vc, L, dr, nbins)
    np.testing.assert_array_equal(cnt, wcnt)
    assert np.all(np.abs(num - want) <= cnt * 2.0**-55 * (vc * vc).sum(1).max() + 2.0**-53 * np.abs(want))


@pytest.mark.parametrize("nbins", [4096, 4097, 6000, 8192])
@pytest.mark.parametrize("kind", ["alike", "wide"])
def test_many_shells(nbins, kind):
    """Both sides of the number of shells from which all pairs take a block's FP64
    histogram."""
    D, L, na = 2, 32.0, 500
    c, x = _state(D, L, na, 77)
    v = np.random.default_rng(78).standard_normal((2 * na, D)).astype(np.float32)
    if kind == "wide":
        v[10:12] *= 4096.0
    dr = 23.0 / nbins                     # past every pair (L 2^-1/2 = 22.6)
    _, _, num, cnt = _run(D, L, x, v, dr, nbins)
    vc = 0.5 * (v[0::2].astype(np.longdouble) + v[1::2].astype(np.longdouble))
    d = c[:, None, :] - c[None, :, :]
    d -= L * np.rint(d / L)
    b = np.floor(np.sqrt((d * d).sum(2)) / dr).astype(np.int64)
    i, j = np.triu_indices(na, 1)
    want, size = np.zeros(nbins, np.longdouble), np.zeros(nbins, np.longdouble)
    np.add.at(want, b[i, j], (vc[i] * vc[j]).sum(1))
    np.add.at(size, b[i, j], np.abs(vc[i] * vc[j]).sum(1))
    np.testing.assert_array_equal(cnt, np.bincount(b[i, j], minlength=nbins))
    v2 = (vc * vc).sum(1).max()
    bound = (cnt + 3) * 2.0**-53 * size if kind == "wide" or nbins > 4096 else cnt * 2.0**-55 * v2 + 2.0**-53 * np.abs(want)
    assert np.all(np.abs(num - want) <= bound)
