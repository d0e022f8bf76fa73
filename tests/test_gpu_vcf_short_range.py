"""The velocity correlation out to an r_max far below the cells' side (no cell
grid holds L / r_max cells a side): FP32 offsets inside such a cell are coarse
beside a shell, so pairs near a shell edge must go to the FP64 expressions."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _pairs(D, L, na, reach, seed):
    """Agents in pairs `reach` apart at most, both beads at one place; pairs on a
    lattice wider than any r_max used here."""
    rng = np.random.default_rng(seed)
    side = int(np.ceil((na / 2) ** (1.0 / D)))
    at = np.stack(np.meshgrid(*[np.arange(side)] * D), -1).reshape(-1, D)[:na // 2]
    a = (at + rng.uniform(0.1, 0.9, at.shape)) * (L / side)
    u = rng.standard_normal(at.shape)
    u *= (rng.uniform(0.0, reach, (len(at), 1)) / np.linalg.norm(u, axis=1, keepdims=True))
    c = np.stack([a, a + u], 1).reshape(-1, D)
    return np.repeat(np.mod(c, L), 2, axis=0)


@pytest.mark.parametrize("D,L,na,dr,nbins", [(2, 1000.0, 40000, 1e-5, 2), (2, 700.0, 40000, 3e-5, 9), (2, 1000.0, 3000, 2e-4, 40),
                                             (3, 300.0, 40000, 1e-5, 3), (3, 200.0, 40000, 7e-5, 20)])
def test_counts(D, L, na, dr, nbins):
    from paper_1310_0998_gb300 import Sim, Sim3
    x = _pairs(D, L, na, 1.2 * nbins * dr, na + nbins)
    v = np.random.default_rng(5).standard_normal(x.shape).astype(np.float32)
    if D == 2:
        with Sim(L, len(x), dt=1e-6) as s:
            s.set_state(x, v, np.zeros_like(v))
            cnt = s.velocity_correlation(dr, nbins)[3]
            xs = s.get_state()[0]
    else:
        with Sim3(L, len(x), dt=1e-6, a=0.0, gamma=0.0, kBT=0.0, k_bond=0.0, f_p=0.0, zeta=0.0) as s:
            s.set_positions(x, v)
            cnt = s.velocity_correlation(dr, nbins)[3]
            xs = s.get_state()[0]
    c = xs[0::2]                       # both beads, hence the centre
    d = c[0::2] - c[1::2]
    d = np.where(d > 0.5 * L, d - L, np.where(d < -0.5 * L, d + L, d))
    r2 = d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]
    if D == 3:
        r2 = r2 + d[:, 2] * d[:, 2]
    b = np.floor(np.sqrt(r2) / dr)
    np.testing.assert_array_equal(cnt, [(b == k).sum() for k in range(nbins)])


def test_few_agents_take_no_million_cells():
    """300 agents out to L / 100,000: as many cells as agents at most, not the
    4,194,304 that the box has room for (7 ms a call in the scan of their counts)."""
    import time

    from paper_1310_0998_gb300 import Sim
    L, na = 1000.0, 300
    x = _pairs(2, L, na, 0.01, 4)
    v = np.random.default_rng(6).standard_normal(x.shape).astype(np.float32)
    with Sim(L, len(x), dt=1e-6) as s:
        s.set_state(x, v, np.zeros_like(v))
        took = []
        for _ in range(8):
            t = time.perf_counter()
            s.velocity_correlation(1e-3, 10)
            took.append(time.perf_counter() - t)
    assert min(took) < 2e-3, took
