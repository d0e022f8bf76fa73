"""The velocity correlation's pair pass against the FP64 oracle where it can go
wrong: histogram words that fill up (one or two shells), shells in thousands
(one warp per block), separations exactly on shell edges, velocities over nine
decades, cells capped below the box's own number, both dimensions."""
import numpy as np
import pytest

from oracle import observables as ob
from paper_1310_0998_gb300 import synth

pytestmark = pytest.mark.gpu


def _check(out, c, vc, L, dr, nbins, sums):
    g, _, num, cnt = out
    numo, cnto = sums(c, vc, L, dr, nbins)
    np.testing.assert_array_equal(cnt, cnto)
    # a product is good to 2^-52 of the largest |v|^2; the oracle's FP64 sums round once per term
    v2 = (vc * vc).sum(1).max()
    assert np.all(np.abs(num - numo) <= cnto * 6e-16 * v2 + 1e-300), np.abs(num - numo).max()


@pytest.mark.parametrize("L,nd,dr,nbins,kind", [
    (32.0, 4096, 10.0, 1, "random"), (32.0, 3000, 16.0, 2, "random"), (32.0, 900, 0.005, 3000, "random"),
    (48.0, 2500, 15.0 / 2048, 2048, "random"), (4100.0, 3000, 0.5, 2, "patch"), (32.0, 1024, 0.25, 40, "lattice"),
    (32.0, 1024, 1.0, 16, "lattice"), (33.1, 700, 0.3, 20, "wide"), (30.0, 33, 0.5, 30, "random"), (9.0, 1, 0.5, 5, "random")])
def test_pair_sums(L, nd, dr, nbins, kind):
    from paper_1310_0998_gb300 import Sim
    x, _ = synth.dimers(nd, 32.0 if kind in ("patch", "wide") else L, 0.5, seed=nd)
    if kind in ("patch", "wide"):
        x = np.mod(np.rint(x / L * 2.0**32), 2.0**32) * (L / 2.0**32)
    v = synth.velocities(2 * nd, 1.0, seed=nd + 1)
    if kind == "lattice":      # centres of mass on multiples of 1: every separation squared a whole number
        c = np.stack(np.meshgrid(np.arange(32.0), np.arange(32.0)), -1).reshape(-1, 2)[:nd]
        x = np.repeat(c, 2, axis=0)
        x[0::2, 0] += 0.25
        x[1::2, 0] -= 0.25
        x %= L
    if kind == "wide":
        v *= np.exp(np.random.default_rng(1).uniform(-14.0, 7.0, (2 * nd, 1))).astype(np.float32)
    with Sim(L, 2 * nd, dt=1e-6) as s:
        s.set_state(x, v, np.zeros_like(v))
        out = s.velocity_correlation(dr, nbins)
        xs, vs = s.get_state()[:2]
    c, vc = ob.agent_com(xs, vs, L)
    _check(out, c, vc, L, dr, nbins, ob.vcf_sums)


@pytest.mark.parametrize("L,nd,dr,nbins", [(12.0, 1500, 4.0, 1), (12.0, 1500, 0.25, 16), (12.0, 900, 3.0, 2),
                                           (20.0, 4000, 0.5, 4), (10.0, 300, 0.002, 2000)])
def test_pair_sums3(L, nd, dr, nbins):
    from paper_1310_0998_gb300 import Sim3
    x, _ = synth.dimers3(nd, L, 0.5, seed=nd)
    v = synth.velocities3(2 * nd, 1.0, seed=nd + 1)
    with Sim3(L, 2 * nd) as s:
        s.set_positions(x, v)
        out = s.velocity_correlation(dr, nbins)
        xs, vs = s.get_state()[:2]
    d = xs[0::2] - xs[1::2]
    d -= L * np.rint(d / L)
    c = np.mod(xs[1::2] + 0.5 * d, L)
    vc = 0.5 * (vs[0::2].astype(np.float64) + vs[1::2].astype(np.float64))
    _check(out, c, vc, L, dr, nbins, ob.vcf_sums3)
