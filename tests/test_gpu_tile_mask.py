"""The candidate-mask tile (variant 2) against the thread-per-bead tile
(variant 1): the same trajectory bits and pair counts over box sides at the
edges of its blocks, populations from a bead in ten cells to windows and
queues that overflow, every option of the pair force, and thermo sums over
velocities from rest to beyond its integer range."""
import numpy as np
import pytest

from paper_1310_0998_gb300 import synth

pytestmark = pytest.mark.gpu


def _run(L, nd, x, v, steps=6, **kw):
    from paper_1310_0998_gb300 import Sim
    with Sim(L, 2 * nd, seed=5, **kw) as s:
        s.set_positions(x, v, step=(1 << 32) - 3)   # the step's low word wraps
        s.step(steps)
        out = s.get_state()[:3]
        return (*out, s.pair_counts()[0], s.thermo_log((1 << 32) - 3 + 1, steps), s.info())


@pytest.mark.parametrize("L,nd,tile,kw", [
    (3.0, 9, 8, {}), (4.5, 20, 4, {}), (9.0, 100, 8, {}), (17.0, 500, 16, {}), (33.25, 900, 16, {}),
    (40.0, 60, 16, {}),                                     # dilute
    (12.0, 1500, 4, {}), (20.0, 2000, 8, {}),               # 20 and 10 beads a cell: several windows, full queues
    (32.0, 1536, 0, dict(exclude_bonded=0)), (32.0, 1536, 8, dict(noise=1)), (32.0, 1536, 16, dict(wexp=1.0)),
    (20.0, 800, 0, dict(rc=0.5, r0=0.75)),                  # bonds longer than r_c
])
def test_same_bits_as_thread_per_bead(L, nd, tile, kw):
    x, _ = synth.dimers(nd, L, kw.get("r0", 0.5), seed=nd)
    v = synth.velocities(2 * nd, 0.7, seed=nd + 1)
    a = _run(L, nd, x, v, variant=2, tile=tile, **kw)
    b = _run(L, nd, x, v, variant=1, tile=8, **kw)
    for u, w in zip(a[:4], b[:4]):
        np.testing.assert_array_equal(u, w)
    # FP64 sums in another order: one rounding per term at most
    np.testing.assert_allclose(a[4], b[4], rtol=2 * nd * 2.3e-16, atol=2 * nd * 2.3e-16 * np.abs(b[4]).max())
    assert a[5].overflow_tiles == 0


@pytest.mark.parametrize("scale", [0.0, 1e-12, 1e-3, 1.0, 300.0])
@pytest.mark.parametrize("one", [0.0, 5.0e2])
def test_thermo_sums_over_velocity_ranges(scale, one):
    """Kinetic energy and momentum of the set-up state against numpy's FP64
    sums, with one bead far above the rest (beyond the tile's integer range)."""
    from paper_1310_0998_gb300 import Sim
    L, nd = 512.0, 300
    x, _ = synth.dimers(nd, L, 0.5, seed=3)
    v = synth.velocities(2 * nd, 1.0, seed=4) * np.float32(scale)
    v[17] = one
    with Sim(L, 2 * nd, seed=1, kBT=0.0, variant=2) as s:
        s.set_positions(x, v)
        ke, p = s.kinetic_energy(), s.momentum()
    w = v.astype(np.float64)
    assert abs(ke - 0.5 * (w * w).sum()) <= 2 * nd * 2.3e-16 * (w * w).sum()
    np.testing.assert_allclose(p, w.sum(0), rtol=0, atol=2 * nd * 2.3e-16 * np.abs(w).sum())


def test_batch_classes_same_bits_as_alone():
    """Replicas of very different density and size (three classes of threads per
    tile, one of them a single block) follow the bits of the same boxes alone."""
    from paper_1310_0998_gb300 import Ensemble, Sim
    pts = [dict(L=L, n_beads=2 * nd, seed=r, replica=r) for r, (L, nd) in
           enumerate([(256.0, 98304), (256.0, 40000), (320.0, 5000), (8.0, 40), (300.0, 20000), (400.0, 200000)])]
    with Ensemble(pts) as ens:
        ens.init_random(2)
        ens.step(11)
        ens.sync()
        got = [ens.replica(r).get_state() for r in range(len(pts))]
    for r, pt in enumerate(pts):
        kw = {k: w for k, w in pt.items() if k not in ("L", "n_beads")}
        with Sim(pt["L"], pt["n_beads"], **kw) as s:
            s.init_random(2 + r)
            s.step(11)
            for u, w in zip(got[r][:3], s.get_state()[:3]):
                np.testing.assert_array_equal(u, w)
