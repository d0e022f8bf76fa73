"""Thermo sums of a dilute box whose tiles have two warps, with a cluster that no
tile's shared memory holds: the tiles that take the global-memory path add all of
kinetic energy and momentum."""
import numpy as np
import pytest

from paper_1310_0998_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [False, True])
def test_sums_with_a_cluster(batch):
    from paper_1310_0998_gb300 import Ensemble, Sim
    L, nd, k = 430.0, 40000, 2500            # 26 x 26 blocks of 16 x 16 cells, 110 beads each on average
    x, _ = synth.dimers(nd, L, 0.5, seed=1)
    c = np.random.default_rng(2).uniform(50.0, 60.0, (k, 2))
    x[0:2 * k:2], x[1:2 * k:2] = c, c + [0.3, 0.2]
    v = synth.velocities(2 * nd, 0.5, seed=3) + np.array([0.25, 0.75], np.float32)
    kw = dict(L=L, n_beads=2 * nd, dt=1e-5, tile=16, variant=2, seed=4)
    if batch:
        with Ensemble([kw, kw]) as ens:
            s = ens.replica(1)
            for r in range(2):
                ens.replica(r).set_positions(x, v)
            ens.step(1)
            ens.sync()
            over, log, (_, vs, _, _) = s.info().overflow_tiles, s.thermo_log(1, 1)[0], s.get_state()
    else:
        with Sim(**kw) as s:
            s.set_positions(x, v)
            s.step(1)
            over, log, (_, vs, _, _) = s.info().overflow_tiles, s.thermo_log(1, 1)[0], s.get_state()
    assert over > 0
    v64 = vs.astype(np.float64)
    want = np.array([0.5 * (v64 * v64).sum(), v64[:, 0].sum(), v64[:, 1].sum()])
    # FP64 sums of 80,000 terms, each tile's to 2^-53 of its terms
    np.testing.assert_allclose(log[:3], want, rtol=0, atol=2 * nd * 2.0**-52 * np.abs(v64).max() ** 2)
