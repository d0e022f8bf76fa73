"""The row-run pair kernel of the cube where its masks, runs and queue turn:
three cells a side (every cell is first or last of its row), ragged sides,
runs beyond 32 slots, nearly empty boxes, each option of the pair force;
and its whole-number thermo sums from rest to one bead far above the rest.
Forces against the FP64 all-pairs oracle (bounds as in test_gpu_3d)."""
import math

import numpy as np
import pytest

from paper_1310_0998_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,nd,kw", [
    (3.0, 14, {}), (3.0, 700, {}), (3.0625, 150, {}), (4.0, 1200, {}),       # 1, 52, 11 and 37 beads a cell
    (5.875, 16, {}), (7.25, 577, {}), (12.0, 9, {}), (9.5, 1290, dict(rc=0.9)),
    (6.0, 324, dict(exclude_bonded=0)), (6.0, 324, dict(noise=1)), (6.0, 333, dict(wexp=1.0)),
])
def test_forces_against_oracle(orc, L, nd, kw):
    from paper_1310_0998_gb300 import Sim3
    p = dict(a=25.0, gamma=4.5, kBT=1.0, rc=1.0, r0=0.5, zeta=0.1, dt=0.01, seed=7, **{k: v for k, v in kw.items() if k != "rc"})
    p["rc"] = kw.get("rc", 1.0)
    x, _ = synth.dimers3(nd, L, 0.5, seed=nd)
    v = synth.velocities3(2 * nd, 1.0, seed=nd + 1)
    step = (1 << 32) + 3
    with Sim3(L, 2 * nd, k_bond=100.0, f_p=1.0, **p) as s:
        s.set_positions(x, v, step=step)
        f = s.get_state()[2].astype(np.float64)
    fo, npairs = orc.forces3(orc.params(L=L, kbond=100.0, fp=1.0, **p), x, v.astype(np.float64), step)
    fn = np.linalg.norm(fo, axis=1)
    err = np.linalg.norm(f - fo, axis=1)
    assert np.linalg.norm(err) <= 1e-5 * np.linalg.norm(fo)
    assert np.max(err / np.maximum(fn, math.sqrt(float(np.mean(fn ** 2))))) <= 1e-5


@pytest.mark.parametrize("scale", [0.0, 1e-12, 1.0, 300.0])
@pytest.mark.parametrize("one", [0.0, 5.0e2])
def test_thermo_sums_over_velocity_ranges(scale, one):
    """Kinetic energy and momentum of the set-up state against numpy's FP64
    sums: one rounding per term at most (three per bead)."""
    from paper_1310_0998_gb300 import Sim3
    L, nd = 16.0, 1300
    x, _ = synth.dimers3(nd, L, 0.5, seed=3)
    v = synth.velocities3(2 * nd, 1.0, seed=4) * np.float32(scale)
    v[17] = one
    with Sim3(L, 2 * nd, seed=1, kBT=0.0, dt=1e-4) as s:   # a drift beyond L/4 is refused
        s.set_positions(x, v)
        th = s.thermo()
    w = v.astype(np.float64)
    assert abs(th[0] - 0.5 * (w * w).sum()) <= 6 * nd * 2.3e-16 * (w * w).sum()
    np.testing.assert_allclose(th[1:4], w.sum(0), rtol=0, atol=2 * nd * 2.3e-16 * np.abs(w).sum())
