"""dpd_set_params with the kernel shape named: what a caller of the default shape
may name, and a change of variant whose tile plan is larger."""
import ctypes

import numpy as np
import pytest

from paper_1310_0998_gb300 import synth

pytestmark = pytest.mark.gpu
STATE = -6


def _set(s, **kw):
    from paper_1310_0998_gb300 import _lib
    from paper_1310_0998_gb300.sim import make_params
    p = make_params(s.L, s.n, **kw)
    return _lib.lib().dpd_set_params(s._h, ctypes.byref(p))


@pytest.mark.parametrize("L,rho", [(24.0, 3.0), (64.0, 1.0), (300.0, 1.0)])
def test_tile_named_for_the_default_one(L, rho):
    """8 stands for the default tile, whatever the box made of it; the tile that
    dpd_get_info reports can be named too, another cannot."""
    from paper_1310_0998_gb300 import Ensemble, Sim
    n = int(rho * L * L) // 2 * 2
    with Sim(L, n) as s:
        tile = s.info().tile
        for t in (4, 8, 16):
            assert _set(s, tile=t) == (0 if t in (8, tile) else STATE)
        s.init_random(1)
        s.step(2)
    with Sim(L, n, tile=4) as s:
        assert [_set(s, tile=t) for t in (4, 8, 16)] == [0, STATE, STATE]
    with Ensemble([dict(L=L, n_beads=n)]) as ens:
        r = ens.replica(0)
        tile = r.info().tile
        for t in (4, 8, 16):
            assert _set(r, tile=t) == (0 if t in (8, tile) else STATE)


def test_variant_with_a_larger_tile_plan():
    """A dense box whose capacity the new variant's plan cannot hold: its tiles get
    a smaller one, and the bits stay."""
    from paper_1310_0998_gb300 import Sim
    L, nd = 64.0, 32768                       # 4096 beads and more in a 16 x 16 block
    x, _ = synth.dimers(nd, L, 0.5, seed=1)
    v = synth.velocities(2 * nd, 0.5, seed=2)
    want = None
    for first, then in ((2, 2), (1, 2), (1, 3), (3, 2), (2, 1)):
        with Sim(L, 2 * nd, dt=1e-3, tile=16, variant=first) as s:
            s.set_positions(x, v)
            s.step(2)
            assert _set(s, dt=1e-3, tile=16, variant=then) == 0
            s.step(2)
            got = s.get_state()
        if want is None:
            want = got
        for a, b in zip(got[:3], want[:3]):
            np.testing.assert_array_equal(a, b)
