"""The default shape in dense boxes, alone and in batches: no block's tile is left
to the global-memory path by the box's mean density, and the bits are those of
the shapes named."""
import numpy as np
import pytest


pytestmark = pytest.mark.gpu


def _beads(L, rho):
    return int(rho * L * L) // 2 * 2


@pytest.mark.parametrize("L,rho", [(24.0, 40.0), (64.0, 24.0), (130.0, 30.0), (290.0, 3.9), (290.0, 6.0), (290.0, 12.0), (300.0, 24.0)])
def test_no_overflow_by_density(L, rho):
    from paper_1310_0998_gb300 import Sim
    n, out = _beads(L, rho), []
    for tile in (0, 8):
        with Sim(L, n, dt=1e-4, tile=tile, seed=2) as s:
            s.init_random(3)
            s.step(3)
            out.append(s.get_state())
            if tile == 0:
                assert s.info().overflow_tiles == 0
    for a, b in zip(out[0][:3], out[1][:3]):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("spec", [[(128.0, 14.0)] * 6, [(48.0, 14.0)] + [(192.0, 0.7)] * 3, [(32.0, 40.0)] + [(192.0, 0.7)] * 3])
def test_no_overflow_in_a_batch(spec):
    from paper_1310_0998_gb300 import Ensemble, Sim
    pts = [dict(L=L, n_beads=_beads(L, rho), dt=1e-4, seed=r) for r, (L, rho) in enumerate(spec)]
    with Ensemble(pts) as ens:
        ens.init_random(5)
        ens.step(3)
        ens.sync()
        assert [ens.replica(r).info().overflow_tiles for r in range(len(pts))] == [0] * len(pts)
        got = ens.replica(0).get_state()
    with Sim(**{k: v for k, v in pts[0].items()}) as s:
        s.init_random(5)
        s.step(3)
        want = s.get_state()
    for a, b in zip(got[:3], want[:3]):
        np.testing.assert_array_equal(a, b)
