"""Cell blocks of a box that leaves the side open: 4 x 4 up to 152 blocks of
8 x 8 with more than 64 beads each, at both edges of that rule, with the bits
of the thread-per-bead kernel on 8 x 8 blocks."""
import numpy as np
import pytest

from paper_1310_0998_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,nd,kw", [
    (32.0, 512, {}), (32.0, 513, {}),              # 64 beads in an 8 x 8 block, and more
    (96.0, 9000, {}), (97.0, 9000, {}),            # 144 and 169 blocks
    (3.0, 14, {}), (7.0, 300, {}),                 # fewer cells than a block; a dense box
    (20.5, 600, dict(rc=0.5, r0=0.75)), (40.0, 1800, dict(exclude_bonded=0)),
])
def test_same_bits_as_general_tile(L, nd, kw):
    from paper_1310_0998_gb300 import Sim
    x, _ = synth.dimers(nd, L, kw.get("r0", 0.5), seed=nd)
    v = synth.velocities(2 * nd, 0.7, seed=nd + 1)
    out = []
    for how in ({}, dict(variant=1, tile=8)):
        with Sim(L, 2 * nd, seed=5, **kw, **how) as s:
            s.set_positions(x, v)
            s.step(7)
            out.append(s.get_state()[:3])
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
