"""Velocity correlations of several host threads at once, each on its own box and
with another number of shells (another size of shared memory)."""
import threading

import numpy as np
import pytest

from paper_1310_0998_gb300 import synth

pytestmark = pytest.mark.gpu


def test_threads_with_different_shells():
    from paper_1310_0998_gb300 import Sim
    L, nd = 32.0, 300
    x, _ = synth.dimers(nd, L, 0.5, seed=1)
    v = synth.velocities(2 * nd, 1.0, seed=2)
    shells, got, errors = (1, 1000, 1, 2500), {}, []

    def work(k, nbins):
        try:
            with Sim(L, 2 * nd, dt=1e-6) as s:
                s.set_state(x, v, np.zeros_like(v))
                for _ in range(300):
                    for dr in (16.0 / nbins, 2.0 / nbins):   # all pairs, cells
                        cnt = s.velocity_correlation(dr, nbins)[3]
                        np.testing.assert_array_equal(cnt, got.setdefault((k, dr), cnt))
        except Exception as e:
            errors.append((nbins, e))

    t = [threading.Thread(target=work, args=a) for a in enumerate(shells)]
    for a in t:
        a.start()
    for a in t:
        a.join()
    assert not errors, errors
