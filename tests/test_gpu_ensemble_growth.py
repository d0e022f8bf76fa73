"""A batch whose tiles outgrow their class's capacity: what growth changes, and
what it leaves alone."""
import ctypes
import time

import numpy as np
import pytest

from paper_1310_0998_gb300 import synth

pytestmark = pytest.mark.gpu

STILL = dict(a=0.0, gamma=0.0, kBT=0.0, k_bond=0.0, f_p=0.0, zeta=0.0, dt=1e-3)   # nothing moves
L, N = 64.0, 4096


def _clustered(k, side=6.0, seed=0):
    """N beads, the first k of them inside a square of `side`, agents spread evenly."""
    x, _ = synth.dimers(N // 2, L, 0.5, seed=seed)
    c = np.random.default_rng(seed + 1).uniform(0.0, side, (k // 2, 2)) + 17.0
    x[0:k:2] = c
    x[1:k:2] = c + [0.25, 0.1]
    return x


def _overflows(ens, r):
    return ens.replica(r).info().overflow_tiles


def test_growth_keeps_parameters_and_bits():
    """The tables keep the parameters that the replicas were created with (a
    replica's own dpd_set_params is for its own steps), and every replica's
    trajectory is that of a box alone."""
    from paper_1310_0998_gb300 import Ensemble, Sim, _lib
    from paper_1310_0998_gb300.sim import make_params
    pts = [dict(L=L, n_beads=N, dt=1e-3, seed=3 + r) for r in range(3)]
    x = [_clustered(2000 if r == 1 else 0, 14.0, seed=r) for r in range(3)]
    v = synth.velocities(N, 0.5, seed=9)
    with Ensemble(pts) as ens:
        for r in range(3):
            ens.replica(r).set_positions(x[r], v)
        other = make_params(L, N, dt=1e-3, seed=4, f_p=7.0)
        lib = _lib.lib()
        assert lib.dpd_set_params(ens.replica(1)._h, ctypes.byref(other)) == 0
        before = _overflows(ens, 1)
        for _ in range(10):
            ens.step(2)
            ens.sync()
        assert _overflows(ens, 1) > before     # there was something to grow for
        got = [ens.replica(r).get_state() for r in range(3)]
    for r in range(3):
        with Sim(L, N, dt=1e-3, seed=3 + r) as s:
            s.set_positions(x[r], v)
            s.step(20)
            want = s.get_state()
        for a, b in zip(got[r][:3], want[:3]):
            np.testing.assert_array_equal(a, b)


def test_growth_stops_at_the_largest_tile():
    """A cluster that no tile can hold takes the global-memory path for good: a
    synchronising call finds it there and leaves the graphs alone."""
    import torch

    from paper_1310_0998_gb300 import Ensemble

    def sync_ms(k):
        pts = [dict(STILL, L=L, n_beads=N + 4096 * (r == 0), seed=r) for r in range(24)]
        with Ensemble(pts) as ens:
            for r, pt in enumerate(pts):
                n = pt["n_beads"]
                x = np.random.default_rng(r).uniform(0.0, L, (n, 2))
                if r == 0 and k:
                    x[:k] = np.random.default_rng(50).uniform(17.0, 22.0, (k, 2))
                ens.replica(r).set_positions(x)
            for _ in range(15):          # up to the largest capacity: a quarter each
                ens.step(1)
                ens.sync()
            a = _overflows(ens, 0)
            took = []
            for _ in range(20):
                ens.step(1)
                torch.cuda.synchronize()
                t = time.perf_counter()
                ens.sync()
                took.append(time.perf_counter() - t)
            return 1e3 * min(took), _overflows(ens, 0) - a, ens.info()

    base, none, _ = sync_ms(0)
    full, some, info = sync_ms(7000)
    assert none == 0 and some > 0        # overflows go on
    assert info["grid"] > 0
    # a copy of statuses, as without overflows: well below the time that sorting the
    # work lists or rewriting a table takes, let alone the graphs of the next step
    assert full < 2.0 * base + 0.05, (base, full)


def test_growth_after_a_replicas_own_call():
    """Overflows that a replica's own synchronising call sees first still grow the
    batch: after a few steps none are left."""
    from paper_1310_0998_gb300 import Ensemble
    pts = [dict(STILL, L=L, n_beads=N, seed=r) for r in range(2)]
    with Ensemble(pts) as ens:
        for r in range(2):
            ens.replica(r).set_positions(_clustered(2600 if r == 0 else 0, 7.0, seed=r))
        for _ in range(12):
            ens.step(1)
            ens.replica(0).temperature()
            ens.sync()
        a = _overflows(ens, 0)
        assert a > 0
        ens.step(5)
        ens.sync()
        assert _overflows(ens, 0) == a
