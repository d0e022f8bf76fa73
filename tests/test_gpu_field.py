"""The window sums and transforms of the filtered field where their whole-number
paths can go wrong: window edges exactly on agents, windows that wrap onto
themselves, wide and empty windows, resting and tiny velocities, and transforms
of every length and number of lines per block."""
import numpy as np
import pytest

from oracle import observables as ob
from paper_1310_0998_gb300 import synth

pytestmark = pytest.mark.gpu


def _same_field(u, n, uo, no):
    np.testing.assert_array_equal(n, no)
    # sums of at most n.max() velocities in another order
    np.testing.assert_allclose(u, uo, rtol=0, atol=2.3e-16 * max(no.max(), 1) * max(np.abs(uo).max(), 1e-30) * 4)


@pytest.mark.parametrize("L,M,eps,kind", [
    (32.0, 64, 1.0, "lattice"), (32.0, 32, 3.0, "lattice"), (32.0, 128, 4.5, "lattice"),   # edges on agents
    (32.0, 8, 33.0, "random"), (32.0, 16, 32.0, "random"),                                  # wrapped windows
    (33.1, 100, 0.05, "random"), (33.1, 128, 14.0, "random"), (64.0, 1024, 1.0, "tiny")])
def test_windows(L, M, eps, kind):
    from paper_1310_0998_gb300 import Sim
    nd = 1024
    x, _ = synth.dimers(nd, 32.0, 0.5, seed=5)
    v = synth.velocities(2 * nd, 1.0, seed=6)
    if kind == "lattice":
        c = np.stack(np.meshgrid(np.arange(32.0), np.arange(32.0)), -1).reshape(-1, 2)
        x = np.repeat(c, 2, axis=0)
        x[0::2, 1] += 0.25
        x[1::2, 1] -= 0.25
        x %= L
    elif kind == "tiny":
        v *= np.float32(1e-39)      # denormal
        v[::3] = 0.0
        v[::7] = 1.5
    with Sim(L, 2 * nd, dt=1e-6) as s:
        s.set_state(x, v, np.zeros_like(v))
        u, n = s.velocity_field(M, eps)
        xs, vs = s.get_state()[:2]
    c, vc = ob.agent_com(xs, vs, L)
    _same_field(u, n, *ob.velocity_field(c, vc, L, M, eps))


@pytest.mark.parametrize("M", [4, 8, 32, 256, 512, 1024])
def test_spectrum_lengths(M):
    from paper_1310_0998_gb300 import Sim
    L, nd = 40.0, 1600
    x, _ = synth.dimers(nd, L, 0.5, seed=M)
    v = synth.velocities(2 * nd, 1.0, seed=M + 1)
    with Sim(L, 2 * nd) as s:
        s.set_positions(x, v)
        eps = min(L * np.sqrt(10.0 / nd), 50.0 * L / M)
        E, (u, _) = s.energy_spectrum(M, eps), s.velocity_field(M, eps)
    Eo = ob.energy_spectrum(u)
    np.testing.assert_allclose(E, Eo, rtol=1e-12, atol=1e-15 * Eo.max())


@pytest.mark.parametrize("L,nd,M,eps", [(12.0, 900, 4, 0.0), (12.0, 900, 8, 13.0), (12.0, 900, 16, 1.5),
                                        (16.0, 2000, 32, 0.0), (16.0, 2000, 128, 2.0)])
def test_cube(L, nd, M, eps):
    from paper_1310_0998_gb300 import Sim3
    x, _ = synth.dimers3(nd, L, 0.5, seed=nd)
    v = synth.velocities3(2 * nd, 1.0, seed=nd + 1)
    with Sim3(L, 2 * nd) as s:
        s.set_positions(x, v)
        u, n = s.velocity_field(M, eps)
        E = s.energy_spectrum(M, eps)
        xs, vs = s.get_state()[:2]
    if M <= 32:
        d = xs[0::2] - xs[1::2]
        d -= L * np.rint(d / L)
        c = np.mod(xs[1::2] + 0.5 * d, L)
        vc = 0.5 * (vs[0::2].astype(np.float64) + vs[1::2].astype(np.float64))
        e = eps if eps > 0 else L * (10.0 / nd) ** (1.0 / 3.0)
        _same_field(u, n, *ob.velocity_field3(c, vc, L, M, e))
    Eo = ob.energy_spectrum3(u)
    np.testing.assert_allclose(E, Eo, rtol=1e-12, atol=1e-15 * Eo.max())
