"""States through page-locked host arrays that kernels read and write
themselves, against the copied route of pageable arrays: the same bits and
thermo sums for arrays at every alignment of their elements, for mixed
arrays, odd and tiny counts, and the same refusal of values that are not
finite."""
import numpy as np
import pytest

from paper_1310_0998_gb300 import synth

pytestmark = pytest.mark.gpu


def _pinned(a, off):
    """Page-locked copy of a whose first element is `off` elements into its
    allocation."""
    import torch
    t = torch.empty(a.size + off + 1, dtype=getattr(torch, str(a.dtype)), pin_memory=True).numpy()
    t[:] = 77.0
    q = t[off:off + a.size].reshape(a.shape)
    q[:] = a
    return t, q


@pytest.mark.parametrize("nd,L", [(1, 4.0), (333, 17.0), (70001, 200.0)])
@pytest.mark.parametrize("offs", [(0, 0, 0), (1, 0, 1), (0, 1, 0), (1, 1, 1), (None, 0, 0), (0, None, 1), (1, 1, None)])
def test_same_bits_as_copied(nd, L, offs):
    from paper_1310_0998_gb300 import Sim
    x, _ = synth.dimers(nd, L, 0.5, seed=nd)
    v = synth.velocities(2 * nd, 1.0, seed=nd + 1)
    with Sim(L, 2 * nd, seed=3) as s:
        s.set_positions(x, v)
        s.step(2)
        ref = s.get_state()
        s.set_state(*ref[:3], 9)
        th = s.thermo_log(9, 1)
        s.step(3)
        out = s.get_state()
        held = [(None, a.copy()) if o is None else _pinned(a, o) for a, o in zip(ref[:3], offs)]
        s.set_state(*[q for _, q in held], 9)
        # the same terms summed by blocks in another order
        np.testing.assert_allclose(s.thermo_log(9, 1), th, rtol=4 * nd * 2.3e-16, atol=4 * nd * 2.3e-16 * np.abs(v).sum())
        s.step(3)
        for _, q in held:
            q[:] = 0
        s.get_state(*[q for _, q in held])
        for (t, q), a, o in zip(held, out[:3], offs):
            np.testing.assert_array_equal(q, a)
            if t is not None:   # nothing written beside the array
                assert np.all(t[:o] == 77.0) and np.all(t[o + a.size:] == 77.0)


@pytest.mark.parametrize("which", [0, 1, 2])
def test_not_finite_is_refused(which):
    from paper_1310_0998_gb300 import Sim
    from paper_1310_0998_gb300._lib import DpdError
    nd, L = 50, 9.0
    x, _ = synth.dimers(nd, L, 0.5, seed=1)
    a = [x, synth.velocities(2 * nd, 1.0, seed=2), np.zeros((2 * nd, 2), np.float32)]
    a[which] = a[which].copy()
    a[which][31, 1] = np.nan
    held = [_pinned(q, 0) for q in a]
    with Sim(L, 2 * nd, seed=3) as s:
        with pytest.raises(DpdError, match="NONFINITE"):
            s.set_state(*[q for _, q in held], 0)
