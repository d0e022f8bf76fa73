"""Host arrays of which two registrations hold the ends and nothing holds the
middle: a kernel must not run across the gap.  Such an array is copied, which
CUDA refuses; arrays inside one registration keep the direct route."""
import ctypes
import mmap

import numpy as np
import pytest

from paper_1310_0998_gb300 import synth

pytestmark = pytest.mark.gpu
PAGE = 1 << 16


def _runtime():
    import torch
    torch.zeros(1, device="cuda")
    return ctypes.CDLL("libcudart.so.13" if torch.version.cuda.startswith("13") else "libcudart.so.12")


def test_gap_between_registrations_is_refused():
    from paper_1310_0998_gb300 import Sim
    from paper_1310_0998_gb300._lib import DpdError
    rt = _runtime()
    L, nd = 100.0, 24 * PAGE // 32            # positions: 16 bytes a bead, 24 pages
    x, _ = synth.dimers(nd, L, 0.5, seed=1)
    v = synth.velocities(2 * nd, 1.0, seed=2)
    m = mmap.mmap(-1, 26 * PAGE)
    buf = np.frombuffer(m, np.uint8)
    off = -buf.ctypes.data % PAGE
    view = buf[off:off + 24 * PAGE].view(np.float64).reshape(2 * nd, 2)
    view[:] = x
    at = view.ctypes.data
    parts = [(at, 8 * PAGE), (at + 16 * PAGE, 8 * PAGE)]
    with Sim(L, 2 * nd, seed=3) as s:
        s.set_state(x, v, np.zeros_like(v))
        want = s.get_state()
        for a, n in parts:
            assert rt.cudaHostRegister(ctypes.c_void_p(a), ctypes.c_size_t(n), 0) == 0
        try:
            with pytest.raises(DpdError, match="CUDA"):
                s.set_state(view, v, np.zeros_like(v))
            rt.cudaGetLastError()
            with pytest.raises(DpdError, match="CUDA"):
                s.get_state(view, None, None)
            rt.cudaGetLastError()
            np.testing.assert_array_equal(view, x)
        finally:
            for a, _ in parts:
                rt.cudaHostUnregister(ctypes.c_void_p(a))
        # the whole array in one registration
        assert rt.cudaHostRegister(ctypes.c_void_p(at), ctypes.c_size_t(24 * PAGE), 0) == 0
        try:
            s.set_state(view, v, np.zeros_like(v))
            view[:] = 0.0
            s.get_state(view, None, None)
            np.testing.assert_array_equal(view, want[0])
        finally:
            rt.cudaHostUnregister(ctypes.c_void_p(at))
