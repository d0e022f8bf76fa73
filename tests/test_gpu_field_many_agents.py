"""The window sums of more agents than 2^27 where 32 lanes share an agent's
windows: the number of threads does not fit in 32 bits."""
import pytest

pytestmark = pytest.mark.gpu


def test_last_agents_are_deposited():
    import torch

    from paper_1310_0998_gb300 import Sim
    na, last, L, M = (1 << 27) + 64, 64, 9000.0, 1024
    if torch.cuda.mem_get_info()[0] < 60 << 30:
        pytest.skip("needs 60 GB of device memory")
    g = torch.Generator("cuda").manual_seed(3)
    c = torch.rand((na, 2), dtype=torch.float64, device="cuda", generator=g) * L
    c[:, 1] *= 0.5                       # every agent below L / 2 but the last ones
    c[-last:, 1] = 0.7 * L + 0.2 * c[-last:, 1]
    # a window's edges lie on half grid points, every 2^21 units of L 2^-32: an axis of
    # an agent exactly there may hold a fifth grid point
    edges = int((torch.round(c * (2.0**32 / L)).to(torch.int64) % (1 << 22) == 1 << 21).sum())
    x = c.repeat_interleave(2, 0)
    del c
    v = torch.zeros((2 * na, 2), dtype=torch.float32, device="cuda")
    v[-2 * last:, 0] = 1.0
    with Sim(L, 2 * na, dt=1e-6) as s:
        s.set_state(x, v, torch.zeros_like(v))
        u, n = s.velocity_field(M, 4.0 * L / M)   # 4 x 4 grid points in each agent's window
    assert 0 <= n.sum() - 16.0 * na <= 5 * edges
    top = slice(int(0.6 * M), int(0.95 * M))
    assert n[top].sum() == 16.0 * last
    assert (u[top][n[top] > 0, 0] == 1.0).all()
