"""The batched training step (every member in one launch, 16- and 32-column
tiles) at row counts around its tiles, and independence of the members: what a
member learns does not depend on how many share its launches."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _data(n, seed):
    rng = np.random.default_rng(seed)
    X = np.stack([rng.uniform(0.1, 0.6, n), rng.uniform(0.5, 10.0, n), rng.uniform(0.01, 1.0, n),
                  rng.uniform(0.0, 3.0, n)], axis=1).astype(np.float32)
    Y = (np.sin(X @ rng.standard_normal((4, 40))) + 0.1 * rng.standard_normal((n, 40))).astype(np.float32)
    return X, Y


@pytest.mark.parametrize("n", [1, 15, 63, 64, 65, 128, 129, 257, 511, 700])
def test_gradients_against_mma_sync(n):
    from paper_1310_0998_gb300.surrogate import Surrogate
    X, Y = _data(n, n)
    s = Surrogate(members=3, max_rows=700, seed=2)
    out = []
    for tc in (True, False):
        s.set_backend(tc)
        out.append(s.gradients(2, X, Y))
    s.close()
    (la, ga), (lb, gb) = out
    assert abs(la - lb) <= 1e-5 * abs(lb)
    for a, b in zip(ga, gb):   # FP32 sums in another order can move a BF16 operand to its neighbour (2^-8)
        assert np.linalg.norm(a - b) <= 2e-3 * np.linalg.norm(b) + 1e-12


@pytest.mark.parametrize("n,batch", [(70, 7), (200, 64), (300, 100), (520, 256), (130, 130)])
def test_members_train_alone_as_together(n, batch):
    from paper_1310_0998_gb300.surrogate import Surrogate
    X, Y = _data(n, n + 1)
    got = []
    for members in (1, 3):
        s = Surrogate(members=members, max_rows=600, seed=9)
        s.gradients(0, X[:5], Y[:5])
        loss = s.fit(X, Y, epochs=3, batch=batch)
        got.append((loss, s.gradients(0, X, Y)[1]))
        s.close()
    assert all(np.isfinite(g[0]) for g in got)
    for a, b in zip(got[0][1], got[1][1]):
        np.testing.assert_array_equal(a, b)
