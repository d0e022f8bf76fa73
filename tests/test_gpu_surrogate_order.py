"""Every row enters every epoch of a training call once, while the host prepares
the next epochs' orders as the device works: at a learning rate that moves no weight the last
epoch's loss is the loss of the whole table, in which a few rows hold most of
the error."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,batch,epochs", [(200000, 2000, 6), (65536, 64, 3), (2000, 100, 60)])
def test_each_row_once_an_epoch(n, batch, epochs):
    from paper_1310_0998_gb300.surrogate import Surrogate
    rng = np.random.default_rng(n)
    X = rng.uniform(0.1, 3.0, (n, 4)).astype(np.float32)
    Y = rng.standard_normal((n, 40)).astype(np.float32)
    Y[rng.choice(n, 20, replace=False)] *= 1000.0
    s = Surrogate(members=1, max_rows=n, seed=4)
    loss = s.fit(X, Y, epochs=epochs, batch=batch, lr=1e-30)
    whole, _ = s.gradients(0, X, Y)      # the scaling is the training call's
    s.close()
    # FP32 sums: 3 adds a row in a minibatch, 3 n in the whole pass, half an ulp each
    # of a running sum at most as large as the total
    assert abs(loss - whole) <= (3 * batch + 3 * n + 64) * 2.0**-24 * whole
