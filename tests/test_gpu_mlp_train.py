"""Training of the skin network at the edges of its tiles and launches: one to
4,097 samples a batch (a partial tile, one tile, several, and more blocks than
an epoch's single launch takes), a partial last batch.

With one batch an epoch is one Adam step, whose size does not depend on
the gradient's: p' = p - lr g / (|g| + 1e-8).  Against the library's own
gradient of the same samples (checked against the oracle elsewhere), whose
sums run in another order (1e-4 of the largest component at most), the sign
and so the step agree wherever |g| exceeds 1e-3 of the largest: to 1e-4 lr and
one rounding of p.  Several batches: bit for bit the same twice, and a lower
loss.
"""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

LR = 1e-2


def _lvb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2208_13770_gb300 import lvb
    return lvb


def _samples(n, seed):
    rng = np.random.default_rng(seed)
    s = rng.normal(size=(n, 9)).astype(np.float32)
    s[:, 8] = 1.0 + 0.5 * np.tanh(s[:, 0] - 0.3 * s[:, 3])
    p0 = (rng.standard_normal(1377) * 0.2).astype(np.float32)
    return s, p0


@pytest.mark.parametrize("n", [2, 63, 64, 65, 513, 4096, 4097])
@pytest.mark.parametrize("kind", [0, 1])
def test_one_batch_is_one_adam_step(n, kind):
    lvb = _lvb()
    s, p0 = _samples(n, n)
    dev = torch.from_numpy(s).cuda()
    yr = np.zeros(2, np.float32)
    p, mu, isd, losses = lvb.mlp_train(dev, epochs=1, batch=n + 3, lr=LR, seed=1, params0=p0,
                                       y_range_out=yr, loss_kind=kind)
    g = np.zeros(1377, np.float32)
    loss = ctypes.c_double(0.0)
    ptr = lambda a: a.ctypes.data
    rc = lvb.lvb_mlp_grad(dev.data_ptr(), n, ptr(p0), ptr(mu), ptr(isd),
                          max(float(yr[0]), 1e-30) if kind else 0.0, ptr(g), ctypes.byref(loss))
    assert rc == lvb.LVB_OK
    assert abs(losses[0] - loss.value) <= 1e-6 * abs(loss.value)
    big = np.abs(g) > 1e-3 * np.abs(g).max()
    assert big.sum() > 300
    want = p0[big] - LR * g[big] / (np.abs(g[big]) + 1e-8)
    assert np.all(np.abs(p[big] - want) <= 1e-4 * LR + 2.0 ** -23 * np.abs(want))


@pytest.mark.parametrize("n,batch", [(1000, 1), (1000, 64), (1000, 65), (5000, 512), (9000, 4096),
                                     (9000, 4100)])
def test_batches_are_repeatable_and_lower_the_loss(n, batch):
    lvb = _lvb()
    s, p0 = _samples(n, 7)
    dev = torch.from_numpy(s).cuda()
    epochs = 3 if batch < 1000 else 30
    runs = [lvb.mlp_train(dev, epochs=epochs, batch=batch, lr=3e-3, seed=5, params0=p0)
            for _ in range(2)]
    for a, b in zip(runs[0][:3], runs[1][:3]):
        assert np.array_equal(a, b)
    losses = runs[0][3]
    assert np.all(np.abs(losses - runs[1][3]) <= 1e-6 * np.abs(losses))
    assert losses[-1] < 0.7 * losses[0] and np.all(np.isfinite(runs[0][0]))
