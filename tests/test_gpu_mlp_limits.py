"""Training where an epoch's blocks do not fit the device at once, and where they wait
too long for one another (both made on the host: a limit on the blocks, and an
arrival that nothing brings)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _lvb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2208_13770_gb300 import lvb
    return lvb


def _train(lvb, n, batch, blocks_max=64, extra=0, spins=1 << 22, epochs=2):
    rng = np.random.default_rng(n)
    s = rng.normal(size=(n, 9)).astype(np.float32)
    s[:, 8] = 1.0 + 0.5 * np.tanh(s[:, 0])
    dev = torch.from_numpy(s).cuda()
    p = (rng.standard_normal(lvb.LVB_MLP_PARAMS) * 0.2).astype(np.float32)
    p0 = p.copy()
    mu, isd = np.zeros(8, np.float32), np.zeros(8, np.float32)
    yr, losses = np.zeros(2, np.float32), np.zeros(epochs, np.float32)
    q = lambda a: a.ctypes.data
    rc = lvb.lvb_mlp_train_limits(dev.data_ptr(), n, epochs, batch, 3e-3, 5, 0, q(p), q(mu), q(isd),
                                  q(yr), q(losses), blocks_max, extra, spins)
    return rc, p, p0, losses


@pytest.mark.parametrize("n,batch", [(1000, 64), (1000, 65), (3000, 512), (9000, 4096)])
def test_launch_for_each_batch_gives_the_same_weights(n, batch):
    lvb = _lvb()
    rc, whole, p0, la = _train(lvb, n, batch)
    assert rc == lvb.LVB_OK
    rc, apart, _, lb = _train(lvb, n, batch, blocks_max=0)
    assert rc == lvb.LVB_OK
    assert np.array_equal(whole, apart) and not np.array_equal(whole, p0)
    assert np.all(np.abs(la - lb) <= 1e-6 * np.abs(la))      # atomic sums of the errors


@pytest.mark.parametrize("batch", [64, 512])
def test_wait_that_runs_out_is_reported(batch):
    lvb = _lvb()
    rc, p, p0, _ = _train(lvb, 3000, batch, extra=1, spins=1 << 10)
    assert rc == lvb.LVB_ETIMEOUT
    assert np.array_equal(p, p0)
    rc, p, p0, _ = _train(lvb, 3000, batch)                  # the device is as usable as before
    assert rc == lvb.LVB_OK and not np.array_equal(p, p0)
