"""lvb_clump_contacts on clumps of up to 64 sub-spheres that overlap one
another deeply: more partners' sub-spheres than fit registers, more pairs and
contacts to a warp than its queue and its buffer hold, sub-spheres right at
their bound; against the oracle's brute force, bit for bit.
"""
import numpy as np
import pytest

from tests.test_gpu_clumps import _dev, _lvb

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,most", [(1, 4), (2, 64), (33, 5), (300, 20), (1000, 4)])
def test_many_sub_spheres_match_oracle(orc, n, most):
    lvb = _lvb()
    rng = np.random.default_rng(100 * n + most)
    k = rng.integers(1, most + 1, size=n)
    k[0] = most
    off = np.concatenate([[0], np.cumsum(k)]).astype(np.int32)
    m = int(off[-1])
    sub = np.zeros((m, 4), np.float32)
    sub[:, :3] = rng.normal(0, 0.5e-3, size=(m, 3))
    sub[:, 3] = rng.uniform(0.1e-3, 0.5e-3, size=m)
    ext = np.linalg.norm(sub[:, :3].astype(np.float64), axis=1) + sub[:, 3]
    R = np.maximum.reduceat(ext, off[:-1]) / (1.0 - 2.0 ** -12)
    R = np.nextafter(R.astype(np.float32), np.float32(1.0))   # the smallest that is allowed
    pos = np.zeros((n, 4), np.float32)
    side = 1.2e-3 * n ** (1 / 3)
    pos[:, :3] = rng.uniform(0, side, size=(n, 3))
    pos[:, 3] = R
    q = rng.normal(size=(n, 4))
    q = (q / np.linalg.norm(q, axis=1, keepdims=True)).astype(np.float32)
    ctx = lvb.LVB(_dev(pos), (-1e-2,) * 3, (side + 1e-2,) * 3, lvb.LVB_SKIN_DIAMETER_FACTOR, 0.1,
                  1e-5, lvb.LVB_TRIGGER_PARTIAL, 1.25)
    got = ctx.clump_contacts(_dev(pos), _dev(q), _dev(off, np.int32), _dev(sub))
    want = orc.clump_contacts(pos, q, off, sub)
    for g, o in zip(got, want):
        assert np.array_equal(g, o)
    if n >= 33:
        assert len(want[0]) >= n
    ctx.close()
