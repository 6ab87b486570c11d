"""Contact history in rows of more than 32 entries (a large sphere among small
ones), whose records past the 32nd have no bit that says whether they need
clearing: every step against the binary64 friction oracle with the springs the
GPU held before it, through contacts that open, rebuilds and a re-layout.
"""
import numpy as np
import pytest

from paper_2208_13770_gb300 import scenes
from tests.test_gpu_friction import (GT_RATIO, KT_RATIO, MU, _check, _lvb, _params, _state)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_long_rows_keep_and_clear_their_springs(orc):
    lvb = _lvb()
    s = scenes.packed(n=3000, seed=29, vsigma=3.0)
    s.mu, s.kt_ratio, s.gt_ratio = MU, KT_RATIO, GT_RATIO
    rng = np.random.default_rng(4)
    s.pos[rng.choice(s.n, size=12, replace=False), 3] *= 3.2
    P = _params(orc, s)
    dem = lvb.DEM(s)
    rows, _ = dem.lvb.pairs_csr()
    assert np.diff(rows).max() > 32
    survived = 0
    for k in range(40):
        if k == 20:
            dem.lvb.set_option(lvb.LVB_OPT_FORCE_RELAYOUT, 1)
        before = _state(dem)
        if k % 2:
            dem.step()
        else:
            dem.advance(1)
        after = _state(dem)
        survived += _check(orc, s, P, before, after, dem.lvb.flags())
    assert dem.sync() == lvb.LVB_OK
    assert survived > 100
    # springs only where there is contact, and both sides opposite
    ci, cj, _, _, xi = dem.contact_history(sides=2)
    fwd = {(int(a), int(b)): q for q, (a, b) in enumerate(zip(ci, cj))}
    i = [q for (a, b), q in fwd.items() if a < b]
    j = [fwd[(b, a)] for (a, b), q in fwd.items() if a < b]
    assert np.array_equal(xi[i], -xi[j]) and np.any(xi != 0)
    dem.close()
