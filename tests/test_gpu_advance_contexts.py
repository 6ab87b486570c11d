"""dem_advance on several contexts in turn.

A launch of the driver works from a copy of its context's state in each
block's shared memory.  Contexts of different sizes are advanced in turn here,
a step or a few at a time, so that what an SM's shared memory held before is
another context's; most sizes leave warps without a particle, which come to
the copy first.  Without contacts every array must equal the same steps phase
by phase bit for bit (the same roundings), and every counter must have gone to
its own context.
"""
import numpy as np
import pytest

from paper_2208_13770_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _lvb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2208_13770_gb300 import lvb
    return lvb


@pytest.mark.parametrize("threads", [256, 512, 1024])
@pytest.mark.parametrize("block", [False, True])
def test_contexts_in_turn_match_the_phases(threads, block):
    lvb = _lvb()

    def make(n):
        s = scenes.ballistic(n=n, seed=71 + n, phi=0.19)
        s.vel[:, :3] *= 400.0              # walls and list updates within a few steps
        return s

    def context(n):
        dem = lvb.DEM(make(n))
        dem.lvb.set_option(lvb.LVB_OPT_BLOCK_THREADS, threads)
        if block:
            dem.lvb.set_option(lvb.LVB_OPT_COMPACT, lvb.LVB_COMPACT_BLOCK)
        return dem

    sizes = (1, 33, 700, 2049, 9000)
    turns = (1, 2, 1, 3, 1, 5)
    here = [context(n) for n in sizes]
    for m in turns:
        for dem in here:
            dem.advance(m)
    flagged = 0
    for n, a in zip(sizes, here):
        b = lvb.DEM(make(n))
        for _ in range(sum(turns)):
            b.step()
        assert a.sync() == lvb.LVB_OK and b.sync() == lvb.LVB_OK
        for x, y in zip(a.state(), b.state()):
            assert np.array_equal(x, y)
        assert np.array_equal(a.lvb.ref(), b.lvb.ref())
        assert np.array_equal(a.lvb.flags(), b.lvb.flags())
        pa, pb = a.lvb.pairs_ij(), b.lvb.pairs_ij()
        assert np.array_equal(pa[0], pb[0]) and np.array_equal(pa[1], pb[1])
        sa, sb = a.lvb.stats(), b.lvb.stats()
        for key in ("steps", "flagged_total", "updated_total", "rebuild_steps"):
            assert sa[key] == sb[key], (n, key)
        flagged += sa["flagged_total"]
        a.close()
        b.close()
    assert flagged > sum(sizes)
