"""A re-layout of the row store on the device under each trigger, in dense
cells (200 slots) and sparse ones:
the pair set equals the oracle's, and both rows of every pair hold it."""
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


def _bed(n):
    s = scenes.packed(n=n, seed=29)
    big = np.random.default_rng(29).choice(n, size=n // 40, replace=False)
    s.pos[big, 3] *= 3.0     # rows of more than 32 entries
    return s


def _same_list(ctx, sm, n):
    pi, pj = ctx.pairs_ij()
    assert np.array_equal(pi, sm.pi) and np.array_equal(pj, sm.pj)
    rows, col = ctx.pairs_csr()
    i = np.repeat(np.arange(n), np.diff(rows))
    assert set(zip(i.tolist(), col.tolist())) == \
        set(zip(pi.tolist(), pj.tolist())) | set(zip(pj.tolist(), pi.tolist()))


@pytest.mark.parametrize("trigger", [0, 1, 2])
@pytest.mark.parametrize("slots", [0, 200])
def test_relayout_keeps_the_list(orc, trigger, slots):
    lvb = _lvb()
    from oracle.statemachine import OracleLVB
    n = 3000
    s = _bed(n)
    x = s.pos.astype(np.float32)
    ctx = lvb.LVB(torch.from_numpy(x).cuda(), s.lo, s.hi, lvb.LVB_SKIN_DIAMETER_FACTOR, 0.1,
                  s.dt, trigger, 1.25)
    if slots:
        ctx.set_option(lvb.LVB_OPT_CELL_CAPACITY, slots)
    sm = OracleLVB(x, orc.SKIN_DIAMETER_FACTOR, 0.1, s.dt, ctx.stats()["rnl_max"], trigger)
    rng = np.random.default_rng(trigger)
    for step in range(4):
        who = rng.choice(n, size=200, replace=False)
        x[who, :3] += rng.normal(0.0, 5e-4, size=(200, 3)).astype(np.float32)
        before = ctx.stats()["relayouts"]
        if step % 2:
            ctx.set_option(lvb.LVB_OPT_FORCE_RELAYOUT, 1)
        ctx.step(torch.from_numpy(x).cuda())
        f, _ = sm.step(x)
        assert f.any() and np.array_equal(ctx.flags(), f)
        assert ctx.stats()["relayouts"] >= before + step % 2
        _same_list(ctx, sm, n)
    ctx.close()
