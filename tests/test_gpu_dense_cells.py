"""Patches in dense cells (more than 64 slots a cell): teams of 1, 4, 8, 16 and
32 warps to a row, by how many particles are flagged at the step, against the
oracle's state machine -- pair set and reference state after every step.

The cells are made dense by their slots (LVB_OPT_CELL_CAPACITY) and by a wide
mix of radii, so that a large particle has several hundred candidates and
more partners than a warp has lanes, and rows and noted candidates are taken up
in several goes.
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


def _bed(n, seed):
    """Spheres of 1 mm on a lattice, one in 40 of them three times as wide."""
    s = scenes.packed(n=n, seed=seed)
    rng = np.random.default_rng(seed)
    big = rng.choice(n, size=max(1, n // 40), replace=False)
    s.pos[big, 3] *= 3.0
    return s, big


@pytest.mark.parametrize("moved", [1, 3, 40, 300, 1500, 5000])
@pytest.mark.parametrize("history", [0, 1])
@pytest.mark.parametrize("threads", [1024, 256])
def test_teams_match_the_oracle(orc, moved, history, threads):
    lvb = _lvb()
    from oracle.statemachine import OracleLVB
    n = 6000
    s, big = _bed(n, 17)
    pos = s.pos.astype(np.float32)
    ctx = lvb.LVB(torch.from_numpy(pos).cuda(), s.lo, s.hi, lvb.LVB_SKIN_DIAMETER_FACTOR, 0.1,
                  s.dt, lvb.LVB_TRIGGER_PARTIAL, 1.25)
    ctx.set_option(lvb.LVB_OPT_CELL_CAPACITY, 512)
    ctx.set_option(lvb.LVB_OPT_BLOCK_THREADS, threads)
    if history:
        ctx.set_option(lvb.LVB_OPT_HISTORY, 1)
    sm = OracleLVB(pos, orc.SKIN_DIAMETER_FACTOR, 0.1, s.dt, ctx.stats()["rnl_max"], 0)
    rng = np.random.default_rng(moved)
    x = pos.copy()
    for step in range(5):
        who = rng.choice(n, size=moved, replace=False)
        if step == 2:
            who[0] = big[0]              # a long row in any case
        d = rng.normal(size=(moved, 3))
        d /= np.linalg.norm(d, axis=1)[:, None]
        x[who, :3] += (d * 0.7e-3).astype(np.float32)
        ctx.step(torch.from_numpy(x).cuda())
        f, _ = sm.step(x)
        assert np.array_equal(ctx.flags(), f)
        assert f.sum() >= moved * 0.5
        assert np.array_equal(ctx.ref().view(np.int32), sm.ref.view(np.int32))
        pi, pj = ctx.pairs_ij()
        assert np.array_equal(pi, sm.pi) and np.array_equal(pj, sm.pj)
        rows, col = ctx.pairs_csr()      # both sides of every pair
        i = np.repeat(np.arange(n), np.diff(rows))
        assert set(zip(i.tolist(), col.tolist())) == \
            set(zip(pi.tolist(), pj.tolist())) | set(zip(pj.tolist(), pi.tolist()))
    st = ctx.stats()
    assert st["cell_capacity"] >= 512
    assert np.diff(rows).max() > 32
    ctx.close()


@pytest.mark.parametrize("trigger", [1, 2])
@pytest.mark.parametrize("reach", [0, 1, 2])
@pytest.mark.parametrize("n", [1, 33, 6000])
def test_whole_lists_match_the_oracle(orc, trigger, reach, n):
    # every row built anew, a lane to a row (cells of 1 to some 100 spheres)
    lvb = _lvb()
    from oracle.statemachine import OracleLVB
    s, _ = _bed(n, 23)
    pos = s.pos.astype(np.float32)
    ctx = lvb.LVB(torch.from_numpy(pos).cuda(), s.lo, s.hi, lvb.LVB_SKIN_DIAMETER_FACTOR, 0.1,
                  s.dt, trigger, 1.25)
    ctx.set_option(lvb.LVB_OPT_CELL_CAPACITY, 200)
    ctx.set_option(lvb.LVB_OPT_STENCIL_REACH, reach)
    sm = OracleLVB(pos, orc.SKIN_DIAMETER_FACTOR, 0.1, s.dt, ctx.stats()["rnl_max"], trigger)
    rng = np.random.default_rng(n)
    x = pos.copy()
    for _ in range(3):
        x[:, :3] += rng.normal(0.0, 2e-4, size=(n, 3)).astype(np.float32)
        ctx.step(torch.from_numpy(x).cuda())
        sm.step(x)
        pi, pj = ctx.pairs_ij()
        assert np.array_equal(pi, sm.pi) and np.array_equal(pj, sm.pj)
        rows, col = ctx.pairs_csr()
        assert rows[-1] == 2 * len(pi) == len(col)
    assert ctx.stats()["cell_capacity"] >= 200
    ctx.close()
