"""Which form the rows take follows how many particles the occupied cells hold,
not how many slots they have: a sparse scene with many slots a cell (one crowded
cell, a growth, LVB_OPT_CELL_CAPACITY) keeps the form for sparse cells, and both
forms give the oracle's list on either side of the line."""
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


def _follow(lvb, orc, s, x, trigger, cell_factor, slots, moved, sigma, steps=4):
    from oracle.statemachine import OracleLVB
    n = len(x)
    ctx = lvb.LVB(torch.from_numpy(x).cuda(), s.lo, s.hi, lvb.LVB_SKIN_DIAMETER_FACTOR, 0.1,
                  s.dt, trigger, cell_factor)
    if slots:
        ctx.set_option(lvb.LVB_OPT_CELL_CAPACITY, slots)
    sm = OracleLVB(x, orc.SKIN_DIAMETER_FACTOR, 0.1, s.dt, ctx.stats()["rnl_max"], trigger)
    rng = np.random.default_rng(n)
    x = x.copy()
    for _ in range(steps):
        who = rng.choice(n, size=min(n, moved), replace=False)
        x[who, :3] += rng.normal(0.0, sigma, size=(len(who), 3)).astype(np.float32)
        ctx.step(torch.from_numpy(x).cuda())
        f, _ = sm.step(x)
        assert np.array_equal(ctx.flags(), f)
        assert np.array_equal(ctx.ref().view(np.int32), sm.ref.view(np.int32))
        pi, pj = ctx.pairs_ij()
        assert np.array_equal(pi, sm.pi) and np.array_equal(pj, sm.pj)
        assert len(ctx.pairs_csr()[1]) == 2 * len(pi)
    ctx.close()


@pytest.mark.parametrize("trigger", [0, 1, 2])
@pytest.mark.parametrize("n,cell_factor", [(11, 4.0), (12, 4.0), (33, 4.0), (700, 2.0),
                                           (700, 2.5), (4000, 3.0), (4000, 4.5)])
def test_forms_on_both_sides_of_the_line(orc, n, cell_factor, trigger):
    # one cell of 11 or 12 or 33; 5.6, 11, 19 and 63 to an occupied cell (7, 16, 23 and 82
    # in the cell of a particle)
    s = scenes.packed(n=n, seed=41)
    _follow(_lvb(), orc, s, s.pos.astype(np.float32), trigger, cell_factor, 0, max(2, n // 5), 3e-4)


@pytest.mark.parametrize("trigger", [0, 2])
def test_one_crowded_cell_in_a_sparse_scene(orc, trigger):
    s = scenes.settling(n=3000, seed=43, footprint=0.03)
    x = s.pos.astype(np.float32)
    near = np.argsort(((x[:, :3] - x[0, :3]) ** 2).sum(1))[:60]     # 60 spheres in one place
    rng = np.random.default_rng(43)
    x[near, :3] = x[0, :3] + rng.uniform(-1e-3, 1e-3, size=(60, 3)).astype(np.float32)
    _follow(_lvb(), orc, s, x, trigger, s.cell_factor, 0, 600, 2e-4)


def test_slots_alone_do_not_change_the_form():
    # a whole list of a sparse scene: with the form for dense cells it takes 3.4
    # times as long, so half as long again lies far from both
    lvb = _lvb()
    s = scenes.settling(n=200_000)
    x = torch.from_numpy(s.pos).cuda()

    def step_ms(slots):
        ctx = lvb.LVB(x, s.lo, s.hi, lvb.LVB_SKIN_DIAMETER_FACTOR, 0.1, s.dt, 2, s.cell_factor)
        if slots:
            ctx.set_option(lvb.LVB_OPT_CELL_CAPACITY, slots)
        times = []
        for _ in range(25):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            ctx.step(x)
            e1.record()
            torch.cuda.synchronize()
            times.append(e0.elapsed_time(e1))
        assert ctx.sync() == lvb.LVB_OK
        assert ctx.stats()["cell_capacity"] >= slots
        ctx.close()
        return float(np.median(times[5:]))

    few, many = step_ms(0), step_ms(512)
    assert many < 1.5 * few, (few, many)
