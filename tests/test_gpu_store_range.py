"""A list whose rows fit 2^31 entries only with the smaller slack: 112M spheres on a
cubic lattice with six partners each want 20 entries a row (2.24e9) at the usual
slack, 16 at the smaller one."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_rows_get_less_slack_where_the_store_needs_it():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.mem_get_info()[0] < 120 << 30:
        pytest.skip("not enough device memory")
    from paper_2208_13770_gb300 import lvb
    m, a = 482, 2e-3
    n = m ** 3
    assert 20 * (n - 6 * m * m) > 2 ** 31 > 17 * n
    i = torch.arange(n, device="cuda")
    pos = torch.empty((n, 4), device="cuda")
    for axis, k in enumerate((i % m, i // m % m, i // (m * m))):
        pos[:, axis] = (k.double() + 0.5) * a
    del i, k
    pos[:, 3] = 1.0e-3
    side = m * a
    # R_NL = 1.1 mm: partners at 2 mm, none at 2.83 mm
    ctx = lvb.LVB(pos, (0.0, 0.0, 0.0), (side, side, side), lvb.LVB_SKIN_DIAMETER_FACTOR, 0.05,
                  1e-6, lvb.LVB_TRIGGER_PARTIAL, 1.25)
    pairs = 3 * m * m * (m - 1)
    assert ctx.stats()["entries"] == 2 * pairs
    pos[12345, 0] += 2.5e-4              # leaves its skin, and its neighbour below in x
    ctx.step(pos)
    assert ctx.sync() == lvb.LVB_OK
    st = ctx.stats()
    assert st["flagged_total"] == 1 and st["entries"] == 2 * (pairs - 1)
    ctx.close()


@pytest.mark.parametrize("n", [1, 700, 30_000])
def test_rounded_rows_take_no_more_memory(n):
    # the store: twice the rows with a slack of half their length and eight, and
    # room for eight more each, whatever the capacities are rounded to
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import numpy as np
    from paper_2208_13770_gb300 import lvb, scenes
    for s in (scenes.packed(n=n, seed=5), scenes.settling(n=n, seed=5, footprint=0.1)):
        ctx = lvb.LVB(torch.from_numpy(s.pos).cuda(), s.lo, s.hi, lvb.LVB_SKIN_DIAMETER_FACTOR, 0.1,
                      s.dt, lvb.LVB_TRIGGER_PARTIAL, s.cell_factor)
        rows = np.diff(ctx.pairs_csr()[0]).astype(np.int64)
        want = 2 * int((rows + 8 + rows // 2).sum()) + 8 * n + 1024
        assert ctx.stats()["row_store_capacity"] == max(want, 4096)
        ctx.close()
