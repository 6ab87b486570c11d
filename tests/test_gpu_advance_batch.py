"""dem_advance on batches of scenes, with drum walls, and with updates deferred to the
rebuild (skin network, rebuild log), against the same steps phase by phase.

The scenes overlap in space, their borders lie inside the chunks of 32 particles
that a warp takes, and something is flagged at most steps of launches of many
steps.  Nobody touches anybody, so every array must be equal bit for bit.
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


def _gas(n, seed, fast=150.0):
    s = scenes.ballistic(n=n, seed=seed, phi=0.19)
    s.vel[:, :3] *= fast
    return s


def _equal(lvb, a, b):
    assert a.sync() == lvb.LVB_OK and b.sync() == lvb.LVB_OK
    for x, y in zip(a.state(), b.state()):
        assert np.array_equal(x, y)
    assert np.array_equal(a.lvb.ref(), b.lvb.ref())
    assert np.array_equal(a.lvb.flags(), b.lvb.flags())
    pa, pb = a.lvb.pairs_ij(), b.lvb.pairs_ij()
    assert np.array_equal(pa[0], pb[0]) and np.array_equal(pa[1], pb[1])
    sa, sb = a.lvb.stats(), b.lvb.stats()
    for key in ("steps", "flagged_total", "updated_total", "rebuild_steps", "entries"):
        assert sa[key] == sb[key], key
    return sa


def _run(dems, calls):
    a, b = dems
    for m in calls:
        a.advance(m)
    for _ in range(sum(calls)):
        b.step()


@pytest.mark.parametrize("sizes", [(33, 700, 1, 65), (2049, 31, 9000, 500), (40, 40)])
@pytest.mark.parametrize("threads,block", [(1024, 0), (512, 1), (256, 0), (256, 1)])
def test_scenes_of_unequal_sizes(sizes, threads, block):
    lvb = _lvb()
    dems = [lvb.DEM([_gas(n, 90 + q) for q, n in enumerate(sizes)]) for _ in range(2)]
    for dem in dems:
        dem.lvb.set_option(lvb.LVB_OPT_BLOCK_THREADS, threads)
        dem.lvb.set_option(lvb.LVB_OPT_COMPACT, block)
    _run(dems, (7, 1, 100, 35))
    st = _equal(lvb, *dems)
    assert st["flagged_total"] > 2 * sum(sizes) and st["rebuild_steps"] > 20
    for dem in dems:
        dem.close()


@pytest.mark.parametrize("trigger", [0, 2])
def test_walls_of_each_scene(trigger):
    # box walls at each scene's own place: forces that need the particle's scene
    lvb = _lvb()
    sizes = (700, 33, 3000)
    make = lambda: [_gas(n, 70 + q) for q, n in enumerate(sizes)]
    dems = []
    for _ in range(2):
        sc = make()
        for s in sc:
            s.wall, s.dt = "box", 1e-6
        dems.append(lvb.DEM(sc, trigger=trigger))
    _run(dems, (3, 120, 77))
    _equal(lvb, *dems)
    hit = np.abs(dems[0].state()[2][:, :3]).max(axis=1) > 100.0
    for lo, hi in zip(dems[0].offsets[:-1], dems[0].offsets[1:]):
        assert hit[lo:hi].any()                            # at a wall in every scene
    for dem in dems:
        dem.close()


@pytest.mark.parametrize("n,steps", [(5000, 101), (20_000, 150)])
def test_drum_walls(n, steps):
    lvb = _lvb()
    dems = []
    for _ in range(2):
        s = scenes.drum(n=n, seed=12, length=0.02, cascade=0.05)
        s.contacts = False
        s.pos[:, [0, 2]] *= np.float32(1.0021)             # the outermost next to the wall
        s.vel[:, :3] += np.random.default_rng(n).normal(0.0, 2.0, size=(n, 3)).astype(np.float32)
        dems.append(lvb.DEM(s))
    _run(dems, (1, steps - 1))
    _equal(lvb, *dems)
    a = dems[0].state()[2]
    assert (np.hypot(a[:, 0], a[:, 2]) > 100.0).any()      # at the drum's wall
    for dem in dems:
        dem.close()


def _network(lvb, horizon):
    rng = np.random.default_rng(4)
    p = (rng.standard_normal(lvb.LVB_MLP_PARAMS) * 0.1).astype(np.float32)
    p[-1] = 1.0
    mu = np.array([1e-2, 1e-5, 0.4, 3, 20, 1.0, 2, 5], np.float32)
    isd = 1.0 / np.array([1e-2, 1e-4, 0.2, 3, 20, 0.1, 2, 5], np.float32)
    return lvb.mlp_weights_device(p, mu, isd, np.array([0.25, 4.0], np.float32), horizon)


@pytest.mark.parametrize("sizes", [(3000,), (700, 33, 2049)])
@pytest.mark.parametrize("learned,log", [(True, False), (False, True), (True, True)])
def test_deferred_updates(sizes, learned, log):
    lvb = _lvb()
    w = _network(lvb, 8.0)
    dems = []
    for _ in range(2):
        sc = [_gas(n, 50 + q) for q, n in enumerate(sizes)]
        kw = dict(skin_kind=lvb.LVB_SKIN_LEARNED, skin_value=0.0, mlp=w) if learned else {}
        dems.append(lvb.DEM(sc if len(sc) > 1 else sc[0], **kw))
        if log:
            dems[-1].lvb.log_enable(10, 200_000)
    _run(dems, (2, 60, 100))
    st = _equal(lvb, *dems)
    assert st["flagged_total"] > sum(sizes)
    if log:
        la, lb = (dem.lvb.log_samples() for dem in dems)
        assert len(la) == len(lb) > sum(sizes)
        assert np.array_equal(la[np.lexsort(la.T)], lb[np.lexsort(lb.T)])
    for dem in dems:
        dem.close()
