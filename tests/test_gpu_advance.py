"""dem_advance against the same steps phase by phase.

dem_advance runs its steps in launches that join the forces of a step with
the half-step and check of the next and pass the state between two buffers;
dem_phase runs every phase as a kernel of its own on one buffer.  Both use
the same roundings, so without contacts every array agrees bit for bit at
every count of steps (odd and even: where the state ends differs) and every
size (one block up to 2,048 particles, a last partial warp, several blocks).
With contacts the two contexts' rows may hold their entries in different
orders, which orders each force sum: a sum of at most 12 terms differs by at
most 12 * 2^-24 of the terms, and over the at most 101 steps of 1 us here a
contact's force of up to k_n delta ~ 0.2 N on 1e-5 kg (2e4 m/s^2) leaves
velocities within 101 * 1e-6 * 2e4 * 12 * 2^-24 = 1.5e-6 m/s; positions then
agree to 101 us of that and to one rounding per step of a 0.04 m coordinate
(2^-29 m each): 101 * 2^-29 = 1.9e-7 m at the very most.
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


def _two(lvb, make, steps):
    a, b = lvb.DEM(make()), lvb.DEM(make())
    a.advance(steps)
    for _ in range(steps):
        b.step()
    assert a.sync() == lvb.LVB_OK and b.sync() == lvb.LVB_OK
    sa, sb = a.lvb.stats(), b.lvb.stats()
    assert sa["steps"] == sb["steps"] == steps
    return a, b, sa, sb


@pytest.mark.parametrize("n", [1, 31, 2048, 2049, 6000])
@pytest.mark.parametrize("steps", [1, 2, 3, 100, 101, 203])
def test_free_flight_is_bitwise_the_phases(n, steps):
    lvb = _lvb()

    def make():
        s = scenes.ballistic(n=n, seed=31 + n, phi=0.19)
        s.vel[:, :3] *= 200.0              # fast: walls and list updates within the run
        return s
    a, b, sa, sb = _two(lvb, make, steps)
    for x, y in zip(a.state(), b.state()):
        assert np.array_equal(x, y)
    assert np.array_equal(a.lvb.ref(), b.lvb.ref())
    assert np.array_equal(a.lvb.flags(), b.lvb.flags())
    assert sa["flagged_total"] == sb["flagged_total"]
    pa, pb = a.lvb.pairs_ij(), b.lvb.pairs_ij()
    assert np.array_equal(pa[0], pb[0]) and np.array_equal(pa[1], pb[1])
    a.close()
    b.close()


@pytest.mark.parametrize("n,steps,mu,wall", [(1, 3, 0.0, "box"), (700, 1, 0.0, "box"),
                                             (700, 2, 0.5, "box"), (3000, 101, 0.0, "box"),
                                             (3000, 50, 0.5, "box"), (3000, 37, 0.0, "specular"),
                                             (20_000, 40, 0.5, "box"), (20_000, 41, 0.0, "box")])
def test_contacts_agree_to_the_order_of_the_sums(n, steps, mu, wall):
    lvb = _lvb()

    def make():
        s = scenes.packed(n=n, seed=5, vsigma=0.05)
        s.mu = mu
        s.wall = wall
        return s
    a, b, sa, sb = _two(lvb, make, steps)
    xa, va, aa, sta = a.state()
    xb, vb, ab, stb = b.state()
    assert np.abs(xa - xb).max() <= 1.9e-7
    for p, q in ((va, vb), (sta, stb)):
        assert np.abs(p[:, :3] - q[:, :3]).max() <= 1.5e-6
        assert np.array_equal(p[:, 3], q[:, 3])
    if n > 1:
        assert np.abs(aa[:, :3]).max() > 20.0          # contacts at work
    if mu:
        for p, q in zip(a.rot_state(), b.rot_state()):
            # dw = r F / I dt of the same force differences, 1/I = 2.5 / (m r^2)
            assert np.array_equal(p[:, 3], q[:, 3])
        wa, wb = a.rot_state()[0], b.rot_state()[0]
        assert np.abs(wa[:, :3] - wb[:, :3]).max() <= 2.5 * 1.5e-6 / 1e-3
        assert np.abs(wa[:, :3]).max() > 0
    a.close()
    b.close()


@pytest.mark.parametrize("trigger,early", [(1, 1000), (2, 1000), (0, 700)])
def test_triggers_that_update_more_than_the_flagged(trigger, early):
    # v* of particles that are updated without a violation of their own
    lvb = _lvb()
    out = []
    for graph in (True, False):
        s = scenes.ballistic(n=3000, seed=8)
        s.vel[:, :3] *= 100.0
        dem = lvb.DEM(s, trigger=trigger, skin_kind=lvb.LVB_SKIN_PAPER_KVDT, skin_value=30.0)
        if early < 1000:
            dem.lvb.set_option(lvb.LVB_OPT_EARLY, early)
        if graph:
            dem.advance(64)
        else:
            for _ in range(64):
                dem.step()
        assert dem.sync() == lvb.LVB_OK
        out.append((dem.state(), dem.lvb.ref(), dem.lvb.pairs_ij(), dem.lvb.stats()))
        dem.close()
    (sa, ra, pa, ta), (sb, rb, pb, tb) = out
    assert all(np.array_equal(x, y) for x, y in zip(sa, sb))
    assert np.array_equal(ra, rb)
    assert all(np.array_equal(x, y) for x, y in zip(pa, pb))
    assert ta["updated_total"] == tb["updated_total"] > 3000
