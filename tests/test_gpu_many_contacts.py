"""dem_advance where the particles have many contacts: its steps then keep the
forces apart from the half-steps.  With specular walls they always do; else a launch
chooses by a sample of the contacts, taken at the start, after dem_set_state and
every 500 steps: one and a half with partners that lie far away in the arrays, or
with friction three of any kind.

Both forms and the phases use the same roundings, and only the order of a row's
entries, which two contexts need not share, orders a force sum.  So the results are
compared bit for bit where that order cannot matter: squares of spheres, of which
none ever has more than one contact, though two each are so close at the start
that the sample counts them, and packed spheres in one context, whose list stays
as it is between the two runs.
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


def squares(n, mu=0.0, wall="box", seed=3, apart=0.0, shuffled=False):
    """Squares A B C D of spheres of 1 mm, 8 mm apart: A and B (along x) overlap by
    2 um, D above A, C above B and C beside D are 0.04 um from touching.  D and C
    move up, away from each other, A and B down, so those distances only grow, and in
    101 steps of 1 us at up to 8 m/s nobody comes near another square.
    apart: by how much more B and C stand off along x.  shuffled: in no order."""
    rng = np.random.default_rng(seed + n)
    k, w = np.arange(n) // 4, np.arange(n) % 4
    side = int(np.ceil((k[-1] + 1) ** (1 / 3)))
    r, near = 1e-3, 4e-8
    pos = np.zeros((n, 4), np.float32)
    pos[:, 0] = 0.004 + 0.008 * (k % side) + np.choose(w, [0.0, 2 * r - 2e-6, 2 * r + near, 0.0]) \
        + apart * ((w == 1) | (w == 2))
    pos[:, 1] = 0.004 + 0.008 * (k // side % side) + (2 * r + near) * (w >= 2)
    pos[:, 2] = 0.0011 + 0.008 * (k // side // side)
    pos[:, 3] = r
    out, vy = rng.uniform(1.0, 8.0, size=n), rng.uniform(3.0, 8.0, size=n)
    vel = np.zeros((n, 4), np.float32)
    vel[:, 0] = np.choose(w, [0.05 * out, -0.05 * out, out, -out])
    vel[:, 1] = np.where(w >= 2, vy, -0.3 * vy)
    vel[:, 2] = rng.uniform(-4.0, 4.0, size=n)
    s = scenes.packed(n=1)
    if shuffled:
        order = rng.permutation(n)
        pos, vel = pos[order], vel[order]
    s.pos, s.vel, s.mu, s.wall = pos, vel, mu, wall
    s.lo, s.hi = (0.0, 0.0, 0.0), (0.008 * side + 0.002,) * 3
    return s


def equal(lvb, a, b):
    """Every array of two contexts, bit for bit."""
    assert a.sync() == lvb.LVB_OK and b.sync() == lvb.LVB_OK
    for x, y in zip(a.state(), b.state()):
        assert np.array_equal(x, y)
    for x, y in zip(a.rot_state(), b.rot_state()):
        assert np.array_equal(x, y)
    assert np.array_equal(a.lvb.ref(), b.lvb.ref())
    assert np.array_equal(a.lvb.flags(), b.lvb.flags())
    pa, pb = a.lvb.pairs_ij(), b.lvb.pairs_ij()
    assert np.array_equal(pa[0], pb[0]) and np.array_equal(pa[1], pb[1])
    for x, y in zip(a.contact_history(2), b.contact_history(2)):
        assert np.array_equal(x, y)
    sa, sb = a.lvb.stats(), b.lvb.stats()
    for key in ("steps", "flagged_total", "updated_total", "rebuild_steps"):
        assert sa[key] == sb[key], key


def run(dems, calls):
    a, b = dems
    for m in calls:
        a.advance(m)
    for _ in range(sum(calls)):
        b.step()
    return a, b


@pytest.mark.parametrize("mu", [0.0, 0.5])
@pytest.mark.parametrize("n,wall", [(24, "specular"), (2048, "specular"), (2049, "specular"),
                                    (20_000, "specular"), (160_000, "box"), (160_000, "specular")])
@pytest.mark.parametrize("calls", [(1, 1, 2), (40,), (3, 37, 61)])
def test_squares_are_bitwise_the_phases(n, wall, mu, calls):
    # (160,000 in no order: the sample has 1.6 far contacts each)
    lvb = _lvb()
    a, b = [lvb.DEM(squares(n, mu, wall=wall, shuffled=True)) for _ in range(2)]
    assert len(a.contact_forces()[0]) == n // 4
    run((a, b), calls)
    equal(lvb, a, b)
    if sum(calls) > 40:
        assert a.lvb.stats()["flagged_total"] > n // 4
    a.close()
    b.close()


@pytest.mark.parametrize("trigger,kind,early", [(1, 1, 1000), (2, 1, 1000), (0, 2, 1000),
                                                (0, 1, 700)])
@pytest.mark.parametrize("threads", [1024, 256])
def test_triggers_and_rules(trigger, kind, early, threads):
    lvb = _lvb()
    dems = [lvb.DEM(squares(9000, wall="specular"), trigger=trigger, skin_kind=kind,
                    skin_value=0.1 if kind == 1 else 15.0) for _ in range(2)]
    for dem in dems:
        dem.lvb.set_option(lvb.LVB_OPT_BLOCK_THREADS, threads)
        if early < 1000:
            dem.lvb.set_option(lvb.LVB_OPT_EARLY, early)
    a, b = run(dems, (60, 41))
    equal(lvb, a, b)
    assert a.lvb.stats()["updated_total"] > 0
    a.close()
    b.close()


@pytest.mark.parametrize("mu", [0.0, 0.5])
def test_batch_of_squares(mu):
    lvb = _lvb()
    sizes = (700, 3001, 24, 1900)
    dems = [lvb.DEM([squares(n, mu, "specular", seed=q) for q, n in enumerate(sizes)])
            for _ in range(2)]
    a, b = run(dems, (1, 20, 70))
    equal(lvb, a, b)
    assert a.lvb.stats()["flagged_total"] > 1000
    a.close()
    b.close()


@pytest.mark.parametrize("mu", [0.0, 0.5])
@pytest.mark.parametrize("n,apart", [(24, 0.0), (2049, 0.0), (9000, 0.0), (2049, 3e-4)])
def test_specular_walls_with_contacts(n, apart, mu):
    # mirrored at the floor within the run, with many contacts and with few
    lvb = _lvb()
    a, b = [lvb.DEM(squares(n, mu, wall="specular", apart=apart)) for _ in range(2)]
    down = (a.state()[1][:, 2] < -2.0).sum()
    run((a, b), (3, 1, 97))
    equal(lvb, a, b)
    assert (a.state()[1][:, 2] < -2.0).sum() < down        # mirrored
    k = a.lvb.stats()["kernels_executed"]
    a.advance(100)
    assert a.lvb.stats()["kernels_executed"] - k <= 4      # not a launch for every step
    a.close()
    b.close()


@pytest.mark.parametrize("n", [700, 3000, 160_000])
@pytest.mark.parametrize("calls", [(1, 2), (40, 61)])
def test_packed_spheres_in_one_context(n, calls):
    lvb = _lvb()
    s = scenes.packed(n=n, seed=11, vsigma=0.05)
    dem = lvb.DEM(s)
    x, v, a, _ = dem.state()
    assert 2 * len(dem.contact_forces()[0]) >= 1.6 * n
    for m in calls:
        dem.advance(m)
    assert dem.sync() == lvb.LVB_OK
    first = dem.state()
    dem.set_state(x, v, a)
    for _ in range(sum(calls)):
        dem.step()
    assert dem.sync() == lvb.LVB_OK
    assert dem.lvb.stats()["flagged_total"] == 0           # the same list all along
    for p, q in zip(first, dem.state()):
        assert np.array_equal(p, q)
    assert np.abs(first[2][:, :3]).max() > 20.0            # contacts at work
    dem.close()


def test_state_set_later_is_sampled():
    # squares pulled apart, then pushed together: both forms in one context
    lvb = _lvb()
    out = []
    for joined in (True, False):
        s, together = (squares(160_000, apart=d, shuffled=True) for d in (3e-4, 0.0))
        dem = lvb.DEM(s)
        assert len(dem.contact_forces()[0]) == 0
        steps = dem.advance if joined else (lambda m: [dem.step() for _ in range(m)])
        steps(10)
        dem.set_state(together.pos, together.vel, np.zeros_like(s.vel))
        steps(30)
        steps(31)
        out.append(dem)
    equal(lvb, *out)
    for dem in out:
        dem.close()


def test_no_slower_than_the_phases():
    # 1M packed spheres with friction in no order: joined passes take a fifth longer
    # than the three phases, this form a little less
    lvb = _lvb()
    s = scenes.packed(n=1_000_000, seed=11, vsigma=0.05)
    s.mu = 0.5
    dem = lvb.DEM(s)

    def ms(f):
        times = []
        for _ in range(7):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            f()
            e1.record()
            torch.cuda.synchronize()
            times.append(e0.elapsed_time(e1))
        return float(np.median(times[2:]))

    joined = ms(lambda: dem.advance(20))
    phases = ms(lambda: [dem.step() for _ in range(20)])
    assert dem.sync() == lvb.LVB_OK
    dem.close()
    assert joined < 1.05 * phases, (joined, phases)
