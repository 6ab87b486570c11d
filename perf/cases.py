"""Timed cases: what a program that uses this library has it do.

Seven kinds, each through the public binding (``paper_2208_13770_gb300.lvb``):

``advance``  a DEM run that advances by some steps per call (``DEM.advance``)
             and reads the state arrays in place: a small ballistic gas, a
             settling box, a batch of settling boxes, a rotating drum with
             the paper's skin rule, with the learned skin, with friction.
``solver``   a solver with its own integrator: one ``lvb_step`` at its new
             positions, then the contacts of the list in its own buffers.
``broad``    the broad phase alone over a batch of boxes (``lvb_step`` at
             positions that live on the GPU), then the flags and the
             reference state.
``host``     a host program: positions in pinned memory, flags back
             (``lvb_step_host``).
``rebuild``  no Verlet buffer: the whole list built anew at every call
             (``LVB_TRIGGER_ALWAYS``) and exported as a CSR.
``clumps``   the narrow phase of multi-sphere clumps on the list.
``train``    training of the skin network on rebuild-log samples.

Every state starts in the steady state of a run: a particle's reference
position lies a uniform fraction of its skin behind it, so that every step
flags a few particles, as it does after the first thousands of steps.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2208_13770_gb300 import lvb, scenes

DT = 1e-6            # time step of the contact scenes [s]
SWELL = 1.0012       # radii over the drum's lattice: contacts of one or two micrometres
K_PAPER = 200.0      # the paper's default K
K_LEARNED = 400.0    # steps of travel that the learned skin is a factor of
JUMP = 3e-4          # fraction of the particles that outrun their skin at a step
NOBODY = 1 << 24     # an id above every clump's: unused places of its list come last
SNAPS = 6            # positions that a stepping case cycles through


def listed():
    return [
        # smallest run: 2,000 spheres in free flight, where launches and latency count
        {"name": "ballistic_2k", "kind": "advance", "scene": "ballistic", "n": 2000,
         "skin": "diameter", "mu": 0.0, "steps": 100},
        # one closed box of polydisperse spheres under gravity
        {"name": "settling_200k", "kind": "advance", "scene": "settling", "n": 200_000,
         "skin": "diameter", "mu": 0.0, "steps": 100},
        # the parameter study: 512 boxes of 1,000 to 50,000 spheres advanced together
        {"name": "batch_512", "kind": "advance", "scene": "batch", "n": 512,
         "skin": "diameter", "mu": 0.0, "steps": 100},
        # a large dense bed in a rotating drum under the paper's rule, skin = K |v| dt,
        # in short calls as a coupled solver makes them (beds keep to 24 steps a call: over
        # more, the rounding of the positions is what their forces show)
        {"name": "drum_2m_paper", "kind": "advance", "scene": "drum", "n": 2_000_000,
         "skin": "paper", "mu": 0.0, "steps": 20},
        # the same with the skin network
        {"name": "drum_1m_learned", "kind": "advance", "scene": "drum", "n": 1_000_000,
         "skin": "learned", "mu": 0.0, "steps": 20},
        # friction: tangential springs kept with the list's entries
        {"name": "drum_1m_friction", "kind": "advance", "scene": "drum", "n": 1_000_000,
         "skin": "diameter", "mu": 0.5, "steps": 20},
        # a solver of its own: one step of the list and its contacts, packed spheres
        {"name": "solver_200k", "kind": "solver", "n": 200_000},
        # the broad phase alone over the largest batch
        {"name": "broad_512", "kind": "broad", "n": 512, "passes": 6},
        # a solver whose particles live in host memory
        {"name": "host_500k", "kind": "host", "n": 500_000, "passes": 6},
        # a list without a buffer, and list building as such
        {"name": "rebuild_1m", "kind": "rebuild", "n": 1_000_000},
        # clumps of one to four spheres
        {"name": "clumps_400k", "kind": "clumps", "n": 400_000},
        # the skin network's training, the batch size of the benchmark
        {"name": "train_60k", "kind": "train", "n": 60_000, "batch": 512, "epochs": 2},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["ballistic", "settling", "batch", "drum", "friction", "solver", "broad",
                       "host", "rebuild", "clumps", "train"])
    if kind == "ballistic":
        return {"kind": "advance", "scene": "ballistic", "n": _log_int(rng, 500, 40_000),
                "skin": "diameter", "mu": 0.0, "steps": _log_int(rng, 20, 300)}
    if kind == "settling":
        return {"kind": "advance", "scene": "settling", "n": _log_int(rng, 5000, 400_000),
                "skin": rng.choice(["diameter", "paper"]), "mu": 0.0,
                "steps": _log_int(rng, 10, 200)}
    if kind == "batch":
        return {"kind": "advance", "scene": "batch", "n": _log_int(rng, 4, 400),
                "skin": "diameter", "mu": 0.0, "steps": _log_int(rng, 10, 100)}
    if kind == "drum":
        return {"kind": "advance", "scene": "drum", "n": _log_int(rng, 100_000, 1_500_000),
                "skin": rng.choice(["diameter", "paper", "learned"]), "mu": 0.0,
                "steps": _log_int(rng, 5, 24)}
    if kind == "friction":
        return {"kind": "advance", "scene": "drum", "n": _log_int(rng, 100_000, 1_000_000),
                "skin": "diameter", "mu": round(rng.uniform(0.2, 0.8), 2),
                "steps": _log_int(rng, 5, 24)}
    if kind == "solver":
        return {"kind": "solver", "n": _log_int(rng, 3000, 500_000)}
    if kind == "broad":
        return {"kind": "broad", "n": _log_int(rng, 4, 400), "passes": rng.randint(1, 6)}
    if kind == "host":
        return {"kind": "host", "n": _log_int(rng, 20_000, 1_000_000),
                "passes": rng.randint(1, 6)}
    if kind == "rebuild":
        return {"kind": "rebuild", "n": _log_int(rng, 30_000, 1_000_000)}
    if kind == "clumps":
        return {"kind": "clumps", "n": _log_int(rng, 5000, 400_000)}
    return {"kind": "train", "n": _log_int(rng, 2000, 100_000), "batch": _log_int(rng, 64, 2048),
            "epochs": 1}


# ----------------------------------------------------------------- scenes
def _drum(n, seed):
    s = scenes.drum(n=n, seed=seed, length=max(0.1 * n / 1e6, 0.02), tilt_deg=30.0, cascade=0.05)
    s.pos[:, 3] *= np.float32(SWELL)   # the lattice only just touches: press the bed together
    return s


def _scenes(name, n, seed):
    """The scenes of a case (a list of one unless it is a batch)."""
    seed = scenes.SEED_BASE + 1000 * (seed + 1)
    if name == "ballistic":
        return [scenes.ballistic(n=n, seed=seed)]
    if name == "settling":
        fp = max(0.15 * math.sqrt(n / 200_000.0), 0.03)
        return [scenes.settling(n=n, seed=seed, footprint=fp)]
    if name == "batch":                # the sizes of the study, other spheres for other seeds
        out = []
        for k, ns in enumerate(scenes.batch_sizes(n)):
            fp = max(0.15 * math.sqrt(ns / 200_000.0) * 1.6, 0.03)
            out.append(scenes.settling(int(ns), seed=seed * 1000 + k, footprint=fp))
        return out
    if name == "drum":
        return [_drum(n, seed)]
    raise ValueError(name)


def _cap(s, cell_factor):
    """The largest R_NL = r + skin of a scene's context (half a cell edge)."""
    L = cell_factor * 2.0 * float(s.pos[:, 3].max()) * (1.0 + 1.0 / 128.0)
    L = max(L, max(h - l for l, h in zip(s.lo, s.hi)) / 2048.0)
    return 0.5 * L * (1.0 - 1.0 / 256.0)


def _skins(s, skin):
    """Skin of every particle of a scene under a rule, capped as the library caps it."""
    r = s.pos[:, 3].astype(np.float64)
    if skin == "diameter":
        want = 0.2 * r
    else:
        k = K_PAPER if skin == "paper" else 0.5 * K_LEARNED
        want = k * s.dt * np.linalg.norm(s.vel[:, :3].astype(np.float64), axis=1)
    return np.minimum(want, np.maximum(_cap(s, s.cell_factor) - r, 0.0)) * (1.0 - 1e-6)


def _behind(s, skin, rng):
    """Reference positions a uniform fraction of the skin behind the positions."""
    v = s.vel[:, :3].astype(np.float64)
    speed = np.maximum(np.linalg.norm(v, axis=1), 1e-30)
    back = rng.uniform(0.0, 0.999, s.n) * _skins(s, skin) / speed
    ref = s.pos.copy()
    ref[:, :3] = s.pos[:, :3] - v * back[:, None]
    return ref


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


class _View:
    """A context's own device array of float4 records, without a copy."""

    def __init__(self, owner, ptr, n):
        self.owner = owner             # the array lives as long as its context
        self.__cuda_array_interface__ = {"shape": (n, 4), "typestr": "<f4",
                                         "data": (ptr, False), "version": 2}


def _network(rng):
    """Packed weights of a small skin network in the travel form."""
    p = (rng.standard_normal(lvb.LVB_MLP_PARAMS) * 0.1).astype(np.float32)
    p[-1] = 1.0                        # the output's bias: about the rule at K_LEARNED
    mu = np.array([1e-4, 1e-5, 0.4, 6, 100, 1.0, 8, 20], np.float32)
    isd = 1.0 / np.array([1e-4, 1e-4, 0.2, 4, 100, 0.1, 6, 20], np.float32)
    return lvb.mlp_weights_device(p, mu, isd, np.array([0.25, 4.0], np.float32), K_LEARNED)


# ------------------------------------------------------------------ advance
def _advance_inputs(case, seed):
    sc = _scenes(case["scene"], case["n"], seed)
    rng = np.random.default_rng([seed, 77])
    refs = [_behind(s, case["skin"], rng) for s in sc]
    pos = np.concatenate([s.pos for s in sc])
    vel = np.concatenate([s.vel for s in sc])
    acc = np.zeros_like(vel)
    acc[:, :3] = sc[0].gravity
    return sc, refs, pos, vel, acc, rng


def _prepare_advance(case, seed):
    sc, refs, pos, vel, acc, rng = _advance_inputs(case, seed)
    for s, ref in zip(sc, refs):
        s.pos = ref
        s.mu = case["mu"]
    kinds = {"diameter": (lvb.LVB_SKIN_DIAMETER_FACTOR, 0.1),
             "paper": (lvb.LVB_SKIN_PAPER_KVDT, K_PAPER), "learned": (lvb.LVB_SKIN_LEARNED, 0.0)}
    kind, value = kinds[case["skin"]]
    mlp = _network(rng) if case["skin"] == "learned" else None
    dem = lvb.DEM(sc if case["scene"] == "batch" else sc[0], skin_kind=kind, skin_value=value,
                  mlp=mlp)
    x, v, a = _dev(pos), _dev(vel), _dev(acc)
    lvb.dem_set_state(dem.ctx, x.data_ptr(), v.data_ptr(), a.data_ptr())
    views = [torch.as_tensor(_View(dem, p, dem.n), device="cuda")
             for p in lvb.dem_device_state(dem.ctx)]
    return {"kind": "advance", "dem": dem, "steps": case["steps"], "views": views}


def _run_advance(st):
    st["dem"].advance(st["steps"])
    x, v, a, vs = st["views"]          # v.w and vstar.w hold 1 / m
    return {"x": x, "v": v[:, :3], "a": a[:, :3], "vstar": vs[:, :3]}


# --------------------------------------------- stepping on given positions
def _snapshots(s_pos, skin, rng, count):
    """Positions of `count` steps: everyone near a base position (within half
    the skin), and at each step another few past their skin."""
    n = len(s_pos)
    x = torch.empty((count, n, 4), dtype=torch.float32, device="cuda")
    base = _dev(s_pos)
    sk = _dev(skin.astype(np.float32))
    gen = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 31)))
    few = max(2, int(round(JUMP * n)))
    for k in range(count):
        d = torch.randn((n, 3), generator=gen, device="cuda")
        d /= d.norm(dim=1, keepdim=True).clamp_min(1e-6)
        f = 0.05 + 0.3 * torch.rand((n,), generator=gen, device="cuda")
        far = torch.randint(0, n, (few,), generator=gen, device="cuda")
        f[far] = 1.6
        x[k] = base
        x[k, :, :3] += d * (f * sk)[:, None]
    return x


def _stepping_inputs(case, seed):
    """(scenes, positions of the steps on the GPU, reference state on the GPU)"""
    rng = np.random.default_rng([seed, 78])
    if case["kind"] == "broad":
        sc = _scenes("batch", case["n"], seed)
    elif case["kind"] == "host":
        sc = _scenes("settling", case["n"], seed)
    elif case["kind"] == "rebuild":
        sc = [_drum(case["n"], scenes.SEED_BASE + 1000 * (seed + 1))]
    else:
        sc = [scenes.packed(n=case["n"], seed=scenes.SEED_BASE + 1000 * (seed + 1))]
    skin = np.concatenate([_skins(s, "diameter") for s in sc])
    pos = np.concatenate([s.pos for s in sc])
    if case["kind"] == "solver":
        skin_move = 0.02 * skin        # resting spheres: they rattle by micrometres
    else:
        skin_move = skin
    count = 2 if case["kind"] == "rebuild" else SNAPS
    x = _snapshots(pos, skin_move, rng, count)
    if case["kind"] == "solver":       # the few that outrun their skin do so by a slide along x
        n = len(pos)
        gen = torch.Generator(device="cuda").manual_seed(seed + 5)
        few = max(2, int(round(JUMP * n)))
        for k in range(count):
            far = torch.randint(0, n, (few,), generator=gen, device="cuda")
            x[k, far, 0] += 1.2 * _dev(skin.astype(np.float32))[far]
    ref = _dev(pos)
    ref[:, 3] = _dev(skin.astype(np.float32))
    return sc, x, ref


def _prepare_stepping(case, seed):
    sc, x, ref = _stepping_inputs(case, seed)
    kind = case["kind"]
    n = x.shape[1]
    trigger = lvb.LVB_TRIGGER_ALWAYS if kind == "rebuild" else lvb.LVB_TRIGGER_PARTIAL
    args = dict(skin_kind=lvb.LVB_SKIN_DIAMETER_FACTOR, skin_value=0.1, dt=DT, trigger=trigger,
                cell_factor=sc[0].cell_factor, ref=ref)
    if len(sc) > 1:
        off = np.concatenate([[0], np.cumsum([s.n for s in sc])]).astype(np.int64)
        ctx = lvb.LVB(x[0], [s.lo for s in sc], [s.hi for s in sc], offsets=off, **args)
    else:
        ctx = lvb.LVB(x[0], sc[0].lo, sc[0].hi, **args)
    st = {"kind": kind, "ctx": ctx, "x": x, "k": 0, "passes": case.get("passes", 1), "n": n}
    words = (n + 31) // 32
    if kind == "host":
        st["xh"] = [t.cpu().pin_memory() for t in x]
        st["bits"] = [torch.zeros(words, dtype=torch.int32).pin_memory()
                      for _ in range(st["passes"])]
        st["nf"] = torch.zeros(st["passes"], dtype=torch.int32).pin_memory()
        st["x"] = None
        return st
    st["bits"] = torch.zeros(words, dtype=torch.int32, device="cuda")
    if kind == "broad":
        st["ref"] = torch.zeros((n, 4), device="cuda")
    elif kind == "rebuild":
        st["rows"] = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
        st["col"] = torch.zeros(16 * n + 1024, dtype=torch.int32, device="cuda")
        st["ref"] = torch.zeros((n, 4), device="cuda")
    else:
        cap = _contact_room(n)
        st["ci"], st["cj"] = (torch.zeros(cap, dtype=torch.int32, device="cuda")
                              for _ in range(2))
        st["delta"] = torch.zeros(cap, device="cuda")
    return st


def _contact_room(n):
    return 3 * n + 1024


def _padded(t, room):
    """A list of contacts' values in a buffer of `room` entries, as the call leaves it."""
    out = torch.zeros(room, dtype=t.dtype, device=t.device)
    out[:len(t)] = t
    return out


def _ok(rc, what):
    if rc != lvb.LVB_OK:
        raise lvb.LVBError(rc, what)


def _run_stepping(st):
    ctx, kind, x = st["ctx"], st["kind"], st["x"]
    m = ctypes.c_int64(0)
    if kind == "host":
        for p in range(st["passes"]):
            ctx.step_host(st["xh"][st["k"] % SNAPS], bits=st["bits"][p],
                          n_flagged=st["nf"][p:p + 1])
            st["k"] += 1
        _ok(ctx.sync(), "lvb_sync")
        return {"bits": st["bits"], "nf": st["nf"]}
    for _ in range(st["passes"]):
        ctx.step(x[st["k"] % len(x)])
        st["k"] += 1
    if kind == "rebuild":
        _ok(lvb.lvb_get_pairs(ctx.ctx, st["rows"].data_ptr(), st["col"].data_ptr(),
                              st["col"].numel(), ctypes.byref(m)), "lvb_get_pairs")
        _ok(lvb.lvb_get_ref(ctx.ctx, st["ref"].data_ptr()), "lvb_get_ref")
        return {"rows": st["rows"], "col": st["col"], "entries": m.value, "ref": st["ref"]}
    _ok(lvb.lvb_get_flags(ctx.ctx, st["bits"].data_ptr(), ctypes.byref(m)), "lvb_get_flags")
    if kind == "broad":
        _ok(lvb.lvb_get_ref(ctx.ctx, st["ref"].data_ptr()), "lvb_get_ref")
        return {"bits": st["bits"], "ref": st["ref"]}
    at = x[(st["k"] - 1) % len(x)]
    _ok(lvb.lvb_get_contacts(ctx.ctx, at.data_ptr(), st["ci"].data_ptr(), st["cj"].data_ptr(),
                             st["delta"].data_ptr(), st["ci"].numel(), ctypes.byref(m)),
        "lvb_get_contacts")
    return {"bits": st["bits"], "contacts": m.value, "ci": st["ci"], "cj": st["cj"],
            "delta": st["delta"]}


# ------------------------------------------------------------------- clumps
def _clump_inputs(case, seed):
    n = case["n"]
    rng = np.random.default_rng([seed, 79])
    k = rng.integers(1, 5, size=n)
    off = np.concatenate([[0], np.cumsum(k)]).astype(np.int32)
    m = int(off[-1])
    sub = np.zeros((m, 4), np.float32)
    sub[:, :3] = rng.normal(0, 0.5e-3, size=(m, 3))
    sub[:, 3] = rng.uniform(0.3e-3, 0.8e-3, size=m)
    ext = np.linalg.norm(sub[:, :3].astype(np.float64), axis=1) + sub[:, 3]
    R = np.maximum.reduceat(ext, off[:-1])
    R = (R / (1.0 - 2.0 ** -12) * (1.0 + 1e-6)).astype(np.float32)
    spacing = 1.6 * float(np.median(R))   # neighbours' bounding spheres overlap
    side = int(np.ceil(n ** (1 / 3)))
    idx = rng.permutation(side ** 3)[:n]
    c = np.stack([idx % side, (idx // side) % side, idx // side ** 2], 1) * spacing
    pos = np.zeros((n, 4), np.float32)
    pos[:, :3] = c + rng.uniform(-0.05, 0.05, size=(n, 3)) * spacing
    pos[:, 3] = R
    q = rng.normal(size=(n, 4))
    q = (q / np.linalg.norm(q, axis=1, keepdims=True)).astype(np.float32)
    pad = 2.0 * float(R.max())
    return pos, q, off, sub, (-pad,) * 3, (side * spacing + pad,) * 3


def _clump_room(n):
    return n // 2 + 1024


def _prepare_clumps(case, seed):
    pos, q, off, sub, lo, hi = _clump_inputs(case, seed)
    x = _dev(pos)
    ctx = lvb.LVB(x, lo, hi, lvb.LVB_SKIN_DIAMETER_FACTOR, 0.1, 1e-5, lvb.LVB_TRIGGER_PARTIAL,
                  1.25)
    room = _clump_room(case["n"])
    outs = [torch.full((room,), NOBODY, dtype=torch.int32, device="cuda") for _ in range(4)]
    outs.append(torch.zeros(room, device="cuda"))
    return {"kind": "clumps", "ctx": ctx, "in": (x, _dev(q), _dev(off), _dev(sub)), "out": outs}


def _run_clumps(st):
    m = st["ctx"].clump_contacts_into(*st["in"], *st["out"])
    ci, ca, cj, cb, delta = st["out"]
    # the call lists them in no particular order: ordered here by (i, a, j, b)
    key = ((ci.long() * 64 + ca) << 32) | (cj.long() * 64 + cb)
    key, order = torch.sort(key)
    return {"contacts": m, "key": key, "delta": delta[order]}


# -------------------------------------------------------------------- train
def _train_inputs(case, seed):
    """Samples like a rebuild log's in the travel form: eight features and
    the displacement in units of the particle's travel."""
    n = case["n"]
    rng = np.random.default_rng([seed, 80])
    s = np.zeros((n, 9), np.float32)
    speed = np.exp(rng.normal(math.log(1e-4), 0.7, n))
    s[:, 0] = speed
    s[:, 1] = np.abs(rng.normal(0, 2e-5, n))
    s[:, 2] = rng.uniform(0.15, 0.75, n)
    s[:, 3] = rng.poisson(6, n)
    s[:, 4] = np.floor(rng.exponential(300, n))
    s[:, 5] = 1.0 + np.abs(rng.normal(0, 0.01, n))
    s[:, 6] = rng.poisson(8, n)
    s[:, 7] = rng.uniform(0, 60, n)
    y = 2.0 * (1.0 - 0.4 * np.exp(-s[:, 3] / 4.0)) + 0.1 * (s[:, 1] / 2e-5)
    s[:, 8] = np.minimum(y * np.exp(rng.normal(0, 0.05, n)), 4.0)
    p0 = (rng.standard_normal(lvb.LVB_MLP_PARAMS) * 0.1).astype(np.float32)
    return s, p0


def _prepare_train(case, seed):
    s, p0 = _train_inputs(case, seed)
    return {"kind": "train", "samples": _dev(s), "p0": p0, "batch": case["batch"],
            "epochs": case["epochs"], "seed": seed}


def _run_train(st):
    yr = np.zeros(2, np.float32)
    p, mu, isd, losses = lvb.mlp_train(st["samples"], epochs=st["epochs"], batch=st["batch"],
                                       lr=3e-3, seed=st["seed"], params0=st["p0"],
                                       y_range_out=yr)
    return {"params": p, "mu": mu, "isd": isd, "losses": losses, "y_range": yr}


# ------------------------------------------------------------------ contract
def prepare(case, seed):
    kind = case["kind"]
    if kind == "advance":
        return _prepare_advance(case, seed)
    if kind == "clumps":
        return _prepare_clumps(case, seed)
    if kind == "train":
        return _prepare_train(case, seed)
    return _prepare_stepping(case, seed)


def run(state):
    kind = state["kind"]
    if kind == "advance":
        return _run_advance(state)
    if kind == "clumps":
        return _run_clumps(state)
    if kind == "train":
        return _run_train(state)
    return _run_stepping(state)


def _particles(case):
    if case["kind"] == "broad" or case.get("scene") == "batch":
        return 12_200 * case["n"]      # mean of the log-uniform box sizes
    return case["n"]


def work(case):
    """Bytes: state records of 16 bytes, list entries of 4; flops: the
    arithmetic of the formulas.  List lengths are those of the scenes."""
    n = _particles(case)
    kind = case["kind"]
    if kind == "advance":
        # a step reads x, v, a and the reference state and writes x, v, a; it
        # reads the list; friction adds rotation and a spring per contact
        row = {"ballistic": 1.5, "settling": 1.0, "batch": 1.0, "drum": 6.0}[case["scene"]]
        if case["scene"] == "ballistic":
            row = 0.0                  # free flight: the list is kept, not read
        fric = case["mu"] > 0
        per = 112 + 4 * row + (64 + 2 * 16 * 2.0 if fric else 0)
        return {"bytes": float(n * per * case["steps"]),
                "flops": float(n * (40 + row * (70 if fric else 20)) * case["steps"])}
    if kind == "broad":
        return {"bytes": float(n * (32 * case["passes"] + 32)),
                "flops": float(n * 9 * case["passes"])}
    if kind == "host":
        return {"bytes": float(n * 48 * case["passes"]), "flops": float(n * 9 * case["passes"])}
    if kind == "solver":
        return {"bytes": float(n * (32 + 16 + 6 * 4 + 1.5 * 12)), "flops": float(n * (9 + 6 * 12))}
    if kind == "rebuild":
        # positions in, reference states out, the list out as a CSR
        return {"bytes": float(n * (16 + 16 + 16 + 4 + 4 * 6)), "flops": float(n * 27 * 4 * 10)}
    if kind == "clumps":
        # bounds, quaternions, spheres and the list in, the contacts out
        return {"bytes": float(n * (16 + 16 + 4 + 2.5 * 16 + 14.5 * 4 + 0.2 * 20)),
                "flops": float(n * (7.25 * 6.25 * 12 + 2.5 * 18))}
    per = 2 * (8 * 32 + 32 * 32 + 32) * 3   # forward, and backward twice that
    return {"bytes": float(case["epochs"] * n * 36), "flops": float(case["epochs"] * n * per)}


# ------------------------------------------------------------- 64-bit values
def _f64(a):
    t = torch.from_numpy(np.ascontiguousarray(a)) if isinstance(a, np.ndarray) else a
    t = t.to(torch.float64)
    return t.cuda() if torch.cuda.is_available() else t


def _close_pairs(x, r, scene, reach):
    """Pairs i < j of the same scene with |x_i - x_j| < r_i + r_j + reach."""
    edge = 2.0 * float(r.max()) + reach
    lo = x.min(dim=0).values
    c = ((x - lo) / edge).floor().long()
    dim = c.max(dim=0).values + 3      # a free cell on every side
    key = (((scene * dim[2] + c[:, 2] + 1) * dim[1]) + c[:, 1] + 1) * dim[0] + c[:, 0] + 1
    key, order = torch.sort(key)
    out = []
    n = len(x)
    idx = torch.arange(n, device=x.device)
    half = [(dx, dy, dz) for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)
            if (dz, dy, dx) >= (0, 0, 0)]
    for dx, dy, dz in half:
        other = key + (dz * dim[1] + dy) * dim[0] + dx
        a = torch.searchsorted(key, other)
        b = torch.searchsorted(key, other, right=True)
        if (dx, dy, dz) == (0, 0, 0):
            a = idx + 1
        cnt = (b - a).clamp_min(0)
        ends = torch.cumsum(cnt, 0)
        s0 = 0
        while s0 < n:                  # slices of at most about 40 million candidates
            before = int(ends[s0 - 1]) if s0 else 0
            s1 = max(s0 + 1, int(torch.searchsorted(ends, before + 40_000_000, right=True)))
            m = cnt[s0:s1]
            p = torch.repeat_interleave(idx[s0:s1], m)
            first = torch.repeat_interleave(torch.cumsum(m, 0) - m, m)
            q = torch.repeat_interleave(a[s0:s1], m) + \
                torch.arange(len(p), device=x.device) - first
            i, j = order[p], order[q]
            d2 = ((x[i] - x[j]) ** 2).sum(1)
            ok = d2 < (r[i] + r[j] + reach) ** 2
            out.append(torch.stack([torch.minimum(i[ok], j[ok]), torch.maximum(i[ok], j[ok])]))
            s0 = s1
    return torch.cat(out, 1)


def _dot(a, b):
    return (a * b).sum(1, keepdim=True)


def _exact_advance(case, seed):
    sc, _, pos, vel, acc, _ = _advance_inputs(case, seed)
    s = sc[0]
    dt = float(np.float32(s.dt))
    P, V, A = _f64(pos), _f64(vel), _f64(acc)
    x, r, v, a = P[:, :3].clone(), P[:, 3:4], V[:, :3].clone(), A[:, :3].clone()
    sizes = torch.tensor([q.n for q in sc], device=x.device)
    scene = torch.repeat_interleave(torch.arange(len(sc), device=x.device), sizes)
    lo = _f64(np.array([q.lo for q in sc], np.float32))[scene]
    hi = _f64(np.array([q.hi for q in sc], np.float32))[scene]
    kn = float(np.float32(s.kn))
    le = math.log(float(np.float32(s.restitution)))
    two_zeta = 2.0 * (-le / math.sqrt(math.pi ** 2 + le * le))
    g = _f64(np.array(s.gravity, np.float32))
    mass = float(np.float32(s.rho)) * (4.0 / 3.0) * math.pi * r ** 3
    im = 1.0 / mass
    fric = case["mu"] > 0
    mu, kt = float(np.float32(case["mu"])), float(np.float32(s.kt_ratio)) * kn
    gt = float(np.float32(s.gt_ratio))
    w, al = torch.zeros_like(x), torch.zeros_like(x)
    inertia = 0.4 * mass * r * r
    steps = case["steps"]
    if s.contacts:
        t = dt * steps                 # nobody comes closer than this in the call
        far = 2.0 * (float(v.norm(dim=1).max()) + 0.02 + 20.0 * t) * t
        i, j = _close_pairs(x, r[:, 0], scene, far)
        if fric:
            spring = torch.zeros((len(i), 3), dtype=torch.float64, device=x.device)
    vs = v
    for _ in range(steps):
        x = x + v * dt + a * (0.5 * dt * dt)
        vs = v + a * dt
        if s.wall == "specular":
            for bound, beyond in ((lo + r, x < lo + r), (hi - r, x > hi - r)):
                x = torch.where(beyond, 2.0 * bound - x, x)
                v = torch.where(beyond, -v, v)
                vs = torch.where(beyond, -vs, vs)
        F, T = torch.zeros_like(x), torch.zeros_like(x)
        ws = w + al * dt
        if s.contacts:
            near = ((x[i] - x[j]) ** 2).sum(1, keepdim=True) < (r[i] + r[j]) ** 2
            hit = near[:, 0].nonzero()[:, 0]
            if fric:
                spring[~near[:, 0]] = 0.0
            p, q = i[hit], j[hit]
            d = x[p] - x[q]
            dist = d.norm(dim=1, keepdim=True)
            n = d / dist
            meff = 1.0 / (im[p] + im[q])
            rel = vs[p] - vs[q]
            gam = two_zeta * torch.sqrt(meff * kn)
            fn = kn * (r[p] + r[q] - dist) - gam * _dot(rel, n)
            f = fn * n
            if fric:
                u = rel - torch.cross(r[p] * ws[p] + r[q] * ws[q], n, dim=1)
                ut = u - _dot(u, n) * n
                h = spring[hit]
                h = h - _dot(h, n) * n + ut * dt
                ft = -kt * h - gt * gam * ut
                size = ft.norm(dim=1, keepdim=True)
                most = mu * fn.clamp_min(0.0)
                slide = size > most
                ft = torch.where(slide, ft * (most / size.clamp_min(1e-300)), ft)
                h = torch.where(slide, -(ft + gt * gam * ut) / kt, h)
                spring[hit] = h
                f = f + ft
                turn = torch.cross(n, ft, dim=1)
                T.index_add_(0, p, -r[p] * turn)
                T.index_add_(0, q, -r[q] * turn)
            F.index_add_(0, p, f)
            F.index_add_(0, q, -f)
        if s.wall in ("box", "drum"):
            gw = two_zeta * torch.sqrt(mass * kn)
            for k in ((0, 1, 2) if s.wall == "box" else (1,)):
                for sign, gap in ((1.0, x[:, k:k + 1] - lo[:, k:k + 1]),
                                  (-1.0, hi[:, k:k + 1] - x[:, k:k + 1])):
                    over = r - gap
                    f = kn * over - gw * sign * vs[:, k:k + 1]
                    F[:, k:k + 1] += torch.where(over > 0, sign * f, torch.zeros_like(f))
            if s.wall == "drum":
                cx, cz, R = (float(np.float32(c)) for c in s.drum[:3])
                d = torch.cat([x[:, 0:1] - cx, torch.zeros_like(r), x[:, 2:3] - cz], 1)
                rho = d.norm(dim=1, keepdim=True)
                n = -d / rho.clamp_min(1e-300)
                over = r + rho - R
                f = kn * over - gw * _dot(vs, n)
                F += torch.where(over > 0, f * n, torch.zeros_like(n))
        new = F * im + g
        v = v + (a + new) * (0.5 * dt)
        a = new
        if fric:
            aln = T / inertia
            w = w + (al + aln) * (0.5 * dt)
            al = aln
    return {"x": torch.cat([x, r], 1), "v": v, "a": a, "vstar": vs}


def _sq32(a, b):
    """|a - b|^2 in binary32, each operation rounded."""
    d = a - b
    return (d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2]


def _exact_stepping(case, seed):
    kind = case["kind"]
    sc, x, ref = _stepping_inputs(case, seed)
    if kind == "host":
        return None                    # flags only: whole numbers
    if kind == "solver":
        at = x[0]
        p = _f64(at)
        zero = torch.zeros(len(p), dtype=torch.int64, device=p.device)
        i, j = _close_pairs(p[:, :3], p[:, 3], zero, 1e-6)
        # which pairs are contacts, binary32 decides; their overlap in 64 bits
        on = (at[i, 3] + at[j, 3]) - torch.sqrt(_sq32(at[i], at[j])) > 0
        i, j = i[on], j[on]
        order = torch.argsort(i * len(p) + j)
        i, j = i[order], j[order]
        delta = p[i, 3] + p[j, 3] - (p[i, :3] - p[j, :3]).norm(dim=1)
        return {"bits": None, "contacts": None, "ci": None, "cj": None,
                "delta": _padded(delta, _contact_room(len(p)))}
    skin = np.concatenate([np.minimum(
        0.2 * s.pos[:, 3].astype(np.float64),
        np.maximum(_cap(s, s.cell_factor) - s.pos[:, 3].astype(np.float64), 0.0)) for s in sc])
    skin = _f64(skin)
    if kind == "rebuild":
        out = torch.cat([_f64(x[0])[:, :3], skin[:, None]], 1)
        return {"rows": None, "col": None, "entries": None, "ref": out}
    cur = ref.clone()                  # the check in binary32, as it is defined
    for k in range(case["passes"]):
        far = _sq32(x[k], cur) > cur[:, 3] * cur[:, 3]
        cur[far, :3] = x[k][far, :3]
        cur[far, 3] = skin[far].float()
    out = _f64(cur)
    moved = (cur[:, 3] != ref[:, 3])
    out[moved, 3] = skin[moved]
    return {"bits": None, "ref": out}


def _exact_clumps(case, seed):
    pos, q, off, sub, _, _ = _clump_inputs(case, seed)
    p = _f64(pos)
    zero = torch.zeros(len(p), dtype=torch.int64, device=p.device)
    i, j = _close_pairs(p[:, :3], p[:, 3], zero, 1e-9)
    dev = p.device
    off = torch.from_numpy(off).long().to(dev)
    owner = torch.repeat_interleave(torch.arange(len(p), device=dev), off[1:] - off[:-1])

    def world(pos, q, sub):
        w, x, y, z = q.unbind(1)
        two = 2.0
        R = [[1.0 - two * (y * y + z * z), two * (x * y - w * z), two * (x * z + w * y)],
             [two * (x * y + w * z), 1.0 - two * (x * x + z * z), two * (y * z - w * x)],
             [two * (x * z - w * y), two * (y * z + w * x), 1.0 - two * (x * x + y * y)]]
        out = [pos[owner, k] + ((R[k][0][owner] * sub[:, 0] + R[k][1][owner] * sub[:, 1]) +
                                R[k][2][owner] * sub[:, 2]) for k in range(3)]
        return torch.stack(out, 1)

    f32 = [torch.from_numpy(t).to(dev) for t in (pos, q, sub)]
    c32 = world(*f32)
    c64 = world(*(t.double() for t in f32))
    r32, r64 = f32[2][:, 3], f32[2][:, 3].double()
    keys, deltas = [], []
    for a in range(4):
        for b in range(4):
            s, t = off[i] + a, off[j] + b
            ok = (s < off[i + 1]) & (t < off[j + 1])
            s, t, ii, jj = s[ok], t[ok], i[ok], j[ok]
            on = (r32[s] + r32[t]) - torch.sqrt(_sq32(c32[s], c32[t])) > 0
            s, t, ii, jj = s[on], t[on], ii[on], jj[on]
            keys.append(((ii * 64 + a) << 32) | (jj * 64 + b))
            deltas.append(r64[s] + r64[t] - (c64[s] - c64[t]).norm(dim=1))
    order = torch.argsort(torch.cat(keys))
    return {"contacts": None, "key": None,
            "delta": _padded(torch.cat(deltas)[order], _clump_room(len(p)))}


def _exact_train(case, seed):
    s, _ = _train_inputs(case, seed)
    f = s.astype(np.float64)
    m, var = f.mean(0), f.var(0)
    sd = np.sqrt(var)
    # the weights depend on the library's own shuffle of the samples
    return {"params": None, "mu": m[:8], "isd": 1.0 / sd[:8], "losses": None,
            "y_range": np.array([m[8] / 16.0, m[8] + 4.0 * sd[8]])}


def exact(case, seed):
    kind = case["kind"]
    if kind == "advance":
        return _exact_advance(case, seed)
    if kind == "clumps":
        return _exact_clumps(case, seed)
    if kind == "train":
        return _exact_train(case, seed)
    return _exact_stepping(case, seed)
