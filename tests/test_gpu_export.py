"""The exported list (lvb_get_pairs, lvb_get_pairs_ij, lvb_get_contacts) into
device arrays, host arrays and a mix of both: rows of 0 to some 100 entries
(registers up to 16, ranks above) and sizes around the kernels' blocks,
against the brute force of the same binary32 formula; a capacity one short
writes the offsets and no entry.
"""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _lvb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2208_13770_gb300 import lvb
    return lvb


def _cloud(n, crowd, seed):
    """n spheres in a box, `crowd` of them in one small corner of it."""
    rng = np.random.default_rng(seed)
    pos = np.zeros((n, 4), np.float32)
    side = 2.2e-3 * max(n, 1) ** (1 / 3) + 4e-3
    pos[:, :3] = rng.uniform(0, side, size=(n, 3))
    pos[:crowd, :3] = 1e-3 + rng.uniform(0, 1.2e-3, size=(crowd, 3))
    pos[:, 3] = rng.uniform(0.5e-3, 1e-3, size=n)
    return pos, side


def _brute(pos, skin_factor, H):
    """Sorted pairs i < j, and of them the contacts with their overlaps."""
    x = pos[:, :3]
    r = pos[:, 3]
    skin = np.minimum(np.float32(skin_factor) * (np.float32(2.0) * r), np.float32(H) - r)
    R = r + skin
    out = []
    for i in range(len(pos)):
        d = x[i] - x[i + 1:]
        d2 = (d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2]
        c = R[i] + R[i + 1:]
        j = np.flatnonzero(d2 <= c * c)
        dl = (r[i] + r[i + 1 + j]) - np.sqrt(d2[j])
        out += [(i, i + 1 + int(q), float(v)) for q, v in zip(j, dl)]
    return out


@pytest.mark.parametrize("n,crowd", [(1, 0), (2, 2), (255, 10), (256, 20), (257, 60), (3000, 100)])
@pytest.mark.parametrize("where", ["device", "host", "mixed"])
def test_lists_match_brute_force(n, crowd, where):
    lvb = _lvb()
    pos, side = _cloud(n, crowd, 3 + n)
    x = torch.from_numpy(pos).cuda()
    ctx = lvb.LVB(x, (0, 0, 0), (side, side, side), lvb.LVB_SKIN_DIAMETER_FACTOR, 0.1, 1e-6)
    want = _brute(pos, 0.1, ctx.stats()["rnl_max"])
    pi, pj = (np.array([p[k] for p in want], np.int32) for k in (0, 1))
    m = len(want)

    def buf(count, dtype, second=False):
        dev = where == "device" or (where == "mixed" and second)
        t = torch.full((max(count, 1),), -7, dtype=dtype, device="cuda" if dev else "cpu")
        return t

    got = ctypes.c_int64(-1)
    # pairs
    a, b = buf(m, torch.int32), buf(m, torch.int32, True)
    assert lvb.lvb_get_pairs_ij(ctx.ctx, a.data_ptr(), b.data_ptr(), m, ctypes.byref(got)) == 0
    assert got.value == m
    assert np.array_equal(a.cpu().numpy()[:m], pi) and np.array_equal(b.cpu().numpy()[:m], pj)
    # rows
    rows, col = buf(n + 1, torch.int32), buf(2 * m, torch.int32, True)
    assert lvb.lvb_get_pairs(ctx.ctx, rows.data_ptr(), col.data_ptr(), 2 * m,
                             ctypes.byref(got)) == 0
    assert got.value == 2 * m
    i2, j2 = np.concatenate([pi, pj]), np.concatenate([pj, pi])
    order = np.lexsort((j2, i2))
    ptr = np.concatenate([[0], np.cumsum(np.bincount(i2, minlength=n))])
    assert np.array_equal(rows.cpu().numpy(), ptr)
    assert np.array_equal(col.cpu().numpy()[:2 * m], j2[order])
    if crowd >= 60:
        assert np.diff(ptr).max() > 16
    # contacts
    touch = [p for p in want if p[2] > 0]
    k = len(touch)
    ci, cj, dl = buf(k, torch.int32), buf(k, torch.int32, True), buf(k, torch.float32)
    assert lvb.lvb_get_contacts(ctx.ctx, x.data_ptr(), ci.data_ptr(), cj.data_ptr(),
                                dl.data_ptr(), k, ctypes.byref(got)) == 0
    assert got.value == k
    assert ci.cpu().numpy()[:k].tolist() == [p[0] for p in touch]
    assert cj.cpu().numpy()[:k].tolist() == [p[1] for p in touch]
    assert np.array_equal(dl.cpu().numpy()[:k], np.array([p[2] for p in touch], np.float32))
    # one place too few
    if m:
        a.fill_(-7)
        assert lvb.lvb_get_pairs_ij(ctx.ctx, a.data_ptr(), b.data_ptr(), m - 1,
                                    ctypes.byref(got)) == lvb.LVB_ECAPACITY
        assert got.value == m and int((a != -7).sum()) == 0
        rows.fill_(-7)
        col.fill_(-7)
        assert lvb.lvb_get_pairs(ctx.ctx, rows.data_ptr(), col.data_ptr(), 2 * m - 1,
                                 ctypes.byref(got)) == lvb.LVB_ECAPACITY
        assert np.array_equal(rows.cpu().numpy(), ptr) and int((col != -7).sum()) == 0
    ctx.close()


def test_device_arrays_off_their_words():
    """Device arrays at an odd address hold the same bytes as aligned ones."""
    lvb = _lvb()
    n = 257
    pos, side = _cloud(n, 60, 11)
    x = torch.from_numpy(pos).cuda()
    ctx = lvb.LVB(x, (0, 0, 0), (side, side, side), lvb.LVB_SKIN_DIAMETER_FACTOR, 0.1, 1e-6)
    want = _brute(pos, 0.1, ctx.stats()["rnl_max"])
    m = len(want)

    def buf(words):
        return torch.zeros(4 * words + 4, dtype=torch.uint8, device="cuda")[1:4 * words + 1]

    def words(t):
        return np.frombuffer(t.cpu().numpy().tobytes(), np.int32)

    got = ctypes.c_int64(-1)
    a, b, rows, col = buf(m), buf(m), buf(n + 1), buf(2 * m)
    assert lvb.lvb_get_pairs_ij(ctx.ctx, a.data_ptr(), b.data_ptr(), m, ctypes.byref(got)) == 0
    assert words(a).tolist() == [p[0] for p in want] and words(b).tolist() == [p[1] for p in want]
    assert lvb.lvb_get_pairs(ctx.ctx, rows.data_ptr(), col.data_ptr(), 2 * m,
                             ctypes.byref(got)) == 0
    i2, j2 = (np.array([p[k] for p in want] + [p[1 - k] for p in want]) for k in (0, 1))
    assert np.array_equal(words(col), j2[np.lexsort((j2, i2))])
    assert np.array_equal(np.diff(words(rows)), np.bincount(i2, minlength=n))
    ref, ref_al = buf(4 * n), torch.zeros(4 * n, dtype=torch.float32, device="cuda")
    assert lvb.lvb_get_ref(ctx.ctx, ref.data_ptr()) == 0
    assert lvb.lvb_get_ref(ctx.ctx, ref_al.data_ptr()) == 0
    assert ref.cpu().numpy().tobytes() == ref_al.cpu().numpy().tobytes()
    ctx.close()
