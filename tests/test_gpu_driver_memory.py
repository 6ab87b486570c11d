"""Device memory of the DEM driver: the second copy of the state, which joined
steps go back and forth between, is allocated by dem_init where it is a small part
of the free memory, else by the first call that needs it, also inside a capture;
and without it the same steps run in place."""
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


def _gas(n):
    s = scenes.ballistic(n=n, seed=77, phi=0.19)
    s.vel[:, :3] *= 100.0
    return s


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.fixture(scope="module")
def measured():
    """(n, bytes of a context of n without its second copy, its state after 5 steps);
    all kernels loaded."""
    lvb = _lvb()
    packed = scenes.packed(n=700)
    packed.wall = "specular"
    for s in (packed, _gas(3000)):
        dem = lvb.DEM(s)
        dem.advance(1)
        dem.advance(3)
        dem.step()
        assert dem.sync() == lvb.LVB_OK
        dem.close()
    n = 6_000_000
    for _ in range(2):                     # the first fills the caching allocator
        before = _free()
        dem = lvb.DEM(_gas(n))
        bytes_ = before - _free() - 48 * n
        dem.advance(5)
        state = dem.state()
        dem.close()
    return n, bytes_, state


@pytest.mark.parametrize("copies", [6, 0.5])
def test_second_copy_where_memory_is_short(measured, copies):
    # so much is left after dem_init: six copies (not an eighth), half a copy (the
    # steps run in place)
    lvb = _lvb()
    n, bytes_, state = measured
    lvb.DEM(_gas(n)).close()               # (the caching allocator holds the inputs' memory)
    filler = torch.empty(_free() - bytes_ - int(copies * 48 * n), dtype=torch.uint8, device="cuda")
    dem = None
    try:
        dem = lvb.DEM(_gas(n))
        left = _free()
        assert abs(left - copies * 48 * n) < 64 << 20
        dem.advance(1)
        assert dem.sync() == lvb.LVB_OK
        assert left - _free() < 4 << 20
        dem.advance(4)
        assert dem.sync() == lvb.LVB_OK
        taken = left - _free()
        assert (48 * n <= taken < 48 * n + (8 << 20)) if copies > 1 else taken < 4 << 20
        for x, y in zip(dem.state(), state):
            assert np.array_equal(x, y)
    finally:
        if dem is not None:
            dem.close()
        del filler
        torch.cuda.empty_cache()


def test_second_copy_where_memory_is_plenty(measured):
    lvb = _lvb()
    n, bytes_, _ = measured
    lvb.DEM(_gas(n)).close()
    before = _free()
    dem = lvb.DEM(_gas(n))
    taken = before - _free()
    assert abs(taken - bytes_ - 48 * n) < 8 << 20
    dem.close()


@pytest.mark.parametrize("n", [700, 6000])
def test_first_call_under_capture(n):
    lvb = _lvb()
    stream = torch.cuda.Stream()
    a = lvb.DEM(_gas(n), stream=stream.cuda_stream)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        a.advance(3)
    for _ in range(4):
        graph.replay()
    torch.cuda.synchronize()
    b = lvb.DEM(_gas(n))
    for _ in range(12):
        b.step()
    assert a.sync() == lvb.LVB_OK and b.sync() == lvb.LVB_OK
    assert a.lvb.stats()["steps"] == 12
    for x, y in zip(a.state(), b.state()):
        assert np.array_equal(x, y)
    assert np.array_equal(a.lvb.ref(), b.lvb.ref())
    a.close()
    b.close()
