"""Device memory of the DEM driver: the second copy of the state, which joined
steps go back and forth between, is allocated by the first call that needs it,
also inside a capture."""
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


def test_phases_and_single_steps_take_no_second_copy():
    lvb = _lvb()
    small = lvb.DEM(_gas(3000))            # the kernels are loaded
    for m in (1, 3):
        small.advance(m)
    small.step()
    small.sync()
    small.close()
    n = 4_000_000
    dem = lvb.DEM(_gas(n))

    def taken(f):
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        f()
        assert dem.sync() == lvb.LVB_OK
        return before - torch.cuda.mem_get_info()[0]

    assert taken(dem.step) < 8 << 20
    assert taken(lambda: dem.advance(1)) < 8 << 20
    assert 48 * n <= taken(lambda: dem.advance(2)) < 48 * n + (8 << 20)
    assert taken(lambda: dem.advance(20)) < 8 << 20
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
