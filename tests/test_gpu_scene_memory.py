"""When a scene's memory is given back."""
import pytest

from test_gpu_treelets import _random_triangles

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2208_10295_gb300 import Lidar
    lid = Lidar(0)
    yield lid
    lid.close()


def test_free_waits_for_other_streams(L):
    """Work on a stream of the caller's (a replayed graph, say) may still read the scene."""
    scene = L.build_scene(*_random_triangles(5000, 1))
    side, done = torch.cuda.Stream(), torch.cuda.Event()
    with torch.cuda.stream(side):
        torch.cuda._sleep(200_000_000)  # about 0.1 s
        done.record(side)
    assert not done.query()
    scene.free()
    assert done.query()
