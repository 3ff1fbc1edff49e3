"""When a scene's memory is given back."""
import ctypes

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


def test_build_under_capture_is_refused():
    """A build synchronises, so a capture cannot hold it: LIDAR_ENOMEM before anything is allocated, the capture goes
    on, and the context builds afterwards, its scenes' memory still from the pool."""
    from paper_2208_10295_gb300 import Lidar, capi
    stream = torch.cuda.Stream()
    lid = Lidar(0, stream)
    verts, tris = _random_triangles(50000, 2)
    dv, dt = torch.tensor(verts, device="cuda"), torch.tensor(tris.view("int32"), device="cuda")
    x = torch.zeros(1, device="cuda")
    torch.cuda.synchronize()
    graph, out = torch.cuda.CUDAGraph(), ctypes.c_void_p()
    with torch.cuda.graph(graph, stream=stream):
        x.add_(1)
        status = capi.lidar_scene_build(lid.handle, dv.data_ptr(), len(verts), dt.data_ptr(), len(tris), None, None,
                                        ctypes.byref(out))
        x.add_(1)
    assert status == capi.LIDAR_ENOMEM and not out
    graph.replay()
    torch.cuda.synchronize()
    assert x.item() == 2
    lid.build_scene(verts, tris).free()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    scene = lid.build_scene(verts, tris)
    assert scene.export()[0].shape[0] == len(tris) - 1
    assert torch.cuda.mem_get_info()[0] == before  # the arrays of the scene that was freed
    scene.free()
    lid.close()
