"""A scene build's blocks wait for one another no longer than the context's wait limit: with 0 ns every block that meets
before the last one gives up, the build returns LIDAR_ETIMEOUT and makes no scene, and the next build gives the tree it
would have given anyway.  (Nothing hangs and nothing faults: the kernels after the one that gave up check what it left.)"""
import numpy as np
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
    if not lid.launch_config()["fused_scatter"]:
        pytest.skip("no cooperative launch on this device")
    yield lid
    lid.close()


def _export(scene):
    return [a.view(np.uint8) for a in (*scene.export(), scene.export_wide(4), scene.export_wide(8))]


def _times_out_and_recovers(L, n, **options):
    from paper_2208_10295_gb300 import capi
    verts, tris = _random_triangles(n, 5 * n)
    limit0, options0 = L.wait_limit(), L.build_options()
    try:
        L.set_build_options(**options)
        scene = L.build_scene(verts, tris)
        want = _export(scene)
        scene.free()
        L.set_wait_limit(0)
        with pytest.raises(capi.LidarError) as e:
            L.build_scene(verts, tris)
        assert e.value.status == capi.LIDAR_ETIMEOUT
        assert L.sync_status() == 0
        L.set_wait_limit(limit0)
        scene = L.build_scene(verts, tris)
        for a, b in zip(want, _export(scene)):
            assert np.array_equal(a, b)
        scene.free()
    finally:
        L.set_wait_limit(limit0)
        L.set_build_options(**options0)


@pytest.mark.parametrize("n", [5000, 70001])
@pytest.mark.parametrize("treelet_rounds", [0, 3])
def test_clustering_gives_up(L, n, treelet_rounds):
    _times_out_and_recovers(L, n, method=1, collapse=0, treelet_rounds=treelet_rounds)


@pytest.mark.parametrize("n", [5000, 70001])
@pytest.mark.parametrize("treelet_rounds", [0, 3])
def test_clustering_gives_up_before_the_dynamic_program(L, n, treelet_rounds):
    """The collapse's program climbs the tree that the clustering did not finish: it must read none of it."""
    _times_out_and_recovers(L, n, method=1, collapse=1, treelet_rounds=treelet_rounds)


def test_collapse_gives_up(L):
    """The tree is whole (the Karras build has no such waits): the levels of the wide trees give up."""
    for collapse in (0, 1):
        _times_out_and_recovers(L, 70001, method=0, collapse=collapse, treelet_rounds=0)


def test_one_block_waits_for_nobody(L):
    verts, tris = _random_triangles(400, 11)
    limit0 = L.wait_limit()
    try:
        L.set_wait_limit(0)
        scene = L.build_scene(verts, tris)
        scene.free()
    finally:
        L.set_wait_limit(limit0)
