"""Scene builds at the sizes where their kernels change shape: warps, blocks and tiles one triangle short, full and
one over.  Whatever the options, the tree has to hold every triangle once under exact boxes, its reported height has
to be its height, and building it again has to give the same tree."""
import numpy as np
import pytest

from test_gpu_treelets import _check_binary_tree, _random_triangles

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


def _height(nodes):
    child = nodes[:, 12:14].view(np.int32)
    depth = np.zeros(len(nodes), int)
    top, todo = 0, [0]
    while todo:
        i = todo.pop()
        depth_i = depth[i] + 1
        top = max(top, depth_i)
        for c in child[i]:
            if c >= 0:
                depth[c] = depth_i
                todo.append(int(c))
    return top


@pytest.mark.parametrize("rounds", [1, 2, 8])
@pytest.mark.parametrize("n", [8, 31, 32, 33, 64, 65, 1000])
def test_treelet_rounds(L, n, rounds):
    verts, tris = _random_triangles(n, 7 * n)
    try:
        for method in (0, 1):
            L.set_build_options(method=method, treelet_rounds=rounds - 1)
            scene = L.build_scene(verts, tris)
            before = _check_binary_tree(*scene.export(), verts, tris)[2]
            scene.free()
            L.set_build_options(method=method, treelet_rounds=rounds)
            scene = L.build_scene(verts, tris)
            nodes, leaf = scene.export()
            assert _check_binary_tree(nodes, leaf, verts, tris)[2] <= before * (1.0 + 1e-6)
            assert scene.info()["max_depth"] == _height(nodes)
            again = L.build_scene(verts, tris)
            assert np.array_equal(again.export()[0].view(np.uint8), nodes.view(np.uint8))
            again.free()
            scene.free()
    finally:
        L.set_build_options(method=1, treelet_rounds=0)
