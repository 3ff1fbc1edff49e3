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


def _morton_order(verts, tris):
    """Triangles by 63-bit Morton key of their centroids, ties in input order.  FP32 as the build rounds it: a
    centroid's product with 1/3 and its offset from the lower bound are one fused operation."""
    f = np.float32
    v = verts[tris]
    total = (v[:, 0] + v[:, 1]) + v[:, 2]
    c = total * f(1.0 / 3.0)
    lo, ext = c.min(0), c.max(0) - c.min(0)
    inv = np.where(ext > 0, f(1.0) / np.where(ext > 0, ext, f(1.0)), f(0.0)).astype(f)
    off = (total.astype(np.float64) * np.float64(f(1.0 / 3.0)) - lo.astype(np.float64)).astype(f)
    q = np.clip(off * inv * f(2097151.0), f(0.0), f(2097151.0)).astype(np.uint64)
    key = np.zeros(len(tris), np.uint64)
    for bit in range(21):
        for axis in range(3):
            key |= ((q[:, axis] >> np.uint64(bit)) & np.uint64(1)) << np.uint64(3 * bit + 2 - axis)
    return np.argsort(key, kind="stable")


@pytest.mark.parametrize("n", [2, 33, 511, 512, 513, 4095, 4096, 4097, 6143, 6145, 70001])
def test_leaves_in_morton_order(L, n):
    """The radix sort's one-block form (up to 4,096 keys) and its tiled passes, with every seventh key repeated."""
    verts, tris = _random_triangles(n, n)
    tris[6::7] = tris[: len(tris[6::7])]
    try:
        L.set_build_options(method=0)
        scene = L.build_scene(verts, tris)
        assert np.array_equal(scene.export()[1], _morton_order(verts, tris))
        scene.free()
    finally:
        L.set_build_options(method=1)
