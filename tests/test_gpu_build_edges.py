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


def _integer_triangles(n, seed):
    """Corners on an integer grid: every area of the build is a whole number below 2^24, exact in FP32."""
    rng = np.random.default_rng(seed)
    at = rng.integers(0, 1000, (n, 1, 3))
    verts = (at + rng.integers(0, 20, (n, 3, 3))).astype(np.float32).reshape(-1, 3)
    return verts, np.arange(3 * n, dtype=np.uint32).reshape(n, 3)


def _ploc_children(lo, hi, radius):
    """Children of every node of the clustering: nearest neighbours within `radius` (ties to the lower position),
    mutual pairs merge at the lower position, ids count down from n - 2."""
    n = len(lo)
    ref, child, top = ~np.arange(n, dtype=np.int32), np.zeros((n - 1, 2), np.int32), n - 2
    while len(ref) > 1:
        m = len(ref)
        best_d, best = np.full(m, np.inf, np.float32), np.full(m, -1)
        for off in [o for o in range(-radius, radius + 1) if o and abs(o) < m]:
            e = slice(max(0, -off), m - max(0, off))
            o = slice(max(0, off), m + min(0, off))
            d = np.maximum(hi[e], hi[o]) - np.minimum(lo[e], lo[o])
            area = d[:, 0] * d[:, 1] + d[:, 1] * d[:, 2] + d[:, 2] * d[:, 0]
            nearer = area < best_d[e]
            best_d[e] = np.where(nearer, area, best_d[e])
            best[e] = np.where(nearer, np.arange(m)[o], best[e])
        mutual = best[best] == np.arange(m)
        left = np.nonzero(mutual & (np.arange(m) < best))[0]
        right = best[left]
        assert len(left)
        ids = top - np.arange(len(left), dtype=np.int32)
        child[ids, 0], child[ids, 1] = ref[left], ref[right]
        lo[left], hi[left] = np.minimum(lo[left], lo[right]), np.maximum(hi[left], hi[right])
        ref[left] = ids
        stay = np.ones(m, bool)
        stay[right] = False
        lo, hi, ref, top = lo[stay], hi[stay], ref[stay], top - len(left)
    return child


@pytest.mark.parametrize("n,radius", [(2, 16), (3, 16), (33, 16), (511, 16), (512, 16), (513, 16), (1023, 16),
                                      (1024, 16), (1025, 16), (4864, 16), (4865, 16), (14593, 16), (34049, 16),
                                      (72961, 16), (150784, 16), (150785, 16), (400, 1), (5000, 1), (200000, 1),
                                      (513, 5), (1000, 5), (90001, 5), (600, 64), (1024, 64), (19457, 64),
                                      (58369, 64), (140000, 64)])
def test_clustering_at_its_widths(L, n, radius):
    """One block alone, 8 / 4 / 2 / 1 lanes a cluster, two clusters a thread, several tiles a block (152 SMs)."""
    verts, tris = _integer_triangles(n, n + radius)
    try:
        L.set_build_options(method=1, ploc_radius=radius)
        scene = L.build_scene(verts, tris)
        nodes, leaf = scene.export()
        v = verts[tris[leaf]]
        assert np.array_equal(nodes[:, 12:14].view(np.int32), _ploc_children(v.min(1), v.max(1), radius))
        scene.free()
    finally:
        L.set_build_options(method=1, ploc_radius=16)


def _wide_children(nodes, width):
    """Wide nodes breadth-first, each the binary references of its children: the one of largest area is opened (ties to
    the first) until there are `width` or only triangles; internal ones first."""
    child = nodes[:, 12:14].view(np.int32)
    b = nodes[:, :12].astype(np.float64)
    lo = np.stack([b[:, [0, 4]], b[:, [2, 6]], b[:, [8, 10]]], -1)
    hi = np.stack([b[:, [1, 5]], b[:, [3, 7]], b[:, [9, 11]]], -1)
    d = hi - lo
    area = d[..., 0] * d[..., 1] + d[..., 1] * d[..., 2] + d[..., 2] * d[..., 0]
    out, frontier = [], [0]
    while frontier:
        below = []
        for node in frontier:
            kids = [(child[node, s], area[node, s]) for s in (0, 1)]
            while len(kids) < width and any(r >= 0 for r, _ in kids):
                at = max((k for k in range(len(kids)) if kids[k][0] >= 0), key=lambda k: (kids[k][1], -k))
                o = kids[at][0]
                kids[at] = (child[o, 0], area[o, 0])
                kids.append((child[o, 1], area[o, 1]))
            refs = [int(r) for r, _ in kids]
            inner = [r for r in refs if r >= 0]
            out.append((inner, [r for r in refs if r < 0]))
            below += inner
        frontier = below
    return out


@pytest.mark.parametrize("n", [2, 3, 4, 5, 8, 9, 33, 257, 1025, 1100, 5000])
def test_wide_nodes(L, n):
    """Children and their order by the largest-area rule, and the layout of both rules' trees."""
    from test_gpu_parity import _wide_tree_invariants
    verts, tris = _integer_triangles(n, 3 * n)
    try:
        for collapse in (0, 1):
            L.set_build_options(method=1, collapse=collapse)
            scene = L.build_scene(verts, tris)
            nodes, leaf = scene.export()
            v = verts[tris[leaf]]
            for width in (4, 8):
                got = scene.export_wide(width)
                _wide_tree_invariants(got, width, n, v.min(1), v.max(1))
                if collapse == 0:
                    code = got.reshape(len(got), -1, 4)[:, 6 * (width // 4):7 * (width // 4)].reshape(len(got), width)
                    first = 1
                    want = np.zeros((len(got), width), np.int32)
                    for i, (inner, leaves) in enumerate(_wide_children(nodes, width)):
                        row = list(range(first, first + len(inner))) + leaves
                        want[i, :len(row)] = row
                        first += len(inner)
                    assert np.array_equal(code.view(np.int32), want)
            scene.free()
    finally:
        L.set_build_options(method=1, collapse=0)


def test_scenes_come_and_go(L):
    """The arrays of freed scenes serve the next ones: scenes of changing sizes, freed out of order, stay whole."""
    kept = []
    for k, n in enumerate([5000, 33, 70001, 2, 4097, 5000]):
        verts, tris = _random_triangles(n, 100 + k)
        kept.append((L.build_scene(verts, tris), verts, tris))
        if k % 2:
            kept.pop(0)[0].free()
    for scene, verts, tris in kept:
        _check_binary_tree(*scene.export(), verts, tris)
        scene.free()
