"""Rounds of treelet restructuring against a full evaluation: every node's treelet in every round, bottom-up, restated
here.  The build looks only at treelets below which something changed near enough to matter; that has to leave the same
tree.  Corners are on an integer grid (every area exact) and the triangle cost a power of two, so that only the sums of
costs are rounded, and those in a stated order.  The scenes of large triangles around small ones have costs so far apart
that a change among the small is lost in the rounding of the costs above it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

K = 7
f32 = np.float32


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


def _partitions():
    """Per size of a subset of the leaves: the subsets, and their parts with the lowest leaf, largest others first."""
    out = []
    for size in range(2, K + 1):
        subsets = [s for s in range(1, 1 << K) if bin(s).count("1") == size]
        parts = []
        for s in subsets:
            low, rest = s & -s, s & (s - 1)
            q, row = rest, []
            while q:
                q = (q - 1) & rest
                row.append(q | low)
            parts.append(row)
        out.append((np.array(subsets), np.array(parts)))
    return out


PARTITIONS = _partitions()
MEMBERS = np.array([[s >> i & 1 for i in range(K)] for s in range(1 << K)], bool)


def _area(lo, hi):
    d = hi - lo
    return d[..., 0] * d[..., 1] + d[..., 1] * d[..., 2] + d[..., 2] * d[..., 0]


class _Tree:
    def __init__(self, nodes, tri_cost):
        self.child = nodes[:, 12:14].view(np.int32).copy()
        b = nodes[:, :12]
        self.lo = np.stack([b[:, [0, 4]], b[:, [2, 6]], b[:, [8, 10]]], -1).copy()
        self.hi = np.stack([b[:, [1, 5]], b[:, [3, 7]], b[:, [9, 11]]], -1).copy()
        self.cost = np.zeros(len(nodes), f32)
        self.tri_cost = f32(tri_cost)
        self.rewritten = 0

    def order(self):
        """Nodes, children before parents."""
        out, todo = [], [0]
        while todo:
            n = todo.pop()
            out.append(n)
            todo += [int(c) for c in self.child[n] if c >= 0]
        return out[::-1]

    def leaf_cost(self, ref, area):
        return self.cost[ref] if ref >= 0 else self.tri_cost * area

    def look(self, node):
        ref = [int(c) for c in self.child[node]]
        lo, hi = np.zeros((K, 3), f32), np.zeros((K, 3), f32)
        lo[:2], hi[:2] = self.lo[node], self.hi[node]
        area = [_area(lo[i], hi[i]) for i in range(2)]
        now = _area(np.minimum(lo[0], lo[1]), np.maximum(hi[0], hi[1]))
        now = f32(now + self.leaf_cost(ref[0], area[0]))
        now = f32(now + self.leaf_cost(ref[1], area[1]))
        inner = [node]
        while len(ref) < K and any(r >= 0 for r in ref):
            at = max((i for i in range(len(ref)) if ref[i] >= 0), key=lambda i: (area[i], -i))
            o, k = ref[at], len(ref)
            inner.append(o)
            ref[at], ref[k:] = int(self.child[o, 0]), [int(self.child[o, 1])]
            lo[at], hi[at], lo[k], hi[k] = self.lo[o, 0], self.hi[o, 0], self.lo[o, 1], self.hi[o, 1]
            area[at], area[k:] = _area(lo[at], hi[at]), [_area(lo[k], hi[k])]
        k = len(ref)
        if k == 2:
            self.cost[node] = now
            return
        member = MEMBERS[:, :, None]
        blo = np.where(member, lo, np.inf).min(1).astype(f32)
        bhi = np.where(member, hi, -np.inf).max(1).astype(f32)
        c, split = np.zeros(1 << K, f32), np.zeros(1 << K, int)
        for i in range(k):
            c[1 << i] = self.leaf_cost(ref[i], area[i])
        full = (1 << k) - 1
        for subsets, parts in PARTITIONS[:k - 1]:
            keep = subsets <= full
            subsets, parts = subsets[keep], parts[keep]
            total = c[parts] + c[subsets[:, None] ^ parts]
            best = total.argmin(1)  # the first of equal ones
            rows = np.arange(len(subsets))
            c[subsets] = _area(blo[subsets], bhi[subsets]) + total[rows, best]
            split[subsets] = parts[rows, best]
        if not c[full] < now * f32(f32(1.0) - f32(1e-5)):
            self.cost[node] = now
            return
        todo, used = [(full, node)], 1
        while todo:
            s, at = todo.pop()
            for side, part in enumerate((split[s], s ^ split[s])):
                if part & (part - 1) == 0:
                    self.child[at, side] = ref[int(part).bit_length() - 1]
                else:
                    self.child[at, side] = inner[used]
                    todo.append((part, inner[used]))
                    used += 1
                self.lo[at, side], self.hi[at, side] = blo[part], bhi[part]
            self.cost[at] = c[s]
        self.rewritten += 1


def _spread(n, seed):
    rng = np.random.default_rng(seed)
    at = rng.integers(0, 1000, (n, 1, 3))
    return (at + rng.integers(0, 20, (n, 3, 3))).astype(f32)


def _large_around_small(n, seed):
    rng = np.random.default_rng(seed)
    big = rng.integers(0, 900, (n // 4, 1, 3)) + rng.integers(0, 1100, (n // 4, 3, 3))
    small = rng.integers(300, 1500, 3) + rng.integers(0, 40, (n - n // 4, 1, 3)) * rng.integers(1, 4, (n - n // 4, 1, 1))
    small = small + rng.integers(0, 4, (n - n // 4, 3, 3))
    return np.concatenate([big, small]).astype(f32)


@pytest.mark.parametrize("make", [_spread, _large_around_small])
@pytest.mark.parametrize("method", [0, 1])
@pytest.mark.parametrize("n,rounds,tri_cost", [(8, 8, 1.0), (33, 3, 1.0), (150, 8, 64.0), (700, 2, 1.0), (700, 8, 64.0)])
def test_rounds_are_those_of_a_full_evaluation(L, n, rounds, tri_cost, method, make):
    v = make(n, n + rounds)
    verts, tris = v.reshape(-1, 3), np.arange(3 * n, dtype=np.uint32).reshape(n, 3)
    options = L.build_options()
    try:
        L.set_build_options(method=method, treelet_rounds=0)
        scene = L.build_scene(verts, tris)
        want = _Tree(scene.export()[0], tri_cost)
        scene.free()
        for _ in range(rounds):
            for node in want.order():
                want.look(node)
        assert want.rewritten > 0
        L.set_build_options(method=method, treelet_rounds=rounds, tri_cost=tri_cost)
        scene = L.build_scene(verts, tris)
        got = _Tree(scene.export()[0], tri_cost)
        assert np.array_equal(got.child, want.child)
        assert np.array_equal(got.lo, want.lo) and np.array_equal(got.hi, want.hi)
        assert scene.info()["treelets"] == want.rewritten
        scene.free()
    finally:
        L.set_build_options(**options)
