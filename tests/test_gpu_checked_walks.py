"""The bounds-checked build walks a 4-wide tree as the normal build does, with 32-bit offsets up to a number of nodes (a
small one there, so that both walks are reached) and 64-bit addresses above; casts and sweeps give bit for bit the
records of the normal build on either side.  The checked library runs in a child process (one library per process)."""
import os
import subprocess
import sys
import textwrap

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
CELLS = {"near": 64, "far": 256}  # terrain cells a side
NEAR_NODES = 1 << 14

CHILD = textwrap.dedent("""
    import sys, numpy as np
    sys.path[:0] = [{root!r}, {here!r}]
    from paper_2208_10295_gb300 import build, capi
    capi.load(build.build_checked())
    import test_gpu_checked_walks as t
    out = {{}}
    for name in t.CELLS:
        records, nodes, walk = t.cast_and_sweep(name)
        assert (nodes > t.NEAR_NODES) == (name == "far"), nodes
        assert walk == (4 if name == "far" else 2), (name, walk)
        out.update({{name + "|" + k: v for k, v in records.items()}})
    np.savez({path!r}, **out)
""")


def _walk(lid, batch, scene, seed, beams):
    """Last template argument of the cast kernel that a cast of the batch launches."""
    import ctypes
    import re

    from test_gpu_launch_shape import _KernelParams
    cuda, graph, n = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p(), ctypes.c_size_t()
    stream = ctypes.c_void_p(lid.stream.cuda_stream)
    assert cuda.cuStreamBeginCapture_v2(stream, 2) == 0  # relaxed
    try:
        batch.cast_into(scene, seed, beams)
    finally:
        assert cuda.cuStreamEndCapture(stream, ctypes.byref(graph)) == 0
    assert cuda.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cuda.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    walks = []
    for node in nodes:
        kind, p, name = ctypes.c_int(), _KernelParams(), ctypes.c_char_p()
        assert cuda.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        if kind.value == 0:
            assert cuda.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node), ctypes.byref(p)) == 0
            if p.func:
                assert cuda.cuFuncGetName(ctypes.byref(name), ctypes.c_void_p(p.func)) == 0
            else:
                assert cuda.cuKernelGetName(ctypes.byref(name), ctypes.c_void_p(p.kernel)) == 0
            walks += re.findall(r"k_castILb0ELi\d+ELi(\d+)E", name.value.decode())
    cuda.cuGraphDestroy(graph)
    assert len(walks) == 1
    return int(walks[0])


def cast_and_sweep(name):
    """Dense records and echoes of two frames and a sweep, the number of 4-wide nodes, the walk of the cast."""
    from gpu_util import setup
    from paper_2208_10295_gb300 import Lidar
    lid = Lidar(0, torch.cuda.Stream())
    w = synth.small_terrain(seed=6, n_cells=CELLS[name], half=40.0, n_frames=2, n_az=128, n_subrays=3, divergence=2e-3)
    scene = setup(lid, w)[0]
    n = lid.total_beams(w.frames)
    beams = lid.alloc_beams(n)
    lid.cast_into(scene, w.frames, w.seed, beams)
    assert lid.sync_status() == 0
    out = {"cast_" + k: v.cpu().numpy() for k, v in beams.items()}
    sweep = synth.make_sweep_frames([(0, 0, w.frames[0]["pose"], w.frames[1]["pose"])])
    dense, echoes = lid.alloc_beams(n // 2), lid.alloc_echoes(n // 2, 2)
    lid.cast_sweep_into(scene, sweep, w.seed, dense, echoes)
    assert lid.sync_status() == 0
    out.update({"sweep_" + k: v.cpu().numpy() for k, v in dense.items()})
    out.update({"echo_" + k: v.cpu().numpy() for k, v in echoes.items()})
    batch = lid.batch(w.frames)
    walk = _walk(lid, batch, scene, w.seed, beams)
    nodes = scene.info()["n_nodes4"]
    batch.free()
    lid.close()
    return out, nodes, walk


def test_checked_build_walks_as_the_normal_one(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    path = str(tmp_path / "checked.npz")
    code = CHILD.format(root=os.path.dirname(HERE), here=HERE, path=path)
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=1200)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    got = np.load(path)
    for name in CELLS:
        records, _, walk = cast_and_sweep(name)
        assert walk == 2
        for k, v in records.items():
            assert np.array_equal(v.view(np.uint8), got[name + "|" + k].view(np.uint8)), (name, k)
