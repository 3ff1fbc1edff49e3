"""The launch shape and the order of the work change no result: what the library chooses by the number of rays against
shapes that a caller sets, and frames and sweeps of equal size, whose tiles take turns, against ones cast beside a
frame of another size, which do not."""
import ctypes
import dataclasses

import numpy as np
import pytest

import synth
from gpu_util import setup
from parity import to_numpy

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def make():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2208_10295_gb300 import Lidar
    made = []

    def new(w, **shape):
        lid = Lidar(0)
        made.append(lid)
        if shape:
            lid.set_launch_config(block_threads=64, blocks_per_sm=1)  # another one first, so that it is the caller's
            lid.set_launch_config(**shape)
        return lid, setup(lid, w)[0]
    yield new
    for lid in made:
        lid.close()


def _workload(n_frames, n_az, beams_off, n_subrays):
    """`beams_off` beams fewer than 32 n_az in slot 0; a smaller sensor in slot 1."""
    w = synth.small_terrain(seed=5, n_frames=n_frames + 1, n_az=n_az, n_subrays=n_subrays,
                            divergence=2e-3 if n_subrays > 1 else 0.0)
    s = w.sensors[0]
    n = s.n_beams - beams_off
    w.sensors[:] = [dataclasses.replace(s, az_rad=s.az_rad[:n], el_rad=s.el_rad[:n]),
                    dataclasses.replace(s, az_rad=s.az_rad[:45], el_rad=s.el_rad[:45])]
    return w


def _cast(lid, scene, w, frames, sweep=False):
    n = lid.total_beams(frames)
    beams = lid.alloc_beams(n)
    if sweep:
        echoes = lid.alloc_echoes(n, 2)
        lid.cast_sweep_into(scene, frames, w.seed, beams, echoes)
        beams = {**beams, **{"echo_" + k: v for k, v in echoes.items()}}
    else:
        lid.cast_into(scene, frames, w.seed, beams)
    assert lid.sync_status() == 0
    return to_numpy(beams)


def _same(a, b, n):
    for k in a:
        assert np.array_equal(a[k][:n].view(np.uint8), b[k][:n].view(np.uint8)), k


@pytest.mark.parametrize("n_frames,n_az,n_subrays", [(1, 64, 1), (3, 1024, 7), (12, 1024, 7)])
def test_chosen_shape_against_set_ones(make, n_frames, n_az, n_subrays):
    """Fewer than 19,456 tiles of 32 rays, fewer than 77,824, and more (on 152 SMs)."""
    w = _workload(n_frames, n_az, 3, n_subrays)
    frames = w.frames[:n_frames]
    lid, scene = make(w)
    own = _cast(lid, scene, w, frames)
    for shape in ({"block_threads": 128, "blocks_per_sm": 4}, {"block_threads": 256, "blocks_per_sm": 3}):
        other, scene2 = make(w, **shape)
        assert {k: other.launch_config()[k] for k in shape} == shape
        _same(own, _cast(other, scene2, w, frames), lid.total_beams(frames))


@pytest.mark.parametrize("sweep", [False, True])
@pytest.mark.parametrize("n_subrays", [1, 7])
@pytest.mark.parametrize("n_frames,beams_off", [(2, 0), (3, 1), (5, 31), (7, 33), (16, 2047)])
def test_turns_of_equal_frames(make, n_frames, beams_off, n_subrays, sweep):
    w = _workload(n_frames, 64, beams_off, n_subrays)
    lid, scene = make(w)
    fr = w.frames
    if sweep:
        fr = synth.make_sweep_frames([(int(fr[k]["sensor"]), int(fr[k]["frame"]), fr[k]["pose"], fr[k + 1]["pose"])
                                      for k in range(n_frames)])
    turns = fr[:n_frames]
    mixed = np.concatenate([turns, turns[:1]])
    mixed[-1]["sensor"] = 1
    _same(_cast(lid, scene, w, turns, sweep), _cast(lid, scene, w, mixed, sweep), lid.total_beams(turns))


class _KernelParams(ctypes.Structure):
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3),
                ("shared", ctypes.c_uint), ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p),
                ("kernel", ctypes.c_void_p), ("context", ctypes.c_void_p)]


def _captured_shape(lid, batch, scene, w, beams):
    """Threads per block and blocks per SM of the kernel that a cast of the batch launches, from a stream capture."""
    cuda = ctypes.CDLL("libcuda.so.1")
    stream, graph, n = ctypes.c_void_p(lid.stream.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t()
    assert cuda.cuStreamBeginCapture_v2(stream, 2) == 0  # relaxed
    try:
        batch.cast_into(scene, w.seed, beams)
    finally:
        assert cuda.cuStreamEndCapture(stream, ctypes.byref(graph)) == 0
    assert cuda.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cuda.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    shapes = []
    for node in nodes:
        kind, p = ctypes.c_int(), _KernelParams()
        assert cuda.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        if kind.value == 0:  # a kernel
            assert cuda.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node), ctypes.byref(p)) == 0
            shapes.append((p.block[0], p.grid[0] / torch.cuda.get_device_properties(0).multi_processor_count))
    cuda.cuGraphDestroy(graph)
    assert len(shapes) == 1  # a dense cast is one kernel
    return shapes[0]


def test_whose_shape_a_cast_runs(make):
    """A shape that a caller sets is what runs, the default values from the first call on included; other fields leave
    it alone; two zeros hand it back."""
    from paper_2208_10295_gb300 import Lidar, capi
    lid = Lidar(0, torch.cuda.Stream())
    try:
        w = _workload(3, 1024, 3, 7)  # more tiles than any shape below keeps resident
        scene = setup(lid, w)[0]
        frames = w.frames[:3]
        beams = lid.alloc_beams(lid.total_beams(frames), ("valid",))
        batch = lid.batch(frames)
        batch.cast_into(scene, w.seed, beams)
        assert lid.sync_status() == 0

        def now():
            c = lid.launch_config()
            return (c["block_threads"], c["blocks_per_sm"]), _captured_shape(lid, batch, scene, w, beams)
        own = now()
        assert own[0] == (0, 0) and own[1][0] == 256
        lid.set_launch_config(ray_order=0)
        assert now() == own
        lid.set_launch_config(ray_order=1, block_threads=128, blocks_per_sm=4)
        assert now() == ((128, 4), (128, 4))
        lid.set_launch_config(ray_order=1)
        assert now() == ((128, 4), (128, 4))
        kept = lid.launch_config()
        lid.set_launch_config(block_threads=64, blocks_per_sm=0)
        assert now() == ((64, 4), (64, 4))
        lid.set_launch_config(block_threads=0, blocks_per_sm=2)
        assert now() == ((128, 2), (128, 2))
        lid.set_launch_config(**kept)
        assert now() == ((128, 4), (128, 4))
        lid.set_launch_config(block_threads=0, blocks_per_sm=0)
        assert now() == own
        for bad in ({"block_threads": -32}, {"blocks_per_sm": -1}, {"block_threads": 288}, {"blocks_per_sm": 65}):
            with pytest.raises(capi.LidarError) as e:
                lid.set_launch_config(**bad)
            assert e.value.status == capi.LIDAR_EINVAL
        assert now() == own
        batch.free()
    finally:
        lid.close()


@pytest.mark.parametrize("n_frames,n_subrays,blocks", [(10, 1, (2, 3)), (24, 1, (3, 4)), (8, 2, (2, 3)), (24, 2, (3, 4))])
def test_where_the_chosen_shape_changes(make, n_frames, n_subrays, blocks):
    """1,216 tiles of 32 beams a frame and one fewer, at the bounds for 152 SMs: 12,160 and 29,184 tiles of 32 rays,
    with sub-rays 19,456 and 58,368."""
    from paper_2208_10295_gb300 import Lidar
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the bounds depend on the number of SMs")
    for off, want in zip((32, 0), blocks):
        lid = Lidar(0, torch.cuda.Stream())
        try:
            w = _workload(n_frames, 1216, off, n_subrays)
            scene = setup(lid, w)[0]
            frames = w.frames[:n_frames]
            beams = lid.alloc_beams(lid.total_beams(frames), ("valid",))
            batch = lid.batch(frames)
            assert _captured_shape(lid, batch, scene, w, beams) == (256, want)
            batch.free()
        finally:
            lid.close()
