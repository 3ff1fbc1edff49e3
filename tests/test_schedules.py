"""The ray schedules a tuner tries, and that it applies the one it names (no GPU); that none changes a result (GPU)."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")


class _Recorder:
    """Stands for the library: notes which schedule the slots get."""

    def __init__(self):
        self.calls = []

    def set_launch_config(self, **cfg):
        assert "schedule" not in cfg

    def reset_schedule(self, slot):
        self.calls.append(("level", slot))

    def morton_schedule(self, slot):
        self.calls.append(("morton", slot))

    def schedule_by_cost(self, scene, frame, seed, mode):
        self.calls.append((("cost", "bucket")[mode], int(frame[0]["sensor"])))


@pytest.mark.parametrize("schedule", ["morton", "level", "cost", "bucket"])
def test_the_tuner_applies_what_it_names(schedule):
    from paper_2208_10295_gb300 import tune
    assert schedule in {c["schedule"] for c in tune.candidates() if c["ray_order"] == 1}
    w = synth.small_terrain(seed=1, n_frames=2, n_az=8)
    frames = w.frames.copy()
    frames["sensor"] = (0, 3)
    cfg = next(c for c in tune.candidates() if c["schedule"] == schedule and c["ray_order"] == 1)
    lib = _Recorder()
    tune.apply(lib, None, cfg, frames, 0)
    assert {slot: name for name, slot in lib.calls} == {0: schedule, 3: schedule}


def test_morton_schedule_arguments():
    from paper_2208_10295_gb300 import build, capi
    capi.load(build.build())
    assert capi.lidar_morton_schedule(None, 0) == capi.LIDAR_EINVAL


@pytest.mark.gpu
def test_schedules_change_no_result():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from gpu_util import gpu_cast
    from paper_2208_10295_gb300 import Lidar, capi
    lid = Lidar(0)
    w = synth.small_terrain(seed=3, n_frames=2, n_az=100)
    want, scene = gpu_cast(lid, w)
    n = lid.total_beams(w.frames)
    for order in (lid.morton_schedule, lid.reset_schedule):
        order(0)
        beams = lid.alloc_beams(n)
        lid.cast_into(scene, w.frames, w.seed, beams)
        assert lid.sync_status() == 0
        for k, v in want.items():
            assert np.array_equal(beams[k].cpu().numpy().view(np.uint8), v.view(np.uint8)), k
    with pytest.raises(capi.LidarError) as e:
        lid.morton_schedule(7)
    assert e.value.status == capi.LIDAR_ESTATE
    lid.close()
