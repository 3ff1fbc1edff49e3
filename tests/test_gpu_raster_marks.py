"""A raster cast tests only the pixels its beams read; what each beam sees has to be what the whole images hold at its
pixel.  Image widths around whole words of marks, from images with every pixel read to sparse ones."""
import numpy as np
import pytest

import synth
from gpu_util import setup
from parity import to_numpy

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


def _pixels(dirs, W, K):
    """Camera, column and row each beam reads (FP32, rounded as the kernels round), -1 where none."""
    f32 = np.float32
    az = -np.pi + (np.arange(K) + 0.5) * 2.0 * np.pi / K
    ck, sk = np.cos(az).astype(f32), np.sin(az).astype(f32)
    f, c = f32(W / (2.0 * np.tan(np.pi / K))), f32(0.5 * W)
    x, y, z = dirs.T
    depth = x[:, None] * ck + y[:, None] * sk
    k = np.argmax(depth, 1)
    zk = depth[np.arange(len(k)), k]
    with np.errstate(divide="ignore", invalid="ignore"):
        px = np.floor(c + f * ((x * -sk[k] + y * ck[k]) / zk))
        py = np.floor(c - f * (z / zk))
    ok = (zk > 0) & (py >= 0) & (py < W)
    return np.where(ok, k, -1), np.clip(px, 0, W - 1).astype(int), np.where(ok, py, 0).astype(int)


@pytest.mark.parametrize("W,K", [(1, 3), (16, 4), (31, 6), (32, 6), (33, 5), (64, 64), (97, 6), (700, 6)])
def test_beams_see_the_whole_images_pixels(L, W, K):
    w = synth.small_terrain(seed=21, n_frames=2, n_az=512)
    scene, _ = setup(L, w)
    n = L.total_beams(w.frames)
    beams = L.alloc_beams(n, ("tri", "inst", "mat", "valid", "theta_deg"))
    L.raster_cast_into(scene, w.frames, w.seed, beams, W, K)
    assert L.sync_status() == 0
    got = to_numpy(beams)
    k, ix, iy = _pixels(L.beam_dirs(0), W, K)
    per = len(k)
    for f in range(2):
        g = {key: v.cpu().numpy().view(np.uint32) for key, v in L.raster_gbuffer(scene, w.frames[f:f + 1], W, K).items()}
        here = {key: v[f * per:(f + 1) * per] for key, v in got.items()}
        tri = np.where(k >= 0, g["tri"][k, iy, ix], 0xFFFFFFFF)
        hit = tri != 0xFFFFFFFF
        assert np.array_equal(here["tri"].astype(np.uint32), tri)
        assert np.array_equal(here["inst"].astype(np.uint32)[hit], g["inst"][k, iy, ix][hit])
        assert np.array_equal(here["mat"].astype(np.uint32)[hit], g["angle_mat"][k, iy, ix][hit] >> 24)
        code = (g["angle_mat"][k, iy, ix] & 0xFFFFFF).astype(np.float32)
        assert np.array_equal(here["theta_deg"][hit], (code * (np.float32(90.0) / np.float32(16777215.0)))[hit])
    scene.free()
