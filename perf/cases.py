"""The framework's work as its users have it done: casts, sweeps, raster frames, fits and scene builds.

Each case is one call pattern through `paper_2208_10295_gb300.torch_api`, on synthetic scenes of the kinds the
repository's own workloads use: boxes on a ground plane, an fBm terrain with objects, a city of extruded buildings.
"""
import math

import numpy as np
import torch

from paper_2208_10295_gb300 import torch_api as api

DEV = "cuda"

# terrain and city trees as the benchmark builds them: treelet rounds, weight of the faces normal to z
TUNED_TERRAIN = {"rounds": 2, "wz": 0.23}
TUNED_CITY = {"rounds": 8, "wz": 0.35}


def listed():
    return [
        # the smallest sensor in a small scene, one frame at a time: launches and latency count
        {"name": "frame_16ch_boxes", "kind": "frame", "scene": "boxes", "size": 64, "objects": 0, "rounds": 0,
         "wz": 1.0, "ch": 16, "az": 1800, "sub": 1, "frames": 1, "mats": 4, "cfg": "default", "dense": True},
        # the 128-channel sensor in a million triangles, one frame at a time, everything at its default
        {"name": "frame_128ch_terrain", "kind": "frame", "scene": "terrain", "size": 512, "objects": 2000,
         "rounds": 0, "wz": 1.0, "ch": 128, "az": 2048, "sub": 1, "frames": 1, "mats": 32, "cfg": "default",
         "dense": False},
        # the same sensor streaming: restructured tree, tuned launch, cost schedule from the pose before, point
        # buffers in turn
        {"name": "stream_128ch_terrain", "kind": "stream", "scene": "terrain", "size": 512, "objects": 2000,
         **TUNED_TERRAIN, "ch": 128, "az": 2048, "sub": 1, "frames": 1, "mats": 32, "cfg": "stream", "dense": False},
        # a vehicle rig (16, 32, 64, 128 channels) over a stretch of its drive as one graph replay
        {"name": "rig_graph_terrain", "kind": "rig", "scene": "terrain", "size": 512, "objects": 2000,
         **TUNED_TERRAIN, "ch": 0, "az": 2048, "sub": 1, "frames": 8, "mats": 32, "cfg": "default", "dense": False},
        # divergent beams in a city: seven sub-rays a beam, strongest return, several frames a call
        {"name": "city_7subrays", "kind": "frame", "scene": "city", "size": 1024, "objects": 5000, **TUNED_CITY,
         "ch": 128, "az": 2048, "sub": 7, "frames": 4, "mats": 64, "cfg": "wide", "dense": False},
        # rolling shutter with first and last echoes in a city
        {"name": "sweep_echoes_city", "kind": "sweep", "scene": "city", "size": 512, "objects": 1200, "rounds": 0,
         "wz": 1.0, "ch": 64, "az": 1024, "sub": 7, "frames": 4, "mats": 16, "cfg": "default", "dense": True},
        # a fitting step over a stretch of frames: tables, forward with tape, fused-MSE adjoint, table gradients
        {"name": "fit_16frames", "kind": "fit", "scene": "terrain", "size": 512, "objects": 2000, **TUNED_TERRAIN,
         "ch": 128, "az": 2048, "sub": 1, "frames": 16, "mats": 32, "cfg": "wide", "dense": True},
        # the adjoint alone, from a stored tape and the user's own dL/dI; odd beam count
        {"name": "adjoint_1m", "kind": "adjoint", "beams": 1000003, "mats": 32},
        # a small scene rebuilt every frame (moving objects) and cast
        {"name": "rebuild_boxes", "kind": "rebuild", "scene": "boxes", "size": 64, "objects": 0, "rounds": 0,
         "wz": 1.0, "ch": 16, "az": 1800, "sub": 1, "frames": 1, "mats": 4, "cfg": "default", "dense": True},
        # a large scene rebuilt and cast
        {"name": "rebuild_terrain", "kind": "rebuild", "scene": "terrain", "size": 512, "objects": 2000, "rounds": 0,
         "wz": 1.0, "ch": 32, "az": 2048, "sub": 1, "frames": 1, "mats": 32, "cfg": "default", "dense": True},
        # a scene loaded once with the restructured tree, then cast
        {"name": "load_city", "kind": "rebuild", "scene": "city", "size": 512, "objects": 1200, **TUNED_CITY,
         "ch": 64, "az": 2048, "sub": 1, "frames": 1, "mats": 64, "cfg": "default", "dense": True},
        # the raster-and-resample sampling of the 128-channel sensor's frame
        {"name": "raster_128ch", "kind": "raster", "scene": "terrain", "size": 512, "objects": 2000, "rounds": 0,
         "wz": 1.0, "ch": 128, "az": 2048, "sub": 1, "frames": 1, "mats": 32, "cfg": "default", "dense": True,
         "width": 1024, "cameras": 6},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["frame", "frame", "stream", "rig", "sweep", "fit", "autograd", "adjoint", "rebuild", "rebuild",
                       "raster"])
    if kind == "adjoint":
        return {"kind": kind, "beams": log_int(20000, 3000000), "mats": rng.choice([1, 4, 7, 32, 64])}
    scene = rng.choice(["boxes", "terrain", "city"]) if kind in ("frame", "rebuild") else (
        "city" if kind == "sweep" else "terrain")
    c = {"kind": kind, "scene": scene, "rounds": 0, "wz": 1.0, "sub": 1, "frames": 1, "cfg": "default",
         "mats": rng.choice([4, 8, 32, 33, 64]), "ch": rng.choice([16, 32, 40, 64, 128]), "az": log_int(300, 2048),
         "dense": rng.random() < 0.5}
    if scene == "boxes":
        c.update(size=log_int(8, 300), objects=0)
    elif scene == "terrain":
        n = log_int(64, 512)
        c.update(size=n, objects=max(4, int(2000 * (n / 512) ** 2)))
    else:
        n = log_int(128, 700)
        c.update(size=n, objects=max(8, int(1200 * (n / 512) ** 2)))
    if scene != "boxes" and rng.random() < 0.4:
        c.update(rounds=rng.choice([1, 2, 3]), wz=rng.choice([0.23, 0.35, 1.0]))
    if kind == "stream":
        c.update(cfg="stream", dense=False)
    if kind == "rig":
        c.update(ch=0, frames=rng.randint(1, 6), dense=False)
    if kind == "frame":
        c.update(frames=rng.choice([1, 1, 2, 5]), cfg=rng.choice(["default", "wide"]))
        if scene == "city" and rng.random() < 0.5:
            c.update(sub=rng.choice([3, 7, 8]), frames=rng.choice([1, 2]))
    if kind == "sweep":
        c.update(sub=rng.choice([1, 3, 7]), frames=rng.randint(1, 3), dense=True)
    if kind == "fit":
        c.update(frames=rng.randint(1, 12), cfg="wide", dense=True)
    if kind == "autograd":
        c.update(size=log_int(32, 128), objects=rng.randint(4, 40), ch=rng.choice([16, 32]), frames=rng.randint(1, 2),
                 mats=8, dense=True, rounds=0, wz=1.0, az=log_int(300, 1024))
    if kind == "rebuild":
        c.update(dense=True)
    if kind == "raster":
        c.update(width=log_int(200, 1100), cameras=rng.choice([4, 6, 8]), dense=True)
    return c


# ------------------------------------------------------------------- scenes

def _fbm(rng, half, amplitude):
    """Height function: six octaves of smoothstep-blended value noise, FP64 on the GPU."""
    octs, wl, amp = [], 128.0, 1.0
    for _ in range(6):
        n = int(math.ceil(2 * half / wl)) + 2
        octs.append((wl, amp, torch.from_numpy(rng.uniform(-1.0, 1.0, (n, n))).to(DEV)))
        wl, amp = wl / 2, amp / 2

    def height(x, y):
        h = torch.zeros_like(x)
        for w, a, lat in octs:
            gx, gy = (x + half) / w, (y + half) / w
            ix = gx.floor().long().clamp(0, lat.shape[1] - 2)
            iy = gy.floor().long().clamp(0, lat.shape[0] - 2)
            fx, fy = gx - ix, gy - iy
            sx, sy = fx * fx * (3 - 2 * fx), fy * fy * (3 - 2 * fy)
            p = lat[iy, ix] * (1 - sx) + lat[iy, ix + 1] * sx
            q = lat[iy + 1, ix] * (1 - sx) + lat[iy + 1, ix + 1] * sx
            h = h + a * (p * (1 - sy) + q * sy)
        return h * (amplitude / 1.2)

    return height


def _box(subdiv):
    v, t = [], []
    g = np.linspace(-0.5, 0.5, subdiv + 1)
    for axis in range(3):
        for sign in (-0.5, 0.5):
            base = len(v)
            for b in g:
                for a in g:
                    p = [0.0, 0.0, 0.0]
                    p[axis], p[(axis + 1) % 3], p[(axis + 2) % 3] = sign, a, b
                    v.append(p)
            n = subdiv + 1
            for j in range(subdiv):
                for i in range(subdiv):
                    k = base + j * n + i
                    t += [[k, k + 1, k + n + 1], [k, k + n + 1, k + n]]
    return np.array(v), np.array(t)


def _ball(n_lat=9, n_lon=20):
    v, t = [], []
    for i in range(n_lat):
        th = math.pi * i / (n_lat - 1)
        for j in range(n_lon):
            ph = 2 * math.pi * j / n_lon
            v.append([math.sin(th) * math.cos(ph), math.sin(th) * math.sin(ph), math.cos(th)])
    for i in range(n_lat - 1):
        for j in range(n_lon):
            a, b = i * n_lon + j, i * n_lon + (j + 1) % n_lon
            if i > 0:
                t.append([a, b, a + n_lon])
            if i < n_lat - 2:
                t.append([b, b + n_lon, a + n_lon])
    return np.array(v), np.array(t)


def _prism(sides=8, storeys=6):
    ang = 2 * np.pi * np.arange(sides) / sides
    v = [[math.cos(a), math.sin(a), z] for z in np.linspace(0, 1, storeys + 1) for a in ang]
    t = []
    for s in range(storeys):
        for e in range(sides):
            a, b = s * sides + e, s * sides + (e + 1) % sides
            t += [[a, b, b + sides], [a, b + sides, a + sides]]
    top = storeys * sides
    t += [[top, top + e, top + e + 1] for e in range(1, sides - 1)]
    return np.array(v), np.array(t)


def _instances(parts, shape, scale, yaw, pos, mats, first):
    """Copies of a template: scaled, turned about z, moved; one label each."""
    v, t = (torch.from_numpy(a).to(DEV) for a in shape)
    scale, yaw, pos = (torch.as_tensor(a, device=DEV, dtype=torch.float64) for a in (scale, yaw, pos))
    p = v[None] * scale[:, None]
    c, s = yaw.cos()[:, None], yaw.sin()[:, None]
    p = torch.stack([p[..., 0] * c - p[..., 1] * s, p[..., 0] * s + p[..., 1] * c, p[..., 2]], -1) + pos[:, None]
    n = p.shape[0]
    base = sum(q[0].shape[0] for q in parts) + torch.arange(n, device=DEV)[:, None, None] * v.shape[0]
    parts.append((p.reshape(-1, 3).float(), (t[None] + base).reshape(-1, 3).int(),
                  np.repeat(mats, t.shape[0]).astype(np.uint16),
                  np.repeat(first + np.arange(n), t.shape[0]).astype(np.uint32)))


def _scene(case, seed):
    """verts, tris (device), materials, instances (host), the ground's height function."""
    rng = np.random.default_rng([seed, 11])
    M, size, n_obj = case["mats"], case["size"], case["objects"]
    parts = []
    if case["scene"] == "boxes":
        half = 100.0
        q = torch.tensor([[-half, -half, 0], [half, -half, 0], [half, half, 0], [-half, half, 0]], device=DEV)
        parts.append((q.float(), torch.tensor([[0, 1, 2], [0, 2, 3]], device=DEV, dtype=torch.int32),
                      np.zeros(2, np.uint16), np.zeros(2, np.uint32)))
        side = rng.uniform(1.0, 10.0, (size, 3))
        c = rng.uniform(-95.0, 95.0, (size, 2))
        c[:, 1] += np.where(c[:, 1] < 0, -8.0, 8.0)
        _instances(parts, _box(1), side, np.zeros(size), np.concatenate([c, side[:, 2:] / 2], 1),
                   rng.integers(0, M, size), 1)

        def height(x, y):
            return torch.zeros_like(x)
    else:
        cell = 1.0 if case["scene"] == "terrain" else 2.0
        half = size * cell / 2
        height = _fbm(rng, half, 5.0 if size > 100 else 1.0)
        g = torch.linspace(-half, half, size + 1, device=DEV, dtype=torch.float64)
        y, x = torch.meshgrid(g, g, indexing="ij")
        verts = torch.stack([x, y, height(x, y)], -1).reshape(-1, 3).float()
        iy, ix = torch.meshgrid(torch.arange(size, device=DEV), torch.arange(size, device=DEV), indexing="ij")
        a = (iy * (size + 1) + ix).reshape(-1)
        b, d = a + 1, a + size + 1
        tris = torch.stack([torch.stack([a, b, d + 1], -1), torch.stack([a, d + 1, d], -1)], 1).reshape(-1, 3).int()
        patch = rng.integers(0, min(4, M), (size // 32 + 1, size // 32 + 1))
        r = np.arange(size) // 32
        mat = np.repeat(patch[np.ix_(r, r)].reshape(-1), 2).astype(np.uint16)
        parts.append((verts, tris, mat, np.zeros(len(mat), np.uint32)))
        lo_m = min(4, M - 1)
        c = rng.uniform(-half * 0.97, half * 0.97, (n_obj, 2))
        if case["scene"] == "terrain":
            c[:, 1] += np.where(c[:, 1] < 0, -8.0, 8.0)
        else:  # one building to a cell of a grid, streets between, none on the road along y = 0
            n = int(2 * half // 28)
            cells = rng.permutation(n * n)[:n_obj]
            c = -half + 28.0 * (np.stack([cells % n, cells // n], 1) + 0.5)
            c[:, 1] += np.where(c[:, 1] < 0, -17.0, 17.0)
            n_obj = len(cells)
        h = height(torch.from_numpy(c[:, 0]).to(DEV), torch.from_numpy(c[:, 1]).to(DEV)).cpu().numpy()
        yaw = rng.uniform(0, 2 * np.pi, n_obj)
        mats = rng.integers(lo_m, M, n_obj)
        if case["scene"] == "terrain":
            k = n_obj // 2
            side = rng.uniform(0.5, 6.0, (k, 3))
            _instances(parts, _box(4), side, yaw[:k], np.concatenate([c[:k], (h[:k] + side[:, 2] / 2 - 0.2)[:, None]], 1),
                       mats[:k], 1)
            r = rng.uniform(0.3, 3.0, n_obj - k)
            _instances(parts, _ball(), np.repeat(r[:, None], 3, 1), yaw[k:],
                       np.concatenate([c[k:], (h[k:] + 0.8 * r)[:, None]], 1), mats[k:], 1 + k)
        else:
            r = rng.uniform(5.0, 13.0, n_obj)
            s = np.stack([r, r * rng.uniform(0.6, 1.0, n_obj), rng.uniform(8.0, 40.0, n_obj)], 1)
            _instances(parts, _prism(), s, yaw, np.concatenate([c, h[:, None] - 1.0], 1), mats, 1)
    v, t, m, i = zip(*parts)
    return torch.cat(v), torch.cat(t), np.concatenate(m), np.concatenate(i), height


class _Sensor:
    """A sensor description, as set_sensor takes it."""

    def __init__(self, az, el, d_max, sub, gain=1.0):
        self.az_rad, self.el_rad = az, el
        self.r_min, self.r_max, self.d_max, self.RL_max = 0.5, d_max, d_max, 0.8
        self.sigma, self.gain, self.range_exp, self.r_ref, self.sigma_k = 0.02, gain, 0.0, 1.0, 0.0
        self.n_subrays, self.divergence_rad = sub, 1e-4 if sub > 1 else 0.0


def _spinning(ch, n_az, d_max, sub=1):
    if ch == 128:  # 0.1 degrees apart about the horizon, coarser below and above
        el = np.concatenate([-25.0 + np.arange(56) * 23.0 / 56.0, np.arange(-20, 21) * 0.1,
                             2.0 + np.arange(1, 32) * 13.0 / 31.0])
    else:
        el = np.linspace(-16.0 if ch < 64 else -25.0, 15.0, ch)
    az = 2.0 * np.pi * np.arange(n_az) / n_az
    return _Sensor(np.repeat(az, ch), np.deg2rad(np.tile(el, n_az)), d_max, sub)


def _poses(case, seed, height, n):
    """Poses along a drive near the origin, 0.6 m a frame, the sensor 2 m above the ground."""
    rng = np.random.default_rng([seed, 23])
    if case["scene"] == "boxes":
        x0, y0 = rng.uniform(-2.0, 2.0, 2)
    else:
        x0, y0 = rng.uniform(-10.0, 0.0), rng.uniform(-1.5, 1.5)
    yaw = rng.uniform(-0.2, 0.2) + 0.01 * np.arange(n)
    x = x0 + 0.6 * np.arange(n)
    y = y0 + 0.6 * np.sin(0.2 * np.arange(n))
    z = height(torch.from_numpy(x).to(DEV), torch.from_numpy(y).to(DEV)).cpu().numpy() + 2.0
    out = np.zeros((n, 12), np.float32)
    c, s = np.cos(yaw), np.sin(yaw)
    for k, col in enumerate([c, -s, 0, x, s, c, 0, y, 0, 0, 1, z]):
        out[:, k] = col
    return out


def _frames(poses, sensors=(0,)):
    fr = np.zeros(len(poses) * len(sensors), api.FRAME_DTYPE)
    for k in range(len(fr)):
        fr[k] = (sensors[k % len(sensors)], k // len(sensors), poses[k // len(sensors)])
    return fr


def _params(case, seed):
    rng = np.random.default_rng([seed, 37])
    a, w = rng.uniform(0.05, 0.9, case["mats"]), rng.uniform(2.0, 10.0, case["mats"])
    s = rng.uniform(0.0, 1.0, case["mats"]) * np.minimum(0.5, 1.0 - a)
    return np.stack([a, s, w], 1).astype(np.float32)


def _d_max(case):
    return 100.0 if case["scene"] == "boxes" else (40.0 if case["size"] <= 128 else 200.0)


def _noise(seed):
    return 2000 + seed


LAUNCH = {"default": {}, "stream": {"block_threads": 256, "blocks_per_sm": 3},
          "wide": {"block_threads": 256, "blocks_per_sm": 4}}
RIG = (16, 32, 64, 128)
TAPE = ("valid", "intensity", "mat", "theta_deg", "rf")


# ------------------------------------------------------------------- prepare

def prepare(case, seed):
    st = {"case": case, "seed": _noise(seed)}
    L = st["L"] = api.Lidar(0)
    par = st["params"] = torch.from_numpy(_params(case, seed)).to(DEV)
    if case["kind"] == "adjoint":
        st.update(_tape(case, seed))
        L.set_materials(L.build_tables(par))
        st["gT"] = torch.zeros((case["mats"], 91), device=DEV)
        st["gg"] = torch.zeros(1, device=DEV)
        return st
    kind = case["kind"]
    st["mesh"] = _scene(case, seed)
    verts, tris, mat, inst, height = st["mesh"]
    L.set_launch_config(**LAUNCH[case["cfg"]])
    L.set_build_options(treelet_rounds=case["rounds"], area_weight=(1.0, 1.0, case["wz"]))
    if kind != "rebuild":
        st["scene"] = L.build_scene(verts, tris, mat, inst)
    L.set_materials(L.build_tables(par))
    d_max = _d_max(case)
    slots = RIG if kind == "rig" else (case["ch"],)
    for k, ch in enumerate(slots):
        L.set_sensor(k, _spinning(ch, case["az"] if ch > 16 else min(case["az"], 1800), d_max, case["sub"]))
    n = case["frames"]
    poses = _poses(case, seed, height, n + 2)
    fr = st["frames"] = _frames(poses[1:n + 1], range(len(slots)))
    nb = L.total_beams(fr)

    def points():
        return {k: v.zero_() for k, v in L.alloc_points(nb).items()}

    if kind in ("frame", "rig"):
        st["points"] = points()
    if kind in ("frame", "rebuild", "raster", "sweep"):
        st["beams"] = L.alloc_beams(nb) if case["dense"] else None
    if kind == "stream":
        L.schedule_by_cost(st["scene"], _frames(poses[:1]), st["seed"], mode=1)
        st["ring"], st["turn"] = [points() for _ in range(4)], 0
    if kind == "rig":
        st["poses"] = torch.from_numpy(np.ascontiguousarray(fr["pose"])).to(DEV)
        st["batch"] = L.batch(fr)
        st["graph"] = st["batch"].graph(st["scene"], st["seed"], points=st["points"], poses=st["poses"])
    if kind == "sweep":
        sw = np.zeros(n, np.dtype([("sensor", np.int32), ("frame", np.int32), ("pose0", np.float32, (12,)),
                                   ("pose1", np.float32, (12,))]))
        for k in range(n):
            sw[k] = (0, k, poses[k], poses[k + 1])
        st["sweeps"], st["echoes"] = sw, L.alloc_echoes(nb, 2)
    if kind in ("fit", "autograd"):
        g = torch.Generator(device=DEV).manual_seed(seed)
        st["target"] = torch.rand(nb, device=DEV, generator=g) * 0.9
        st["tvalid"] = (torch.rand(nb, device=DEV, generator=g) < 0.9).to(torch.uint8)
    if kind == "fit":
        st["tape"] = L.alloc_beams(nb, TAPE)
        st["gT"] = torch.zeros((case["mats"], 91), device=DEV)
        st["gg"], st["loss"] = torch.zeros(1, device=DEV), torch.zeros(1, device=DEV)
    if kind == "autograd":
        st["params"] = par.requires_grad_(True)
        st["gain"] = torch.tensor(1.0, device=DEV, requires_grad=True)
    return st


def _tape(case, seed):
    """A stored tape, its values as casts give them: neighbouring beams see one material, angles drift."""
    n, M = case["beams"], case["mats"]
    g = torch.Generator(device=DEV).manual_seed(seed)
    theta = (45.0 + 44.9 * torch.sin(torch.arange(n, device=DEV) * 0.013)
             + torch.randn(n, device=DEV, generator=g) * 2.0).clamp(0.0, 90.0)
    runs = torch.randint(0, M, (n // 19 + 1,), device=DEV, generator=g)
    return {"tape": {"valid": (torch.rand(n, device=DEV, generator=g) < 0.8).to(torch.uint8),
                     "mat": runs.repeat_interleave(19)[:n].to(torch.int16),
                     "theta_deg": theta.contiguous(),
                     "rf": (0.5 + 1.5 * torch.rand(n, device=DEV, generator=g))},
            "gI": torch.randn(n, device=DEV, generator=g) * 1e-3}


# ------------------------------------------------------------------- run

def run(st):
    L, case = st["L"], st["case"]
    kind = case["kind"]
    if kind == "frame":
        L.cast_into(st["scene"], st["frames"], st["seed"], st["beams"], st["points"])
        return {**st["points"], **{"dense_" + k: v for k, v in (st["beams"] or {}).items()}}
    if kind == "stream":
        p = st["ring"][st["turn"] % 4]
        st["turn"] += 1
        L.cast_into(st["scene"], st["frames"], st["seed"], None, p)
        return p
    if kind == "rig":
        st["graph"].launch()
        return st["points"]
    if kind == "sweep":
        L.cast_sweep_into(st["scene"], st["sweeps"], st["seed"], st["beams"], st["echoes"], mode=1, separation=0.5)
        return {**st["beams"], **{"echo_" + k: v for k, v in st["echoes"].items()}}
    if kind == "raster":
        L.raster_cast_into(st["scene"], st["frames"], st["seed"], st["beams"], case["width"], case["cameras"])
        return st["beams"]
    if kind == "rebuild":
        verts, tris, mat, inst, _ = st["mesh"]
        scene = L.build_scene(verts, tris, mat, inst)
        L.cast_into(scene, st["frames"], st["seed"], st["beams"])
        scene.free()
        return st["beams"]
    if kind == "adjoint":
        st["gT"].zero_()
        st["gg"].zero_()
        L.cast_backward(st["tape"], 1.0, st["gI"], st["gT"], st["gg"])
        return [st["gT"], st["gg"]]
    if kind == "fit":
        L.set_materials(L.build_tables(st["params"]))
        L.cast_into(st["scene"], st["frames"], st["seed"], st["tape"])
        st["gT"].zero_()
        st["gg"].zero_()
        L.cast_backward_mse(st["tape"], 1.0, st["target"], st["tvalid"], st["loss"], st["gT"], st["gg"])
        gp = L.build_tables_backward(st["params"], st["gT"])
        return {"loss": st["loss"], "gT": st["gT"], "gg": st["gg"], "gp": gp, **st["tape"]}
    st["params"].grad = st["gain"].grad = None
    I, valid = api.LidarCast.apply(st["params"], st["gain"], L, st["scene"], st["frames"], st["seed"], 0)
    loss = ((I - st["target"]).square() * (valid * st["tvalid"])).mean()
    loss.backward()
    return {"I": I, "valid": valid, "loss": loss, "gp": st["params"].grad, "gg": st["gain"].grad}


# ------------------------------------------------------------------- work

def _n_tris(case):
    if case["scene"] == "boxes":
        return 2 + 12 * case["size"]
    n = 2 * case["size"] ** 2
    if case["scene"] == "terrain":
        return n + (case["objects"] // 2) * 192 + (case["objects"] - case["objects"] // 2) * 280
    return n + 102 * min(case["objects"], int(2 * case["size"] // 28) ** 2)


def work(case):
    if case["kind"] == "adjoint":
        return {"bytes": 15.0 * case["beams"] + 3 * 4 * 91.0 * case["mats"], "flops": 12.0 * case["beams"]}
    n_tris = _n_tris(case)
    if case["kind"] == "rig":
        per = sum(ch * (case["az"] if ch > 16 else min(case["az"], 1800)) for ch in RIG)
    else:
        per = case["ch"] * (case["az"] if case["ch"] > 16 else min(case["az"], 1800))
    beams = per * case["frames"]
    rays = beams * case["sub"]
    # every ray: the boxes of one path down a 4-wide tree, two triangles, the model; every beam's direction once,
    # its record written once, one triangle per beam read (each triangle of the scene once at most)
    flops = rays * (math.log(max(n_tris, 4), 4) * 80.0 + 2 * 40.0 + 200.0)
    out = {"frame": 46 + (42 if case["dense"] else 0), "stream": 46, "rig": 46, "sweep": 42 + 27, "raster": 42,
           "fit": 15 + 5, "autograd": 15, "rebuild": 42}[case["kind"]]
    data = per * 12.0 + beams * out + 48.0 * min(n_tris, beams)
    if case["kind"] == "rebuild":
        # indices, vertices and labels in; leaf-ordered triangles, the binary and both wide trees out
        data += n_tris * (12 + 6 + 6 + 52 + 64 + 64 + 86)
        flops += n_tris * 200.0 * (1 + case["rounds"])
    if case["kind"] == "raster":
        data += 48.0 * n_tris
        flops += case["frames"] * n_tris * 60.0
    return {"bytes": float(data), "flops": float(flops)}


# ------------------------------------------------------------------- exact (64 bits)

def _mulhi(a, b):
    m = np.uint64(0xFFFFFFFF)
    s = np.uint64(32)
    al, ah, bl, bh = a & m, a >> s, b & m, b >> s
    mid = ah * bl + ((al * bl) >> s)
    mid2 = al * bh + (mid & m)
    return ah * bh + (mid >> s) + (mid2 >> s)


def _normal(seed, beam, frame):
    """Box-Muller on the first two words of Philox4x64-10, counter (beam, frame, 0, 0), key (seed, 0)."""
    with np.errstate(over="ignore"):
        x = [beam.astype(np.uint64), np.full(beam.shape, frame, np.uint64), np.zeros(beam.shape, np.uint64),
             np.zeros(beam.shape, np.uint64)]
        k = [np.uint64(seed), np.uint64(0)]
        M0, M1 = np.uint64(0xD2E7470EE14C6C93), np.uint64(0xCA5A826395121157)
        for r in range(10):
            if r:
                k = [k[0] + np.uint64(0x9E3779B97F4A7C15), k[1] + np.uint64(0xBB67AE8584CAA73B)]
            x = [_mulhi(M1, x[2]) ^ x[1] ^ k[0], M1 * x[2], _mulhi(M0, x[0]) ^ x[3] ^ k[1], M0 * x[0]]
    u = [((v >> np.uint64(11)).astype(np.float64) + 0.5) * 2.0 ** -53 for v in x[:2]]
    return np.sqrt(-2.0 * np.log(u[0])) * np.cos(2.0 * np.pi * u[1])


def _exact_frames(case, seed, table):
    """Dense records of every beam: brute force over the triangles, FP64 (one sensor, one ray a beam)."""
    verts, tris, mat, _, height = _scene(case, seed)
    n = case["frames"]
    poses = _poses(case, seed, height, n + 2)[1:n + 1]
    sn = _spinning(case["ch"], case["az"] if case["ch"] > 16 else min(case["az"], 1800), _d_max(case))
    d = np.stack([np.cos(sn.el_rad) * np.cos(sn.az_rad), np.cos(sn.el_rad) * np.sin(sn.az_rad), np.sin(sn.el_rad)], 1)
    dirs = torch.from_numpy(d.astype(np.float32)).to(DEV).double()
    tv = verts.double()[tris.long()]
    t_max = sn.d_max + 9.0 * sn.sigma
    mats = torch.from_numpy(mat.astype(np.int64)).to(DEV)
    rows = []
    for f in range(n):
        P = torch.from_numpy(poses[f].astype(np.float64)).to(DEV).reshape(3, 4)
        w = dirs @ P[:, :3].T
        v0 = tv[:, 0] - P[:, 3]
        e1, e2 = tv[:, 1] - tv[:, 0], tv[:, 2] - tv[:, 0]
        face = torch.linalg.cross(e1, e2)
        q0, q1, q2 = torch.linalg.cross(e2, v0), torch.linalg.cross(v0, e1), (v0 * face).sum(1)
        best = torch.full((len(w),), math.inf, device=DEV, dtype=torch.float64)
        idx = torch.full((len(w),), -1, device=DEV, dtype=torch.int64)
        step = max(1, (1 << 25) // max(1, len(tv)))
        for b in range(0, len(w), step):
            det = w[b:b + step] @ face.T
            u, v, t = (w[b:b + step] @ q0.T) / det, (w[b:b + step] @ q1.T) / det, q2 / det
            t = torch.where((u >= 0) & (v >= 0) & (u + v <= 1) & (t > 1e-4) & (t <= t_max), t, math.inf)
            best[b:b + step], idx[b:b + step] = t.min(1)
        hit = torch.isfinite(best)
        nrm = face[idx]
        nrm = nrm / nrm.norm(dim=1, keepdim=True)
        dn = (w * nrm).sum(1)
        nrm = torch.where((dn > 0)[:, None], -nrm, nrm)
        theta = torch.atan2(torch.linalg.cross(w, nrm).norm(dim=1), dn.abs()) * (180.0 / math.pi)
        i = theta.floor().clamp(max=89).long()
        fr = theta - i
        m = mats[idx]
        R = table[m, i] * (1 - fr) + table[m, i + 1] * fr
        z = torch.from_numpy(_normal(_noise(seed), np.arange(len(w)), f)).to(DEV)
        rng = best + sn.sigma * z
        valid = hit & (rng >= sn.r_min) & (rng <= sn.d_max) & (sn.RL_max * rng / sn.d_max <= R)
        zero = torch.zeros_like(best)
        rows.append({"valid": valid, "t": best, "range": torch.where(hit, rng, math.inf),
                     "intensity": torch.where(hit, R, zero), "R": R, "i": i, "fr": fr, "m": m,
                     "normal": torch.where(hit[:, None], nrm @ P[:, :3], zero[:, None]),
                     "theta_deg": torch.where(hit, theta, zero), "rf": hit.double()})
    return {k: torch.cat([r[k] for r in rows]) for k in rows[0]}


def _exact_table(params):
    k = torch.arange(91, device=DEV, dtype=torch.float64)
    a, s, w = (params.double()[:, j:j + 1] for j in range(3))
    return a * torch.cos(k * math.pi / 180.0) + s * torch.exp(-k * k / (2 * w * w))


def _exact_grad_table(m, i, fr, g, M):
    gT = torch.zeros(M * 91, device=DEV, dtype=torch.float64)
    gT.index_add_(0, m * 91 + i, g * (1 - fr))
    gT.index_add_(0, m * 91 + i + 1, g * fr)
    return gT.reshape(M, 91)


def exact(case, seed):
    kind = case["kind"]
    par = torch.from_numpy(_params(case, seed)).to(DEV)
    if kind == "adjoint":
        t = _tape(case, seed)
        # the reflectance table is an input of the adjoint: FP32, as the program holds it
        table = _exact_table(par).float().double()
        use = t["tape"]["valid"].bool()
        th = t["tape"]["theta_deg"].double()[use]
        i = th.floor().clamp(max=89).long()
        fr, m = th - i, t["tape"]["mat"].long()[use]
        g, rf = t["gI"].double()[use], t["tape"]["rf"].double()[use]
        R = table[m, i] * (1 - fr) + table[m, i + 1] * fr
        return [_exact_grad_table(m, i, fr, g * rf, case["mats"]), (g * rf * R).sum().reshape(1)]
    if kind not in ("frame", "rebuild", "autograd") or case["sub"] > 1:
        return None
    if _n_tris(case) * case["ch"] * case["az"] * case["frames"] > 8e9:
        return None
    if kind == "autograd":
        p = par.double().requires_grad_(True)
        table = _exact_table(p)
        r = _exact_frames(case, seed, table.detach())
        nb = len(r["t"])
        g = torch.Generator(device=DEV).manual_seed(seed)
        target = (torch.rand(nb, device=DEV, generator=g) * 0.9).double()
        tvalid = (torch.rand(nb, device=DEV, generator=g) < 0.9)
        use = (r["valid"] & tvalid).double()
        loss = ((r["intensity"] - target).square() * use).mean()
        gI = 2 * (r["intensity"] - target) * use / nb
        # the adjoint leaves out the beams that were not kept
        gI = gI * r["valid"]
        hit = torch.isfinite(r["t"])
        gT = _exact_grad_table(r["m"][hit], r["i"][hit], r["fr"][hit], gI[hit], case["mats"])
        table.backward(gT)
        return {"I": r["intensity"], "valid": None, "loss": loss, "gp": p.grad, "gg": (gI * r["R"])[hit].sum()}
    r = _exact_frames(case, seed, _exact_table(par))
    dense = {k: r.get(k) if k in ("t", "range", "intensity", "normal", "theta_deg", "rf") else None
             for k in ("valid", "tri", "t", "range", "intensity", "normal", "mat", "inst", "sub", "theta_deg", "rf")}
    if kind == "rebuild":
        return dense
    pts = {k: None for k in ("xyz", "range", "intensity", "normal", "material", "instance", "beam", "frame", "count")}
    return {**pts, **({"dense_" + k: v for k, v in dense.items()} if case["dense"] else {})}
