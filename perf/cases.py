"""Performance cases of the motion-focus path: what a program that uses this library has it do.

Every case is one way in which frames reach the library, at a size, a window and a storage type:

* ``live``     one open stream, one new frame per pass (a camera loop): ``mf_push_frames`` of one pose
               (host memory) with its depth plane (device), ``mf_get_maps`` of that frame;
* ``clip``     a whole clip at once: ``mf_reset_stream``, one push of every frame, one ``mf_get_maps``;
* ``wrapper``  the same through ``MotionFocusStream`` (torch in, torch and numpy out, points too);
* ``batches``  a clip as sliding inference batches in their own frames and depth scales, with shared
               frames: anchoring and depth alignment of every batch after the first;
* ``noalloc``  ``mf_render_noalloc``: the last frames of a pose window, nothing allocated;
* ``engine``   one tick of the batched engine: a push of every stream, then ``mf_engine_tick``.

Poses come from a walking camera (head sway and bob, turns, pose noise; ``walk`` = "steady" at a
constant pace, whose acceleration points are mostly out of view, or "pace", speeding up and slowing
down, whose points are mostly in view).  Depth is a ground plane with boxes in front of it, with
1 % noise, and 0 where the scene ends.
"""
import math
from fractions import Fraction

import numpy as np
import torch

import paper_2601_07154_gb300 as mf

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
CODES = {"f32": mf.MF_F32, "bf16": mf.MF_BF16, "f16": mf.MF_F16}
MODES = {"accel": mf.MF_MODE_ACCEL, "heading": mf.MF_MODE_HEADING}
RESOLUTIONS = ((640, 480), (1280, 720), (1920, 1080), (3840, 2160))
FPS = 30.0
LIVE_FRAMES = 900        # poses of a live or engine stream before its clip starts again
DEPTH_RING = 8           # depth planes a live stream cycles through
ENGINE_PLANES = 8        # depth and map planes per engine stream: at most this many frames a tick


def listed():
    """The cases that are always measured, smallest first."""
    return [
        # a camera loop at 320x240, one frame at a time: launches and latency are all there is
        _case("live_qvga", "live", 320, 240, 1, 8),
        # the same loop at 1080p: one frame is 25 MB of traffic, a few microseconds of memory time
        _case("live_1080p", "live", 1920, 1080, 1, 16, walk="pace"),
        # a plugin with a fixed memory budget that renders the last half second of a 640x480 camera
        _case("noalloc_vga_f16", "noalloc", 640, 480, 16, 12, mode="heading", storage="f16"),
        # a 2 s clip at 320x240 through the torch wrapper, motion points returned as well
        _case("clip_qvga", "wrapper", 320, 240, 64, 8),
        # two depth-model batches of 60 frames at its 504-pixel input size, 10 frames shared,
        # intrinsics of the 1080p camera, depth scales aligned
        _case("batches_504", "batches", 504, 280, 60, 16, walk="pace", overlap=10, calib=1920),
        # widescreen 480p: an odd width, so no two rows start at the same alignment
        _case("clip_480p_odd", "clip", 853, 480, 120, 12, walk="pace"),
        # maps scaled to peak at 1 (display)
        _case("clip_720p_max", "clip", 1280, 720, 120, 16, walk="pace", norm="max"),
        # 10 s of 1080p at the default options: the benchmark's stream
        _case("clip_1080p", "clip", 1920, 1080, 300, 16),
        # the longest window with every motion point in view, 16-bit storage
        _case("clip_1080p_bf16", "clip", 1920, 1080, 150, 32, mode="heading", storage="bf16"),
        # the largest frames
        _case("clip_2160p_f16", "clip", 3840, 2160, 24, 24, walk="pace", storage="f16"),
        # a server's tick at 128 live streams of mixed sizes and windows, one frame each
        _case("engine_live", "engine", 0, 0, 1, 0, walk="pace", streams=128),
        # the batched workload: 64 mixed streams, 8 frames each, 16-bit storage
        _case("engine_mixed_bf16", "engine", 0, 0, 8, 0, walk="pace", streams=64, storage="bf16"),
    ]


def _case(name, kind, width, height, frames, window, mode="accel", storage="f32", walk="steady",
          norm="count", smooth=15, streams=1, overlap=0, calib=0):
    c = dict(kind=kind, width=width, height=height, frames=frames, window=window, mode=mode,
             storage=storage, walk=walk, norm=norm, smooth=smooth, streams=streams, overlap=overlap,
             calib=calib)
    return dict(c, name=name) if name else c


def draw(rng):
    """One more case of the same ranges: frames of 64x48 to 3840x2160 (odd sizes too), windows 1 to 32,
    1 to 300 frames, every storage type, mode and normalisation."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("live", "noalloc", "wrapper", "batches", "clip", "clip", "clip", "engine"))
    storage = rng.choice(("f32", "f32", "bf16", "f16"))
    mode, walk = rng.choice(("accel", "accel", "heading")), rng.choice(("steady", "pace"))
    window = rng.randint(1, 32)
    smooth = rng.choice((3, 7, 15, 15, 31))
    if kind == "engine":
        streams = log_int(4, 128)
        frames = rng.randint(1, max(1, min(ENGINE_PLANES, 256 // streams)))
        return _case(None, kind, 0, 0, frames, 0, mode, storage, walk, "count", smooth, streams)
    width = log_int(64, 3840)
    height = max(48, int(round(width / rng.choice((4 / 3, 16 / 9, 16 / 9)))))
    norm = rng.choice(("count", "count", "count", "max"))
    most = max(1, min(300, 300 * 1920 * 1080 // (width * height)))
    if kind == "live":
        return _case(None, kind, width, height, 1, window, mode, storage, walk, norm, smooth)
    if kind == "batches":
        frames = rng.randint(8, 60)
        frames = max(4, min(frames, most // 2))
        return _case(None, kind, width, height, frames, window, mode, storage, walk, norm, smooth,
                     overlap=rng.randint(1, max(1, frames // 4)), calib=rng.choice((0, 1920)))
    most = min(most, 128 if kind == "noalloc" else 300)
    return _case(None, kind, width, height, log_int(1, most), window, mode, storage, walk, norm, smooth)


# ---------------------------------------------------------------- inputs --
def _rng(seed, *more):
    return np.random.default_rng([int(seed), *more])


def walker(n, rng, pace):
    """(n, 3, 4) world-to-camera poses of a walking camera at 30 fps."""
    t = np.arange(n) / FPS

    def segments(lo, hi, value):
        out, k = np.zeros(n), 0
        while k < n:
            m = max(1, int(rng.uniform(lo, hi) * FPS))
            out[k:k + m] = value()
            k += m
        return out

    yaw = np.concatenate([[0.0], np.cumsum(segments(1.0, 3.0, lambda: math.radians(rng.uniform(-45, 45))))[:-1] / FPS])
    speed = np.full(n, 1.4)
    if pace:
        sign = [1.0]

        def acc():
            sign[0] = -sign[0]
            return -sign[0] * 1.5 * rng.uniform(0.6, 1.0)
        a = segments(1.0, 2.5, acc)
        for k in range(1, n):
            speed[k] = min(3.0, max(0.5, speed[k - 1] + a[k - 1] / FPS))
    step = np.stack([speed * np.sin(yaw), np.zeros(n), speed * np.cos(yaw)], 1) / FPS
    centre = np.concatenate([np.zeros((1, 3)), np.cumsum(step, 0)[:-1]]) + rng.normal(0, 0.01, (n, 3))
    yaw = yaw + math.radians(10) * np.sin(2 * math.pi * 0.5 * t)
    pitch = math.radians(3) * np.sin(2 * math.pi * 2.0 * t)
    rot = _axis_angle(rng.normal(0, math.radians(0.5), (n, 3))) @ _rot_y(yaw) @ _rot_x(pitch)
    w2c = rot.transpose(0, 2, 1)
    return np.ascontiguousarray(np.concatenate([w2c, -(w2c @ centre[:, :, None])], 2))


def _rot_y(a):
    c, s, o, z = np.cos(a), np.sin(a), np.ones_like(a), np.zeros_like(a)
    return np.stack([c, z, s, z, o, z, -s, z, c], -1).reshape(-1, 3, 3)


def _rot_x(a):
    c, s, o, z = np.cos(a), np.sin(a), np.ones_like(a), np.zeros_like(a)
    return np.stack([o, z, z, z, c, -s, z, s, c], -1).reshape(-1, 3, 3)


def _axis_angle(w):
    th = np.maximum(np.linalg.norm(w, axis=1), 1e-300)[:, None, None]
    k = w[:, None, :] / th
    z = np.zeros(len(w))
    kx = np.stack([z, -k[:, 0, 2], k[:, 0, 1], k[:, 0, 2], z, -k[:, 0, 0], -k[:, 0, 1], k[:, 0, 0], z], -1).reshape(-1, 3, 3)
    return np.eye(3) + np.sin(th) * kx + (1 - np.cos(th)) * (kx @ kx)


def depth_planes(n, width, height, seed, dtype, out=None, scale=1.0, noise_seed=0):
    """n depth planes: ground 1.6 m below the camera, a dozen boxes, nothing beyond 200 m."""
    rng = _rng(seed, 7)
    dev = torch.device("cuda")
    out = torch.empty((n, height, width), dtype=dtype, device=dev) if out is None else out
    rows = torch.arange(height, device=dev, dtype=torch.float32)[:, None]
    boxes = [(rng.uniform(0, 1), rng.uniform(0.02, 0.15), rng.uniform(0.25, 0.5), rng.uniform(0.5, 0.9), rng.uniform(1.0, 20.0))
             for _ in range(12)]
    gen = torch.Generator(device=dev).manual_seed(int(seed) * 7919 + noise_seed)
    noise = 1 + 0.01 * torch.randn((height, width), device=dev, generator=gen)
    for k in range(n):
        slope = (rows - height / 2) / (0.8 * width) + 0.05 * math.sin(0.4 * k)
        ground = torch.where(slope > 1.6 / 200, 1.6 / slope.clamp(min=1e-3), torch.zeros_like(slope))
        plane = ground.expand(height, width).clone()
        for x, w, top, bottom, z in sorted(boxes, key=lambda b: -b[4]):
            x0 = int((x + 0.004 * k) % 1.0 * width)
            plane[int(top * height):int(bottom * height) + 1, x0:x0 + 1 + int(w * width)] = z * (1 - 0.002 * k)
        out[k] = (plane * noise.roll(17 * k, 1) / scale).to(dtype)
    return out


def _intrinsics(case, width, height):
    """(fx, fy, cx, cy) at the calibration resolution and that resolution (0: the map's)."""
    if case["calib"]:
        cw = case["calib"]
        ch = int(round(cw * height / width))
        return np.array([0.78125 * cw, 0.78125 * cw, cw / 2.0, ch / 2.0]), (cw, ch)
    return np.array([0.8 * width, 0.8 * width, width / 2.0, height / 2.0]), (0, 0)


def _streams(case):
    """(width, height, window) of every engine stream: the size mix of the batched workload."""
    return [RESOLUTIONS[i % 4] + (8 + (i * 7) % 25,) for i in range(case["streams"])]


def _desc(case, width, height, window, stream):
    _, (cw, ch) = _intrinsics(case, width, height)
    dt = CODES[case["storage"]]
    local = case["kind"] == "batches"
    return mf.mf_stream_desc_init(
        width=width, height=height, calib_width=cw, calib_height=ch, window=window,
        smooth_len=case["smooth"], mode=MODES[case["mode"]],
        pose_frame=mf.MF_POSES_BATCH_LOCAL if local else mf.MF_POSES_WORLD, overlap=case["overlap"],
        depth_dtype=dt, map_dtype=dt, max_pending=512,
        flags=mf.MF_FLAG_DEPTH_ALIGN if local else 0,
        normalize=mf.MF_NORM_MAX if case["norm"] == "max" else mf.MF_NORM_COUNT, cuda_stream=stream)


def _info_views(buf, n):
    """The fields of n device records by type, as views of the buffer."""
    i4, f4, i8, f8 = (buf.view(t).view(n, -1) for t in (torch.int32, torch.float32, torch.int64, torch.float64))
    return {"frame": i8[:, 0], "flags": i4[:, 2:6], "focus": f8[:, 3:5], "pixels": i4[:, 10:14],
            "map_max": f4[:, 14], "depth_scale": f4[:, 15]}


class _Stream:
    """An open mf_stream, closed with the state that holds it."""

    def __init__(self, desc):
        self.handle = mf.mf_open_stream(desc)

    def __del__(self):
        if self.handle:
            mf.mf_close_stream(self.handle)
            self.handle = None


def _local_batches(case, poses, seed):
    """The clip's two batches in frames of their own: [(poses, depth scale), ...]."""
    n, o = case["frames"], case["overlap"]
    out = []
    for b, lo in enumerate((0, n - o)):
        rng = _rng(seed, 11, b)
        c = 1.0 if b == 0 else float(rng.uniform(0.6, 1.6))
        H = np.eye(4)
        if b:
            H[:3, :3] = _rot_y(np.array([rng.uniform(-math.pi, math.pi)]))[0]
            H[:3, 3] = rng.uniform(-5, 5, 3)
        L = poses[lo:lo + n] @ H
        L[:, :, 3] /= c
        out.append((np.ascontiguousarray(L), c))
    return out


def _batch_poses(case, seed):
    return walker(2 * case["frames"] - case["overlap"], _rng(seed, 1), case["walk"] == "pace")


def prepare(case, seed):
    kind, dev = case["kind"], torch.device("cuda")
    w, h, n, win, dt = case["width"], case["height"], case["frames"], case["window"], DTYPES[case["storage"]]
    pace = case["walk"] == "pace"
    handle = torch.cuda.current_stream().cuda_stream or 1
    if kind == "engine":
        return _prepare_engine(case, seed)
    K, calib = _intrinsics(case, w, h)
    st = {"kind": kind, "n": n, "K": K}
    if kind == "batches":
        o = case["overlap"]
        poses = _batch_poses(case, seed)
        st["pushes"] = []
        for b, (L, c) in enumerate(_local_batches(case, poses, seed)):
            depth = torch.empty((n, h, w), dtype=dt, device=dev)
            lo = b * (n - o)
            depth_planes(lo + n, w, h, seed, torch.float32, _Tail(depth, lo), c, 1 + b)
            emit = n - (o if b else 0)
            st["pushes"].append((torch.from_numpy(L).to(dev), depth, lo + (o if b else 0), emit))
        total = 2 * n - o
    else:
        total = n
    st["M"] = torch.zeros((total, h, w), dtype=dt, device=dev)
    st["G"] = torch.zeros_like(st["M"])
    st["info"] = torch.zeros(total * 64, dtype=torch.uint8, device=dev)
    st["out"] = {"M": st["M"], "G": st["G"], "info": _info_views(st["info"], total)}
    if kind == "live":
        st["poses"] = walker(LIVE_FRAMES, _rng(seed, 1), pace)
        st["depth"] = list(depth_planes(DEPTH_RING, w, h, seed, dt))
        st["stream"] = _Stream(_desc(case, w, h, win, handle))
        hist = win + case["smooth"] - 2
        if hist:
            mf.mf_push_frames(st["stream"].handle, hist, st["poses"], None, K)
            mf.mf_get_maps(st["stream"].handle, hist)
        st["at"] = hist
    elif kind == "noalloc":
        poses = walker(n + win + case["smooth"] - 2, _rng(seed, 1), pace)
        st["poses"] = torch.from_numpy(poses).to(dev)
        st["depth"] = depth_planes(n, w, h, seed, dt)
        st["desc"] = _desc(case, w, h, win, handle)
    elif kind == "wrapper":
        st["poses"] = torch.from_numpy(walker(n, _rng(seed, 1), pace)).to(dev)
        st["depth"] = depth_planes(n, w, h, seed, dt)
        st["stream"] = mf.MotionFocusStream(w, h, window=win, smooth_len=case["smooth"], mode=case["mode"],
                                            depth_dtype=dt, map_dtype=dt, normalize=case["norm"])
    else:
        if kind == "clip":
            st["poses"] = torch.from_numpy(walker(n, _rng(seed, 1), pace)).to(dev)
            st["depth"] = depth_planes(n, w, h, seed, dt)
        st["stream"] = _Stream(_desc(case, w, h, win, handle))
    torch.cuda.synchronize()
    return st


class _Tail:
    """The last planes of a longer clip: planes before `first` are not kept."""

    def __init__(self, planes, first):
        self.planes, self.first = planes, first

    def __setitem__(self, k, plane):
        if k >= self.first:
            self.planes[k - self.first] = plane


def _prepare_engine(case, seed):
    dev, dt, n = torch.device("cuda"), DTYPES[case["storage"]], case["frames"]
    streams = _streams(case)
    total = sum(n * w * h for w, h, _ in streams)
    M = torch.zeros(total, dtype=dt, device=dev)
    G = torch.zeros_like(M)
    info = torch.zeros(len(streams) * n * 64, dtype=torch.uint8, device=dev)
    eng = mf.MotionFocusEngine(depth_dtype=dt, map_dtype=dt)
    pushes = np.zeros(len(streams), mf.PUSH_DTYPE)
    depth = torch.empty(total, dtype=dt, device=dev)
    planes = {}
    for i, (w, h, win) in enumerate(streams):
        if (w, h) not in planes:
            planes[w, h] = depth_planes(n, w, h, seed, dt)
    keep, at, hist = [], 0, 48
    for i, (w, h, win) in enumerate(streams):
        K, _ = _intrinsics(case, w, h)
        poses = walker(LIVE_FRAMES, _rng(seed, 1, i), case["walk"] == "pace")
        slot = eng.add_stream(w, h, window=win, smooth_len=case["smooth"], mode=case["mode"])
        depth[at:at + n * w * h].view(n, h, w).copy_(planes[w, h])
        size = dt.itemsize
        pushes[i] = (slot, hist // 2, poses.ctypes.data, 0, K.ctypes.data, 0, 0, 0, 0)
        keep.append((poses, K, at * size))
        at += n * w * h
    base = pushes["poses"].copy()
    for half in range(2):                             # the streams' first frames: their windows are full
        pushes["poses"] = base + half * (hist // 2) * 96
        mf.mf_engine_submit_batch(eng.handle, pushes)
        eng.wait(eng.tick())
    for i, (poses, K, off) in enumerate(keep):
        pushes[i]["n"] = n
        pushes[i]["depth"] = depth.data_ptr() + off
        pushes[i]["focus_map"] = M.data_ptr() + off
        pushes[i]["guided_depth"] = G.data_ptr() + off
        pushes[i]["info"] = info.data_ptr() + i * n * 64
    torch.cuda.synchronize()
    return {"kind": "engine", "n": n, "engine": eng, "pushes": pushes, "base": base, "at": hist, "keep": keep,
            "depth": depth, "M": M, "G": G, "info": info,
            "out": {"M": M, "G": G, "info": _info_views(info, len(streams) * n)}}


# ---------------------------------------------------------------- the pass --
def run(state):
    kind, n = state["kind"], state["n"]
    if kind == "engine":
        at = state["at"] if state["at"] + n <= LIVE_FRAMES else 0
        state["pushes"]["poses"] = state["base"] + at * 96
        state["at"] = at + n
        mf.mf_engine_submit_batch(state["engine"].handle, state["pushes"])
        state["engine"].tick()
        return state["out"]
    if kind == "noalloc":
        mf.mf_render_noalloc(state["desc"], len(state["poses"]), state["poses"], n, state["depth"], state["K"],
                             state["M"], state["G"], state["info"])
        return state["out"]
    if kind == "wrapper":
        s = state["stream"]
        s.reset()
        s.push(state["poses"], state["depth"], state["K"])
        M, G, info, points = s.get_maps(out=(state["M"], state["G"]))
        return {"M": M, "G": G, "info": {"flags": np.stack([info[k] for k in ("status", "n_valid", "valid_mask", "focus_valid")], 1).astype(np.int64),
                                         "focus": np.stack([info["focus_u"], info["focus_v"]], 1),
                                         "pixels": np.stack([info[k] for k in ("focus_px_x", "focus_px_y", "argmax_x", "argmax_y")], 1),
                                         "map_max": info["map_max"]},
                "points": {"uvs": np.stack([points[k] for k in ("u", "v", "sigma", "s")], 2), "valid": points["valid"]}}
    s = state["stream"].handle
    if kind == "live":
        at = state["at"] if state["at"] < LIVE_FRAMES else 0
        state["at"] = at + 1
        mf.mf_push_frames(s, 1, state["poses"][at], state["depth"][at % DEPTH_RING], state["K"])
        mf.mf_get_maps(s, 1, state["M"], state["G"], state["info"])
        return state["out"]
    mf.mf_reset_stream(s)
    if kind == "clip":
        mf.mf_push_frames(s, n, state["poses"], state["depth"], state["K"])
        mf.mf_get_maps(s, n, state["M"], state["G"], state["info"])
        return state["out"]
    for poses, depth, first, emit in state["pushes"]:
        mf.mf_push_frames(s, n, poses, depth, state["K"])
        mf.mf_get_maps(s, emit, state["M"][first:first + emit], state["G"][first:first + emit],
                       state["info"][first * 64:(first + emit) * 64])
    return state["out"]


# ------------------------------------------------------------- exact values --
def _weights(k, mode):
    """Least-squares derivative weights over the k newest samples (exact rationals, rounded once)."""
    deg = 2 if k >= 3 else 1
    rows = [[Fraction(-j) ** e for e in range(deg + 1)] for j in range(k)]
    a = [[sum(r[i] * r[j] for r in rows) for j in range(deg + 1)] + [Fraction(int(i == (2 if mode == "accel" else 1)))]
         for i in range(deg + 1)]
    for i in range(deg + 1):
        a[i] = [v / a[i][i] for v in a[i]]
        for r in range(deg + 1):
            if r != i:
                a[r] = [x - a[r][i] * y for x, y in zip(a[r], a[i])]
    c = [row[-1] * (2 if mode == "accel" else 1) for row in a]
    return np.array([float(sum(x * y for x, y in zip(c, r))) for r in rows])


def _motion_points(poses, frames, K, case, width, height, window, calib):
    """(u, v, sigma, s, valid) of the given frames of a pose sequence, each (len(frames), window)."""
    ks = case["smooth"]
    wts = _weights(ks, case["mode"])
    centre = -np.einsum("nji,nj->ni", poses[:, :, :3], poses[:, :, 3])
    fx, fy, cx, cy = K
    if calib[0]:
        sx, sy = width / calib[0], height / calib[1]
        fx, cx, fy, cy = fx * sx, (cx + 0.5) * sx - 0.5, fy * sy, (cy + 0.5) * sy - 0.5
    out = np.zeros((4, len(frames), window))
    valid = np.zeros((len(frames), window), bool)
    for f, g in enumerate(frames):
        j0 = max(0, g - window - ks + 2)
        q = (centre[j0:g + 1] - centre[g]) @ poses[g, :, :3].T
        rho = np.linalg.norm(q, axis=1).max()
        if not (rho > 0 and rho > 1e-12 * np.linalg.norm(centre[j0:g + 1], axis=1).max()):
            continue
        d = np.zeros((window, 3))
        for s in range(window):
            i = g - window + 1 + s
            if i - ks + 1 >= 0:
                d[s] = wts @ q[i - j0 - ks + 1:i - j0 + 1][::-1]
        nd = np.linalg.norm(d, axis=1)
        ok = (nd > 1e-9 * rho) & (np.abs(d[:, 2]) > 1e-3 * nd)
        if not ok.any():
            continue
        valid[f] = ok
        s = np.clip(nd[ok] / nd[ok].mean(), 0.25, 4.0)
        out[:, f, ok] = np.stack([cx + fx * d[ok, 0] / d[ok, 2], cy + fy * d[ok, 1] / d[ok, 2], 0.1 * fx * s, s])
    return out, valid


def _maps(pts, valid, width, height, depth, norm, scale=None):
    """M, G and the map maximum in 64 bits; `depth` (n, height, width)."""
    dev = depth.device
    u, v, sig, _ = (torch.from_numpy(np.ascontiguousarray(a)).to(dev) for a in pts)
    ok = torch.from_numpy(valid).to(dev)
    c = torch.where(ok, 0.5 / sig.clamp(min=1e-300) ** 2, torch.zeros_like(sig))
    xs = torch.arange(width, device=dev, dtype=torch.float64)
    ys = torch.arange(height, device=dev, dtype=torch.float64)
    count = ok.sum(1).clamp(min=1).double()
    M = torch.empty(depth.shape, dtype=torch.float64, device=dev)
    G = torch.empty_like(M)
    top = torch.empty(len(depth), dtype=torch.float64, device=dev)
    for f in range(len(depth)):
        ex = torch.exp(-(xs[None] - u[f, :, None]) ** 2 * c[f, :, None])
        ey = torch.exp(-(ys[None] - v[f, :, None]) ** 2 * c[f, :, None]) * (ok[f, :, None] / count[f])
        M[f] = ey.T @ ex
        top[f] = M[f].max()
        if norm == "max" and top[f] >= 2.0 ** -20:
            M[f] /= top[f].clone()
            top[f] = 1.0
        D = depth[f].double() * (1.0 if scale is None else scale[f])
        G[f] = M[f] * torch.where(D > 0, (1.0 / D.clamp(min=1e-300)).clamp(max=1.0), torch.zeros_like(D))
    return M, G, top


def _exact_info(pts, valid, top, scale=None, wrapper=False):
    focus = np.stack([pts[0][:, -1], pts[1][:, -1]], 1)
    info = {"flags": None, "focus": focus, "pixels": None, "map_max": top}
    if not wrapper:
        info.update(frame=None, depth_scale=np.ones(len(focus)) if scale is None else scale)
    return info


def exact(case, seed):
    kind, n, win, dt = case["kind"], case["frames"], case["window"], DTYPES[case["storage"]]
    w, h, pace = case["width"], case["height"], case["walk"] == "pace"
    if kind == "engine":
        Ms, Gs, foci, tops = [], [], [], []
        planes = {}
        for i, (w, h, win) in enumerate(_streams(case)):
            K, calib = _intrinsics(case, w, h)
            poses = walker(LIVE_FRAMES, _rng(seed, 1, i), pace)
            pts, valid = _motion_points(poses, range(48, 48 + n), K, case, w, h, win, calib)
            if (w, h) not in planes:
                planes[w, h] = depth_planes(n, w, h, seed, dt)
            M, G, top = _maps(pts, valid, w, h, planes[w, h], "count")
            Ms.append(M.reshape(-1)), Gs.append(G.reshape(-1)), tops.append(top)
            foci.append(np.stack([pts[0][:, -1], pts[1][:, -1]], 1))
        return {"M": torch.cat(Ms), "G": torch.cat(Gs),
                "info": {"frame": None, "flags": None, "focus": np.concatenate(foci), "pixels": None,
                         "map_max": torch.cat(tops), "depth_scale": np.ones(len(foci) * n)}}
    K, calib = _intrinsics(case, w, h)
    scale = None
    if kind == "batches":
        poses, depth, scale = _exact_batches(case, seed)
        frames = range(len(poses))
    elif kind == "live":
        poses = walker(LIVE_FRAMES, _rng(seed, 1), pace)
        at = win + case["smooth"] - 2
        frames, depth = [at], depth_planes(DEPTH_RING, w, h, seed, dt)[at % DEPTH_RING][None]
    else:
        hist = win + case["smooth"] - 2 if kind == "noalloc" else 0
        poses = walker(n + hist, _rng(seed, 1), pace)
        frames, depth = range(hist, hist + n), depth_planes(n, w, h, seed, dt)
    pts, valid = _motion_points(poses, frames, K, case, w, h, win, calib)
    M, G, top = _maps(pts, valid, w, h, depth, case["norm"], scale)
    out = {"M": M, "G": G, "info": _exact_info(pts, valid, top, scale, kind == "wrapper")}
    if kind == "wrapper":
        out["points"] = {"uvs": np.stack(list(pts), 2), "valid": None}
    return out


def _exact_batches(case, seed):
    """World poses, depth planes and depth scales of the emitted frames of both batches."""
    n, o, w, h, dt = case["frames"], case["overlap"], case["width"], case["height"], DTYPES[case["storage"]]
    dev = torch.device("cuda")
    (A, ca), (B, cb) = _local_batches(case, _batch_poses(case, seed), seed)
    planes = []
    for b, c in enumerate((ca, cb)):
        d = torch.empty((n, h, w), dtype=dt, device=dev)
        depth_planes(b * (n - o) + n, w, h, seed, torch.float32, _Tail(d, b * (n - o)), c, 1 + b)
        planes.append(d)
    prev, cur = planes[0][n - o:].float(), planes[1][:o].float()
    ok = (prev > 0) & (cur > 0) & torch.isfinite(prev) & torch.isfinite(cur)
    ratios = (prev[ok] / cur[ok]).sort().values
    s = float(ratios[(len(ratios) - 1) // 2]) if len(ratios) else 1.0
    B = B.copy()
    B[:, :, 3] *= s
    Ta, La = np.eye(4), np.eye(4)
    Ta[:3], La[:3] = A[n - 1], B[o - 1]
    R = Ta[:3, :3].T @ La[:3, :3]
    H = np.eye(4)
    H[:3, :3] = _rot_y(np.array([math.atan2(R[0, 2] - R[2, 0], R[0, 0] + R[2, 2])]))[0]
    H[:3, 3] = -Ta[:3, :3].T @ Ta[:3, 3] + H[:3, :3] @ (La[:3, :3].T @ La[:3, 3])
    world = np.concatenate([A, B[o:] @ np.linalg.inv(H)])
    return world, torch.cat([planes[0], planes[1][o:]]), np.concatenate([np.ones(n), np.full(n - o, s)])


def work(case):
    """Every depth plane read once, both maps and the records written once; one multiply-add per motion
    point and pixel, and the weight of the guided depth."""
    kind, n = case["kind"], case["frames"]
    size = DTYPES[case["storage"]].itemsize
    if kind == "engine":
        streams = _streams(case)
    else:
        streams = [(case["width"], case["height"], case["window"])]
    frames = 2 * n - case["overlap"] if kind == "batches" else n
    px = sum(frames * w * h for w, h, _ in streams)
    nbytes = 3 * px * size + frames * len(streams) * (96 + 64)
    flops = sum(frames * w * h * (2 * win + 3) for w, h, win in streams)
    if kind == "batches":                  # both sides of the shared frames are compared as well
        nbytes += 2 * case["overlap"] * case["width"] * case["height"] * size
    return {"bytes": nbytes, "flops": flops}
