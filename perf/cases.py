"""The calls that users of this detector and tracker make, for measuring them.

listed()  a camera frame, batches of cameras, large stills, the parameter
          sweep, the tracker, the frontend loop, host buffers and serving
draw(rng) one more case of the same ranges
prepare / run / work / exact: the inputs, one pass, what a pass cannot do
          without, and its values in 64 bits

Frames are drawn on the GPU after the recipe of the package's synthetic
frames: value noise on an 8-pixel lattice (mean 128, std 30) with rectangles
and triangles of uniform intensity; tracker pairs are sums of plane waves with
a sub-pixel motion and a gain and offset between the two frames.

Detector outputs are whole numbers, defined bit by bit, so exact() has no
value for them; it gives the tracker's positions and intensity parameters.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2003_13493_gb300 import synth, vio

MIXED = synth.MIXED_SIZES
SAD_B, SAD_A, MT = vio.SCORE_SAD_B, vio.SCORE_SAD_A, vio.SCORE_MT


def listed():
    mixed = dict(sizes="mixed", w=1920, h=1080, shapes=40)
    return [
        # one 752x480 camera frame per call (EuRoC's size), three levels: the latency of a live camera
        dict(name="frame_752", kind="detect", sizes="same", w=752, h=480, frames=1, shapes=40, levels=3, thresh=20,
             arc=9, cell=32, score=SAD_B, radius=1),
        # a batch of 64 frames from cameras of four resolutions, as bench.py's default workload
        dict(name="mixed64", kind="detect", frames=64, levels=3, thresh=15, arc=9, cell=32, score=SAD_B, radius=1,
             **mixed),
        # crops of odd sizes: rows that end anywhere, addresses and pitches that TMA cannot read in place
        dict(name="ragged24", kind="detect", sizes="ragged", w=1021, h=765, frames=24, shapes=40, levels=4, thresh=12,
             arc=9, cell=32, score=SAD_B, radius=1),
        # the threshold score (MT), a few frames of each camera
        dict(name="mixed16_mt", kind="detect", frames=16, levels=3, thresh=15, arc=9, cell=64, score=MT, radius=1,
             **mixed),
        # the widest NMS window, one level, FAST-10: features far apart
        dict(name="mixed16_nms9", kind="detect", frames=16, levels=1, thresh=10, arc=10, cell=32, score=SAD_B,
             radius=4, **mixed),
        # 4K stills with the strict arc (FAST-12) and the arc's own score (SAD-A)
        dict(name="large8_fast12", kind="detect", sizes="same", w=3840, h=2160, frames=8, shapes=400, levels=4,
             thresh=20, arc=12, cell=64, score=SAD_A, radius=1),
        # 4K stills, the whole grid of settings (bench.py's large4k workload): choosing thresholds
        dict(name="large32_sweep", kind="sweep", sizes="same", w=3840, h=2160, frames=32, shapes=400, levels=4,
             thresholds="5 10 20 40", arcs="12 9", cell=64),
        # tracking one camera's 100 features (Table VI's setting)
        dict(name="track_100", kind="track", w=752, h=480, pairs=1, grid_x=10, grid_y=10, levels=3, iters=30, model=3),
        # tracking 64 cameras with 256 features each in one call
        dict(name="track_64x256", kind="track", w=752, h=480, pairs=64, grid_x=16, grid_y=16, levels=3, iters=30,
             model=3),
        # the frontend of one camera: detect in the new frame, track the previous frame's features into it
        dict(name="frontend_752", kind="frontend", w=752, h=480, levels=3, thresh=10, arc=9, cell=32),
        # 64 frames in host memory, results wanted in host memory, one call at a time
        dict(name="host_mixed64", kind="host", frames=64, levels=3, thresh=15, arc=9, cell=32, score=SAD_B, radius=1,
             **mixed),
        # 16 cameras hand in a frame each and wait for the results
        dict(name="serve16", kind="serve", frames=16, levels=3, thresh=15, arc=9, cell=32, **mixed),
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    kind = rng.choice(["detect"] * 6 + ["sweep", "track", "track", "frontend", "host", "serve"])
    w = _log(rng, 160, 3840)
    h = max(120, min(2160, round(w * rng.uniform(0.5, 0.8))))
    cell = rng.choice([32, 32, 64])
    if kind == "track":
        w, h = _log(rng, 320, 1920), _log(rng, 240, 1080)
        pairs = _log(rng, 1, 64)
        while pairs * w * h > 64 * 752 * 480:
            pairs = max(1, pairs // 2)
        return dict(kind=kind, w=w, h=h, pairs=pairs, grid_x=rng.randint(4, 16), grid_y=rng.randint(4, 16),
                    levels=rng.randint(2, 4), iters=rng.choice([10, 30]), model=rng.choice([1, 2, 3, 3]))
    if kind == "frontend":
        return dict(kind=kind, w=_log(rng, 320, 1920), h=_log(rng, 240, 1080), levels=rng.randint(2, 4),
                    thresh=rng.randint(8, 40), arc=rng.choice([9, 10, 12]), cell=cell)
    sizes = rng.choice(["same", "mixed", "ragged"]) if kind == "detect" else rng.choice(["same", "mixed"])
    if sizes == "mixed":
        w, h = 1920, 1080
    area = 915000 if sizes == "mixed" else w * h  # the mixed sizes' mean
    frames = _log(rng, 1, 64)
    while frames * area > 60e6:
        frames = max(1, frames // 2)
    c = dict(kind=kind, sizes=sizes, w=w, h=h, frames=frames, shapes=max(20, 40 * w * h // 2000000),
             levels=rng.randint(1, 4), cell=cell)
    if kind == "sweep":
        ts = sorted(rng.sample([5, 8, 10, 15, 20, 30, 40, 60], rng.randint(2, 4)))
        c.update(thresholds=" ".join(map(str, ts)), arcs=rng.choice(["9", "12 9", "10"]))
        return c
    c.update(thresh=rng.randint(5, 40), arc=rng.choice([9, 9, 10, 11, 12]))
    if kind != "serve":
        c.update(score=rng.choice([SAD_B, SAD_B, SAD_A, MT]), radius=rng.choice([1, 1, 1, 2, 3, 4]))
    return c


# ---- frames -----------------------------------------------------------------


def _sizes(case):
    n, w, h = case["frames"], case["w"], case["h"]
    if case["sizes"] == "mixed":
        return [MIXED[i * len(MIXED) // n if n >= len(MIXED) else i] for i in range(n)]
    if case["sizes"] == "ragged":
        return [(w - 7 * (i % 9), h - 5 * (i % 7)) for i in range(n)]
    return [(w, h)] * n


def _scene(w, h, n_shapes, gen, rs):
    """One h x w uint8 frame."""
    lat = 128 + 30 * torch.randn((1, 1, (h + 7) // 8 + 1, (w + 7) // 8 + 1), generator=gen, device="cuda")
    img = torch.nn.functional.interpolate(lat, scale_factor=8, mode="bilinear", align_corners=False)[0, 0, :h, :w]
    img = img.round().clamp_(0, 255).to(torch.uint8)
    top = max(8, min(w, h) // 4) + 1
    for _ in range(n_shapes):
        x0, y0, fill = rs.randint(0, w), rs.randint(0, h), int(rs.randint(0, 256))
        if rs.randint(0, 2):
            img[y0:y0 + rs.randint(8, top), x0:x0 + rs.randint(8, top)] = fill
            continue
        e = rs.randint(8, top)
        (ax, ay), (bx, by), (cx, cy) = [(x0 + rs.randint(-e, e + 1), y0 + rs.randint(-e, e + 1)) for _ in range(3)]
        area = (bx - ax) * (cy - ay) - (by - ay) * (cx - ax)
        xl, xh = max(0, min(ax, bx, cx)), min(w, max(ax, bx, cx) + 1)
        yl, yh = max(0, min(ay, by, cy)), min(h, max(ay, by, cy) + 1)
        if area == 0 or xl >= xh or yl >= yh:
            continue
        px = torch.arange(xl, xh, device="cuda")[None, :]
        py = torch.arange(yl, yh, device="cuda")[:, None]
        s = 1 if area > 0 else -1
        hit = None
        for x1, y1, x2, y2 in ((ax, ay, bx, by), (bx, by, cx, cy), (cx, cy, ax, ay)):
            side = s * ((x2 - x1) * (py - y1) - (y2 - y1) * (px - x1)) >= 0
            hit = side if hit is None else hit & side
        img[yl:yh, xl:xh].masked_fill_(hit, fill)
    return img


def _frames(case, seed):
    """The frames of a case, each a tensor of its own.  At most 16 scenes are painted (8 for 4K): the others are
    their mirror images, which a detector sees as new frames."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rs = np.random.RandomState(seed % (1 << 32))
    sizes = _sizes(case)
    most = 8 if case["w"] * case["h"] > 4_000_000 else 16
    scenes, out = {}, []
    for i, (w, h) in enumerate(sizes):
        have = scenes.setdefault((w, h), [])
        k = sum(1 for s in sizes[:i] if s == (w, h))
        if k < max(1, most * sizes.count((w, h)) // len(sizes)):
            have.append(_scene(w, h, case["shapes"], gen, rs))
            out.append(have[-1])
        else:
            turn = [(0,), (1,), (0, 1)][(k // len(have) - 1) % 3]
            out.append(torch.flip(have[k % len(have)], turn).contiguous())
    return out


def _wave_pair(w, h, seed):
    """(prev, next): a scene of six plane waves, moved, and its intensities mapped."""
    rs = np.random.RandomState(seed % (1 << 32))
    dx, dy, gain, off = rs.uniform(-4, 4), rs.uniform(-4, 4), rs.uniform(0.9, 1.1), rs.uniform(-10, 10)
    f, a, p = rs.uniform(0.05, 0.3, 6), rs.uniform(0, 2 * math.pi, 6), rs.uniform(0, 2 * math.pi, 6)
    amp = rs.uniform(12, 28, 6) * np.array([1, 0.8] * 3)

    def frame(dx, dy, gain, off):
        x = torch.arange(w, device="cuda", dtype=torch.float64)[None, :] - dx
        y = torch.arange(h, device="cuda", dtype=torch.float64)[:, None] - dy
        v = torch.full((h, w), 128.0, device="cuda", dtype=torch.float64)
        for i in range(6):
            v += amp[i] * torch.sin(f[i] * math.cos(a[i]) * x + f[i] * math.sin(a[i]) * y + p[i])
        return (gain * v + off + 0.5).floor_().clamp_(0, 255).to(torch.uint8)

    return frame(0, 0, 1, 0), frame(dx, dy, gain, off)


def _track_inputs(case, seed):
    pairs = [_wave_pair(case["w"], case["h"], seed * 1009 + i) for i in range(case["pairs"])]
    rs = np.random.RandomState((seed + 77) % (1 << 32))
    nx, ny, w, h = case["grid_x"], case["grid_y"], case["w"], case["h"]
    # far enough from the border that a coarse patch and the motion stay inside
    m = min(6 * 2 ** (case["levels"] - 1) + 8, min(w, h) // 3)
    pts = []
    for _ in range(case["pairs"]):
        gx, gy = np.meshgrid(np.linspace(m, w - 1 - m, nx), np.linspace(m, h - 1 - m, ny))
        q = np.stack([gx.ravel(), gy.ravel()], axis=1) + rs.uniform(-2, 2, (nx * ny, 2))
        pts.append(torch.from_numpy(q.astype(np.float32)).cuda())
    return [a for a, _ in pairs], [b for _, b in pairs], pts


# ---- one pass ---------------------------------------------------------------


def _pointers(tensors):
    return (ctypes.c_void_p * len(tensors))(*[t.data_ptr() for t in tensors])


def _dims(frames):
    return (vio.Dims * len(frames))(*[vio.Dims(f.shape[1], f.shape[0], f.stride(0)) for f in frames])


def _cells(frames, cell, settings=1):
    """One buffer for all cells of a call, and its parts by setting and frame."""
    n = [vio.num_cells(f.shape[1], f.shape[0], cell) for f in frames] * settings
    buf = torch.empty((sum(n), 4), dtype=torch.int32, device="cuda")
    return buf, list(buf.split(n))


def _settings(case):
    return [(int(t), int(a)) for a in case["arcs"].split() for t in case["thresholds"].split()]


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case)
    if kind in ("detect", "sweep"):
        frames = _frames(case, seed)
        n = len(frames)
        settings = _settings(case) if kind == "sweep" else [(case["thresh"], case["arc"])]
        s["det"] = vio.Detector(max_frames=n, score=case.get("score", SAD_B), nms_radius=case.get("radius", 1))
        s["cells"], parts = _cells(frames, case["cell"], len(settings))
        s["counts"] = torch.empty((len(settings), n), dtype=torch.int32, device="cuda")
        s["keep"] = frames
        s["call"] = (_pointers(frames), _dims(frames), n)
        s["out"] = (_pointers(parts), ctypes.c_void_p(s["counts"].data_ptr()))
        s["set"] = tuple((ctypes.c_int * len(settings))(*v) for v in zip(*settings)) + (len(settings),)
    elif kind == "track":
        s["prev"], s["next"], s["pts"] = _track_inputs(case, seed)
        n = case["grid_x"] * case["grid_y"]
        s["det"] = vio.Detector(max_frames=case["pairs"])
        s["tracks"] = torch.empty((n * case["pairs"], vio.TRACK_RESULT_WORDS), dtype=torch.float32, device="cuda")
        s["outs"] = list(s["tracks"].split([n] * case["pairs"]))
        s["params"] = dict(levels=case["levels"], max_iters=case["iters"], model=case["model"])
    elif kind == "frontend":
        prev, new = _frontend_frames(case, seed)
        s["det"] = det = vio.Detector(max_frames=1)
        (s["old_cells"], _), (s["cells"], _) = _cells([prev], case["cell"]), _cells([new], case["cell"])
        s["counts"] = torch.empty(1, dtype=torch.int32, device="cuda")
        n = s["cells"].shape[0]
        s["tracks"] = torch.empty((n, vio.TRACK_RESULT_WORDS), dtype=torch.float32, device="cuda")
        s["tp"] = vio.TrackParams()
        det.lib.vio_track_params_default(ctypes.byref(s["tp"]))
        s["tp"].levels = case["levels"]
        # the previous frame's features, as the loop's last turn left them
        det.detect([prev], case["thresh"], case["arc"], case["cell"], case["levels"], outs=[s["old_cells"]],
                   counts=s["counts"])
        s["keep"] = (prev, new)
        s["ptr"] = [_pointers([t]) for t in (prev, new, s["old_cells"], s["cells"], s["tracks"])]
        s["dims"], s["n_cells"] = _dims([new]), (ctypes.c_int * 1)(n)
    elif kind == "host":
        frames = _frames(case, seed)
        n = len(frames)
        s["det"] = vio.Detector(max_frames=n, score=case["score"], nms_radius=case["radius"])
        # a camera ring's slots: pinned, back to back, rows as wide as the frame
        room = [-(-f.numel() // 256) * 256 for f in frames]
        s["ring"] = torch.empty(sum(room), dtype=torch.uint8, pin_memory=True)
        views, cells, at = [], [], 0
        total = [vio.num_cells(f.shape[1], f.shape[0], case["cell"]) for f in frames]
        s["cells"] = torch.empty((sum(total), 4), dtype=torch.int32, pin_memory=True)
        s["counts"] = torch.empty(n, dtype=torch.int32, pin_memory=True)
        for f, r, c in zip(frames, room, s["cells"].split(total)):
            v = s["ring"][at:at + f.numel()].view(f.shape)
            v.copy_(f)
            views.append(v.numpy())
            cells.append(c.numpy())
            at += r
        s["batch"] = vio.HostBatch(views, cells, s["counts"].numpy())
    elif kind == "serve":
        s["frames_host"] = [f.cpu().pin_memory().numpy() for f in _frames(case, seed)]
        s["det"] = vio.Detector(max_frames=len(s["frames_host"]))
        s["det"].serve_start(thresh=case["thresh"], arc_len=case["arc"], cell_size=case["cell"],
                             levels=case["levels"])
    return s


def run(s):
    kind, det = s["kind"], s["det"]
    if kind == "detect":
        det.detect_ptrs(*s["call"], s["thresh"], s["arc"], s["cell"], s["levels"], *s["out"], _stream())
        return s["cells"], s["counts"]
    if kind == "sweep":
        th, ar, n = s["set"]
        det.detect_sweep_ptrs(*s["call"], th, ar, n, s["cell"], s["levels"], *s["out"], _stream())
        return s["cells"], s["counts"]
    if kind == "track":
        det.track(s["prev"], s["next"], s["pts"], s["params"], outs=s["outs"])
        return _fields(s["tracks"])
    if kind == "frontend":
        prev, new, old_cells, cells, tracks = s["ptr"]
        stream = _stream()
        det.detect_ptrs(new, s["dims"], 1, s["thresh"], s["arc"], s["cell"], s["levels"], cells,
                        ctypes.c_void_p(s["counts"].data_ptr()), stream)
        det.track_cells_ptrs(prev, new, s["dims"], 1, old_cells, s["n_cells"], s["tp"], tracks, stream)
        return (s["cells"], s["counts"]) + _fields(s["tracks"])
    if kind == "host":
        det.detect_host_batch(s["batch"], s["thresh"], s["arc"], s["cell"], s["levels"])
        return s["cells"], s["counts"]
    tickets = [det.submit(i, f) for i, f in enumerate(s["frames_host"])]
    det.drain()
    got = [det.poll(t, f.shape[1], f.shape[0]) for t, f in zip(tickets, s["frames_host"])]
    return np.concatenate([g[1] for g in got]), np.array([g[2] for g in got])


def _stream():
    return ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)


def _fields(tracks):
    """Views of the records: positions, gain, offset, residual; status and iterations (32-bit whole numbers)."""
    return tracks[:, 0:2], tracks[:, 2], tracks[:, 3], tracks[:, 6], tracks.view(torch.int32)[:, 4:6]


def _frontend_frames(case, seed):
    """Two frames of a camera that moves by whole pixels over a scene, with a little noise in the second."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rs = np.random.RandomState(seed % (1 << 32))
    w, h, dx, dy = case["w"], case["h"], int(rs.randint(-3, 4)), int(rs.randint(-3, 4))
    big = _scene(w + 8, h + 8, 40, gen, rs)
    prev, new = big[4:4 + h, 4:4 + w], big[4 + dy:4 + dy + h, 4 + dx:4 + dx + w]
    new = new.to(torch.int32) + torch.randint(-1, 2, (h, w), generator=gen, device="cuda")
    # rows of a multiple of 16 bytes, as a camera driver lays them out
    out = [torch.zeros((h, -(-w // 16) * 16), dtype=torch.uint8, device="cuda")[:, :w] for _ in range(2)]
    out[0].copy_(prev)
    out[1].copy_(new.clamp_(0, 255))
    return out


# ---- what a pass cannot do without ------------------------------------------


def work(case):
    """Bytes: frames and features read once, records written once.  Operations: for a detection the four compass
    compares of every pixel of every level (each a subtraction, a magnitude and a compare) and 60 for each of the
    twentieth or so of the pixels that are corners; for a track 14 for each of the patch's pixels, in a template and
    in four iterations a level."""
    levels = case["levels"]
    pyramid = sum(0.25 ** k for k in range(levels))
    if case["kind"] in ("detect", "sweep", "host", "serve"):
        sizes = _sizes(case)
        px = sum(w * h for w, h in sizes)
        n = len(case["thresholds"].split()) * len(case["arcs"].split()) if case["kind"] == "sweep" else 1
        cells = sum(-(-w // case["cell"]) * -(-h // case["cell"]) for w, h in sizes)
        return {"bytes": px + n * (16 * cells + 4 * len(sizes)), "flops": (12 + 3 * n) * px * pyramid}
    px = case["w"] * case["h"]
    if case["kind"] == "frontend":
        n = -(-case["w"] // case["cell"]) * -(-case["h"] // case["cell"])
        byte, ops = 2 * px + n * (16 + 16 + 32) + 4, 15 * px * pyramid
    else:
        n = case["pairs"] * case["grid_x"] * case["grid_y"]
        byte, ops = 2 * px * case["pairs"] + n * (8 + 32), 0
    return {"bytes": byte, "flops": ops + n * 5 * 14 * (256 + 64 * (levels - 1))}


# ---- the tracker in 64 bits -------------------------------------------------


def exact(case, seed):
    if case["kind"] == "track":
        prev, nxt, pts = _track_inputs(case, seed)
        got = [_track64(a, b, q, case["levels"], case["iters"], case["model"]) for a, b, q in zip(prev, nxt, pts)]
        return tuple(torch.cat(v) for v in zip(*got)) + (None,)
    return None


def _levels64(img, levels):
    out = [img.to(torch.float64)]
    for _ in range(levels - 1):
        a = out[-1][:out[-1].shape[0] // 2 * 2, :out[-1].shape[1] // 2 * 2]
        out.append(((a[0::2, 0::2] + a[0::2, 1::2] + a[1::2, 0::2] + a[1::2, 1::2] + 2) / 4).floor())
    return out


def _sample64(img, x, y):
    h, w = img.shape
    fx, fy = x.floor().clamp(0, w - 2), y.floor().clamp(0, h - 2)
    ax, ay = x - fx, y - fy
    at = (fy * w + fx).long()
    f = img.reshape(-1)
    return (1 - ay) * ((1 - ax) * f[at] + ax * f[at + 1]) + ay * ((1 - ax) * f[at + w] + ax * f[at + w + 1])


def _track64(prev, nxt, pts, levels, max_iters, model, patch=(16, 8), min_update=0.01):
    """Inverse compositional tracking with gain and offset, coarse to fine, all features of a pair at once: positions,
    gains, offsets, residuals (features that leave the image are not expected)."""
    p, q = _levels64(prev, levels), _levels64(nxt, levels)
    n = pts.shape[0]
    xy = pts.double()
    t, ab = torch.zeros_like(xy), torch.zeros_like(xy)
    res = torch.zeros(n, dtype=torch.float64, device=xy.device)
    use = torch.tensor([True, True, bool(model & 1), bool(model & 2)], device=xy.device)
    for k in reversed(range(levels)):
        size = patch[min(k, 1)]
        c = (xy + 0.5) / 2 ** k - 0.5
        off = torch.arange(-1, size + 1, device=xy.device, dtype=torch.float64) - (size - 1) / 2
        gx = (c[:, 0, None, None] + off[None, None, :]).expand(n, size + 2, size + 2)
        gy = (c[:, 1, None, None] + off[None, :, None]).expand(n, size + 2, size + 2)
        g = _sample64(p[k], gx, gy)
        tm = g[:, 1:-1, 1:-1]
        gain = 1 + ab[:, 0, None, None]
        u = torch.stack([gain * (g[:, 1:-1, 2:] - g[:, 1:-1, :-2]) / 2, gain * (g[:, 2:, 1:-1] - g[:, :-2, 1:-1]) / 2,
                         tm, torch.ones_like(tm)], -1).reshape(n, -1, 4) * use
        hess = u.transpose(1, 2) @ u + torch.diag((~use).double())
        on = torch.ones(n, dtype=torch.bool, device=xy.device)
        for _ in range(max_iters):
            v = _sample64(q[k], gx[:, 1:-1, 1:-1] + t[:, 0, None, None], gy[:, 1:-1, 1:-1] + t[:, 1, None, None])
            r = (v - (1 + ab[:, 0, None, None]) * tm - ab[:, 1, None, None]).reshape(n, -1, 1)
            d = torch.linalg.solve(hess, u.transpose(1, 2) @ r)[:, :, 0] * on[:, None]
            res = torch.where(on, r.square().mean((1, 2)).sqrt(), res)
            t, ab = t - d[:, :2], ab + d[:, 2:]
            on = on & (d[:, :2].norm(dim=1) >= min_update)
            if not on.any():
                break
        if k:
            t = 2 * t
    return xy + t, ab[:, 0], ab[:, 1], res
