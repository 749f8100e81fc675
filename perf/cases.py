"""What a program that uses this renderer has it do, as cases to be timed.

A case is one of these kinds of work, each through the public entry points:

  render   views of a canvas that is resident on the GPU, into a device image (`render`)
  host     the same into host memory (`render_host`: the end-to-end frame)
  paint    a stamp table painted into a new canvas, then a look at it (`paint_spheres`, `render`), and for small
           canvases the pools read back as a program that saves the painting does (`download_octree`)
  session  an editing session: a painting opened from its stamps, strokes appended with a frame after each
           (`paint_append`, `render`), then saved
  upload   pools in host memory made the current canvas, then a frame (`upload_octree`, `render`)
  recolour new values for a range of leaves, then a frame (`update_leaves`, `render`)

The library keeps one canvas per process. A resident canvas is what a program keeps between calls, so it comes from
the case alone (`canvas_seed`); what changes from call to call (the cameras, the stamps that are painted, the strokes,
the new leaf values) comes from the seed. The canvases are the recipes of this repository's configurations: a unit cube
of depth 8, a 1 km hall of depth 16, and rooms in a 40 km canvas of depth 24 or 27, at their sizes or reduced ones.
"""
import math

import numpy as np
import torch

import paper_1704_02724_gb300 as cx

CAMERA = np.dtype([("eye", "<f8", (3,)), ("right", "<f8", (3,)), ("up", "<f8", (3,)), ("forward", "<f8", (3,)),
                   ("tan_half_fov_y", "<f8"), ("width", "<i4"), ("height", "<i4"), ("out_offset_px", "<i8"),
                   ("background", "<f4", (4,))])
SKY = (0.25, 0.35, 0.5, 1.0)
T_MIN = 2.0 ** -20
N_ROOMS = 4

# Per scene: depth and side of the canvas, and what a pass over it costs per ray and per stamp (leaf steps of a ray;
# bytes of the canvas that a ray's own cells take; records and leaves per small stamp), counted on these recipes.
SCENES = {
    "cube": dict(depth=8, extent=1.0, steps=18, ray_bytes=100, rec_per_stamp=430, leaf_per_stamp=2000),
    "hall": dict(depth=16, extent=1000.0, steps=10, ray_bytes=1, rec_per_stamp=550, leaf_per_stamp=3500),
    "rooms24": dict(depth=24, extent=40000.0, steps=300, ray_bytes=14, rec_per_stamp=190, leaf_per_stamp=1200),
    "rooms27": dict(depth=27, extent=40000.0, steps=320, ray_bytes=100, rec_per_stamp=460, leaf_per_stamp=3000),
}


def listed():
    return [
        # A thumbnail of a small object: the smallest call a viewer makes, all latency.
        dict(name="cube_256", kind="render", scene="cube", n_small=1000, width=256, height=256, pairs=0, views=1, precision="mixed", graph=False),
        # One HD frame inside opaque paint: few leaves per ray, so the per-ray work counts.
        dict(name="hall_1080p", kind="render", scene="hall", n_small=100000, width=1920, height=1080, pairs=0, views=1, precision="mixed", graph=False),
        # The stereo frame of a headset inside a room of the depth-24 canvas: the headline workload.
        dict(name="rooms24_stereo_2160", kind="render", scene="rooms24", n_small=200000, width=2160, height=2160, pairs=1, views=0, precision="mixed", graph=False),
        # Stereo pairs at two scales in the depth-27 canvas, replayed from a CUDA graph as a frame loop does.
        dict(name="rooms27_two_pairs_graph", kind="render", scene="rooms27", n_small=100000, width=721, height=719, pairs=2, views=0, precision="mixed", graph=True),
        # Many small views of uneven size in one call: thumbnails and light probes of the rooms.
        dict(name="rooms27_64_views", kind="render", scene="rooms27", n_small=100000, width=200, height=200, pairs=0, views=64, precision="mixed", graph=False),
        # The same image with every step in 64 bits: the accurate final frame (at preview size).
        dict(name="rooms24_fp64_540", kind="render", scene="rooms24", n_small=20000, width=540, height=540, pairs=1, views=0, precision="fp64", graph=False),
        # A headset frame at 1680 x 1512 per eye, delivered in host memory.
        dict(name="rooms24_host_1680", kind="host", scene="rooms24", n_small=20000, width=1680, height=1512, pairs=1, views=0, precision="mixed", graph=False),
        # A small painting built and saved: launches, synchronisations and allocations count.
        dict(name="paint_cube_save", kind="paint", scene="cube", n_small=1000, save=True),
        # The depth-24 painting of 210,000 stamps built and looked at.
        dict(name="paint_rooms24", kind="paint", scene="rooms24", n_small=200000, save=False),
        # Strokes added to an open painting, a frame after each, then saved.
        dict(name="session_rooms24", kind="session", scene="rooms24", n_small=3000, strokes=2, stroke_stamps=200),
        # A saved canvas loaded from host memory and shown.
        dict(name="upload_cube", kind="upload", scene="cube", n_small=1000, width=256, height=256),
        # A recoloured region of the canvas and the frame after it.
        dict(name="recolour_hall", kind="recolour", scene="hall", n_small=10000, leaves=300000, width=960, height=540),
    ]


def _log_int(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["render", "render", "render", "render", "host", "paint", "session", "upload", "recolour"])
    c = dict(kind=kind, canvas_seed=rng.randrange(1 << 20))
    if kind in ("render", "host"):
        c["scene"] = rng.choice(["cube", "hall", "rooms24", "rooms27"])
        top = {"cube": 3000, "hall": 100000, "rooms24": 200000, "rooms27": 100000}[c["scene"]]
        c["n_small"] = _log_int(rng, top // 20, top)
        c["precision"] = "fp64" if kind == "render" and rng.random() < 0.2 else "mixed"
        c["graph"] = kind == "render" and rng.random() < 0.3
        c["pairs"] = rng.choice([0, 0, 1, 2]) if c["scene"].startswith("rooms") else 0
        c["views"] = 0 if c["pairs"] else rng.choice([1, 1, 2, _log_int(rng, 4, 64)])
        views = 2 * c["pairs"] + c["views"]
        most = {"cube": 2e6, "hall": 4e6}.get(c["scene"], 2e6) / (6 if c["precision"] == "fp64" else 1)
        c["width"] = _log_int(rng, 31, max(64, min(2160, int(1.2 * math.sqrt(most / views)))))
        c["height"] = max(17, int(c["width"] * rng.uniform(0.5, 1.1)))
    elif kind == "paint":
        c["scene"] = rng.choice(["cube", "hall", "rooms24", "rooms27"])
        c["n_small"] = _log_int(rng, 200, {"cube": 3000, "hall": 60000, "rooms24": 200000, "rooms27": 60000}[c["scene"]])
        c["save"] = c["scene"] == "cube"
    elif kind == "session":
        c.update(scene=rng.choice(["rooms24", "rooms27"]), n_small=_log_int(rng, 500, 5000), strokes=rng.randint(1, 3),
                 stroke_stamps=_log_int(rng, 10, 600))
    elif kind == "upload":
        c.update(scene="cube", n_small=_log_int(rng, 100, 2000), width=_log_int(rng, 65, 700), height=_log_int(rng, 65, 700))
    else:
        c.update(scene=rng.choice(["cube", "hall"]), leaves=_log_int(rng, 1000, 300000), width=_log_int(rng, 65, 1000),
                 height=_log_int(rng, 65, 700))
        c["n_small"] = 1000 if c["scene"] == "cube" else _log_int(rng, 3000, 10000)
    return c


# ---------------------------------------------------------------------------
# canvases: stamps of the repository's recipes
# ---------------------------------------------------------------------------

def _log_u(u, a, b):
    return np.exp(math.log(a) + u * (math.log(b) - math.log(a)))


def _paint_sigma(flag, u):
    return np.where(flag < 0.3, _log_u(u, 200.0, 2000.0), 0.5 + 19.5 * u)


def _rooms(canvas_seed):
    """Low corners of the 1 m rooms: in the central 2 km, kept apart by the chance of the draw."""
    return -1000.0 + np.random.default_rng([canvas_seed, 1]).random((N_ROOMS, 3)) * 1999.0


def _fine_stamps(r, corner, n, depth, extent, lo=0.0, hi=1.0):
    """n semi-transparent spheres in the room at `corner` (its part [lo, hi] per axis)."""
    u = r.random((n, 8))
    radius = _log_u(u[:, 3], extent * 2.0 ** -depth, 0.1)
    rgba = np.concatenate([u[:, 4:7], (_log_u(u[:, 7], 0.002, 0.2) / (2.0 * radius))[:, None]], axis=1)
    return corner + lo + u[:, :3] * (hi - lo), radius, rgba


def _stamps(scene, n_small, canvas_seed, seed):
    """The stamp table of a painting: (depth, extent, centres [n, 3], radii [n], rgba [n, 4])."""
    depth, extent = SCENES[scene]["depth"], SCENES[scene]["extent"]
    r = np.random.default_rng([seed, 2])
    if scene == "cube":
        u = r.random((n_small, 8))
        c, radius = (u[:, :3] - 0.5) * extent, (2.0 + 18.0 * u[:, 3]) * (extent / 256.0)
        q = np.concatenate([u[:, 4:7], 0.5 + 19.5 * u[:, 7:8]], axis=1)
    elif scene == "hall":
        u = r.random((n_small, 9))
        c, radius = (u[:, :3] - 0.5) * extent, _log_u(u[:, 3], extent * 2.0 ** -depth, 50.0)
        q = np.concatenate([u[:, 4:7], _paint_sigma(u[:, 7], u[:, 8])[:, None]], axis=1)
    else:
        rooms = _rooms(canvas_seed)
        n_bg = max(500, min(10000, n_small // 2))
        u = r.random((2 * n_bg, 9))
        c, radius = (u[:, :3] - 0.5) * extent, _log_u(u[:, 3], 100.0, 1000.0)
        near = np.zeros(2 * n_bg, dtype=bool)
        for p in rooms:  # the background stays 10 m clear of the rooms
            near |= np.linalg.norm(np.maximum(np.maximum(p - c, 0.0), c - p - 1.0), axis=1) < radius + 10.0
        keep = np.flatnonzero(~near)[:n_bg]
        q = np.concatenate([u[:, 4:7], _paint_sigma(u[:, 7], u[:, 8])[:, None]], axis=1)
        parts = [(c[keep], radius[keep], q[keep])]
        parts += [_fine_stamps(r, p, n_small // N_ROOMS, depth, extent) for p in rooms]
        c, radius, q = (np.concatenate([p[i] for p in parts]) for i in range(3))
    return depth, extent, np.ascontiguousarray(c), np.ascontiguousarray(radius), np.ascontiguousarray(q, dtype=np.float32)


_canvas = {"key": None, "table": None}


def _resident(case):
    """Make the case's canvas the current one, if it is not."""
    cs = case.get("canvas_seed", 7)
    key = (case["kind"] == "recolour", case["scene"], case["n_small"], cs)
    if _canvas["key"] != key:
        t = _stamps(case["scene"], case["n_small"], cs, cs)
        cx.paint_spheres(*t)
        _canvas.update(key=key, table=t)
    return cs


# ---------------------------------------------------------------------------
# cameras
# ---------------------------------------------------------------------------

def _look(eye, f, tan, width, height, offset, bg):
    f = f / np.linalg.norm(f)
    r = np.cross(f, [0.0, 1.0, 0.0])
    r /= np.linalg.norm(r)
    c = np.zeros((), dtype=CAMERA)
    c["eye"], c["right"], c["up"], c["forward"] = eye, r, np.cross(r, f), f
    c["tan_half_fov_y"], c["width"], c["height"], c["out_offset_px"], c["background"] = tan, width, height, offset, bg
    return c


def _heading(u):
    yaw, pitch = 2 * math.pi * u[0], (u[1] - 0.5) * 0.6
    return np.array([math.cos(pitch) * math.sin(yaw), math.sin(pitch), math.cos(pitch) * math.cos(yaw)])


def _cameras(scene, canvas_seed, table, seed, width, height, pairs, views):
    """Views by the scene: from outside at the cube, inside the hall clear of paint, inside the rooms (stereo pairs at
    scales 1 and 0.01 in turn, single views of uneven size and scale)."""
    r = np.random.default_rng([seed, 3])
    cams, off = [], 0

    def add(eye, f, tan, w, h, bg):
        nonlocal off
        cams.append(_look(eye, f, tan, w, h, off, bg))
        off += w * h

    for v in range(pairs + views):
        u = r.random(8)
        w, h = width, height
        if views > 2:  # uneven sizes around the nominal one
            s = math.exp(((v * 0.618034) % 1.0 - 0.5) * 2.0)
            w, h = max(8, int(width * s)), max(8, int(height * s))
        if scene == "cube":
            d = np.array([0.4 + u[0], 0.3 + u[1], 1.0 + u[2]])
            eye = 2.5 * d / np.linalg.norm(d)
            add(eye, -eye, math.tan(math.radians(30)), w, h, (0, 0, 0, 0))
        elif scene == "hall":
            best = -math.inf
            for p in (r.random((128, 3)) - 0.5) * 900.0:  # the first point that is 1 m clear of paint, or the clearest
                clear = np.min(np.linalg.norm(table[2] - p, axis=1) - table[3])
                if clear > best:
                    eye, best = p, clear
                if best > 1.0:
                    break
            add(eye, _heading(u), math.tan(math.radians(30)), w, h, SKY)
        else:
            corner = _rooms(canvas_seed)[v % N_ROOMS]
            if v < pairs:
                scale = 1.0 if v % 2 == 0 else 0.01
                head, f = corner + 0.5 + (u[2:5] - 0.5) * 0.2 * scale, _heading(u)
                side = np.cross(f, [0.0, 1.0, 0.0])
                side *= 0.032 * scale / np.linalg.norm(side)
                add(head - side, f, 1.0, w, h, SKY)
                add(head + side, f, 1.0, w, h, SKY)
            else:
                scale = _log_u(u[6], 1e-3, 1.0)
                add(corner + 0.5 + (u[2:5] - 0.5) * 0.4 * scale, _heading(u), 1.0, w, h, SKY)
    return np.stack(cams), off


# ---------------------------------------------------------------------------
# the passes
# ---------------------------------------------------------------------------

def prepare(case, seed):
    kind, scene = case["kind"], case["scene"]
    s = dict(kind=kind, case=case)
    if kind in ("render", "host", "recolour"):
        cs = _resident(case)
        s["cams"], n = _cameras(scene, cs, _canvas["table"], seed, case["width"], case["height"], case.get("pairs", 0),
                                case.get("views", 1))
        s["opts"] = dict(precision=cx.PREC_FP64_LINKS if case.get("precision") == "fp64" else cx.PREC_MIXED,
                         use_graph=int(bool(case.get("graph"))), count_reads=0)
        if kind == "host":
            s["out"] = torch.empty((n, 4), dtype=torch.float32, pin_memory=True).numpy()
        else:
            s["out"] = torch.empty((n, 4), dtype=torch.float32, device="cuda")
        if kind == "recolour":
            n_leaf = cx.canvas_info()[1]
            s["first"], count = n_leaf // 8, min(case["leaves"], n_leaf // 4)
            r = np.random.default_rng([seed, 4])
            v = np.concatenate([r.random((count, 3)), _paint_sigma(r.random(count), r.random(count))[:, None]], axis=1)
            s["values"] = v.astype(np.float16).view(np.uint16)
        return s
    cs = case.get("canvas_seed", 7)
    if kind == "upload":
        # the pools as a program that saved this painting has them on the host
        cx.paint_spheres(*_stamps(scene, case["n_small"], cs, seed))
        _canvas["key"] = None
        s["nodes"], s["leaves"] = cx.download_octree()
        s["cams"], n = _cameras(scene, cs, None, seed, case["width"], case["height"], 0, 1)
    else:
        s["table"] = _stamps(scene, case["n_small"], cs, seed)
        side = 256 if scene == "cube" else 400
        s["cams"], n = _cameras(scene, cs, s["table"], seed, side, side, 0, 1)
        if kind == "session":
            r = np.random.default_rng([seed, 5])
            room = _rooms(cs)[0]
            s["strokes"] = [tuple(np.ascontiguousarray(x, dtype=t) for x, t in zip(
                _fine_stamps(r, room, case["stroke_stamps"], s["table"][0], s["table"][1], 0.1 + 0.2 * k, 0.4 + 0.2 * k),
                (np.float64, np.float64, np.float32))) for k in range(case["strokes"])]
        if kind == "session" or case["save"]:
            # where the program keeps the painting that it saves: room for the most that its stamps can make
            most = s["table"][3].size + sum(x[1].size for x in s.get("strokes", ()))
            s["nodes"] = np.zeros((1500 * most + 20000, 8), dtype=np.int32)
            s["leaves"] = np.zeros((7000 * most + 50000, 4), dtype=np.int16)  # FP16 bits
    s["out"] = torch.empty((n, 4), dtype=torch.float32, device="cuda")
    return s


def _save(s, size):
    if size[0] > len(s["nodes"]) or size[1] > len(s["leaves"]):
        raise RuntimeError("a painting of %d records and %d leaves does not fit" % tuple(size))
    if cx.lib().canvox_download_octree(s["nodes"].ctypes.data, s["leaves"].ctypes.data):
        raise RuntimeError(cx.last_error())
    return s["nodes"], s["leaves"]


def run(s):
    kind, case = s["kind"], s["case"]
    if kind in ("render", "host", "recolour"):
        _resident(case)
        if kind == "host":
            cx.render_host(s["cams"], s["out"], **s["opts"])
        else:
            if kind == "recolour":
                cx.update_leaves(s["first"], s["values"])
            cx.render(s["cams"], s["out"], **s["opts"])
        return s["out"]
    _canvas["key"] = None  # the calls below replace the resident canvas
    if kind == "upload":
        d = SCENES[case["scene"]]
        cx.upload_octree(s["nodes"], s["leaves"], d["depth"], d["extent"])
        cx.render(s["cams"], s["out"])
        return s["out"]
    got = {"size": list(cx.paint_spheres(*s["table"]))}
    cx.render(s["cams"], s["out"])
    if kind == "session":
        frames = [s["out"].clone()]
        for stroke in s["strokes"]:
            got["size"] += cx.paint_append(*stroke)
            cx.render(s["cams"], s["out"])
            frames.append(s["out"].clone())
        got["frames"] = frames
    else:
        got["frames"] = [s["out"]]
    if kind == "session" or case["save"]:
        got["nodes"], got["leaves"] = _save(s, got["size"][-2:])
    return got


def work(case):
    """Bytes: the image written, the canvas cells a view's rays need, stamps in and pools out. Flops: 30 per leaf step of
    a ray (three plane times, the opacity and three colour sums), 40 per stamp and cell it refines."""
    d, kind = SCENES[case["scene"]], case["kind"]
    if kind in ("render", "host", "recolour", "upload"):
        rays = case["width"] * case["height"] * (2 * case.get("pairs", 0) + case.get("views", 1))
        frames = 1
    else:
        rays = 256 * 256 if case["scene"] == "cube" else 400 * 400
        frames = 1 + case.get("strokes", 0)
    w = {"bytes": frames * rays * (16.0 + d["ray_bytes"]), "flops": frames * rays * d["steps"] * 30.0}
    if kind == "recolour":
        w["bytes"] += 8.0 * case["leaves"]
    if kind in ("paint", "session", "upload"):
        n = case["n_small"] + case.get("strokes", 0) * case.get("stroke_stamps", 0)
        w["bytes"] += n * (56.0 + 32.0 * d["rec_per_stamp"] + 8.0 * d["leaf_per_stamp"])
        if kind != "upload":
            w["flops"] += 40.0 * n * d["rec_per_stamp"]
    return w


# ---------------------------------------------------------------------------
# the images in 64 bits
# ---------------------------------------------------------------------------

def _pixel_rays(cam):
    """Directions [3, W H] of the rays through the pixel centres of one view."""
    f64 = dict(dtype=torch.float64, device="cuda")
    W, H, tan = int(cam["width"]), int(cam["height"]), float(cam["tan_half_fov_y"])
    f = cam["forward"] / np.linalg.norm(cam["forward"])
    u = cam["up"] - (cam["up"] @ f) * f
    u /= np.linalg.norm(u)
    r = cam["right"] - (cam["right"] @ f) * f - (cam["right"] @ u) * u
    r /= np.linalg.norm(r)
    x = (2.0 * torch.arange(W, **f64) + 1.0) / W - 1.0
    y = 1.0 - (2.0 * torch.arange(H, **f64) + 1.0) / H
    f, u, r = (torch.tensor(v, **f64)[:, None, None] for v in (f, u, r))
    d = ((f + (x * tan * (W / H))[None, None, :] * r) + (y * tan)[None, :, None] * u).reshape(3, -1)
    return d / d.square().sum(0).sqrt()


def _exact_image(nodes, leaves, scene, cams):
    """The views' images in plain FP64: every step locates the leaf from the root and crosses to its nearest far face;
    emission-absorption per leaf; a ray ends below transmittance 2^-20 or outside the canvas."""
    f64 = dict(dtype=torch.float64, device="cuda")
    depth, extent = SCENES[scene]["depth"], SCENES[scene]["extent"]
    half = 0.5 * extent
    nodes = torch.from_numpy(nodes).cuda()
    leaves = torch.from_numpy(leaves.view(np.float16)).cuda()
    d = torch.cat([_pixel_rays(c) for c in cams], dim=1)
    each = torch.tensor([int(c["width"]) * int(c["height"]) for c in cams], device="cuda")
    o = torch.tensor(cams["eye"], **f64).t().repeat_interleave(each, dim=1)
    bg = torch.tensor(cams["background"].astype(np.float64), **f64).t().repeat_interleave(each, dim=1)
    d = torch.where(d == 0, torch.full_like(d, 1e-300), d)  # a ray in a plane runs on its high side
    pos = d > 0
    lo, hi = (-half - o) / d, (half - o) / d
    t, t1 = torch.where(pos, lo, hi).amax(0).clamp(min=0.0), torch.where(pos, hi, lo).amin(0)
    C, T = torch.zeros_like(d), torch.ones_like(t)
    live = torch.nonzero(t < t1)[:, 0]
    o, d, pos, t, t1, c, tr = o[:, live], d[:, live], pos[:, live], t[live], t1[live], C[:, live], T[live]
    weight = torch.tensor([1, 2, 4], device="cuda")[:, None]
    while live.numel():
        rec, slot = torch.zeros_like(live), torch.ones_like(live)
        cell, level = torch.zeros_like(d), torch.zeros_like(t)
        for lev in range(depth):
            M = (2.0 * cell + 1.0) * (extent * 2.0 ** -(lev + 1)) - half
            tm = (M - o) / d
            b = torch.where(pos, tm <= t, tm > t)
            s = nodes[rec, (b.to(torch.int64) * weight).sum(0)].to(torch.int64)
            go = slot > 0
            cell = torch.where(go, 2.0 * cell + b, cell)
            level = torch.where(go, lev + 1.0, level)
            slot = torch.where(go, s, slot)
            rec = torch.where(slot > 0, slot, rec)
            if lev % 4 == 3 and not bool((slot > 0).any()):
                break
        M = (cell + pos) * (extent * torch.exp2(-level)) - half
        te = torch.minimum(((M - o) / d).amin(0), t1)
        v = leaves[(-slot - 1).clamp(min=0)].double()
        v = torch.where((slot < 0)[:, None], v, torch.zeros_like(v))
        em = torch.expm1(-v[:, 3] * (te - t))
        c = c - tr * em * v[:, :3].t()
        tr = tr + tr * em
        t = te
        stay = (tr >= T_MIN) & (te < t1)
        if not bool(stay.all()):
            end = ~stay
            C[:, live[end]], T[live[end]] = c[:, end], tr[end]
            live, t, t1, tr = (x[stay] for x in (live, t, t1, tr))
            o, d, pos, c = (x[:, stay] for x in (o, d, pos, c))
    return torch.cat([C + T * bg[:3], (1.0 - T)[None]]).t()


def exact(case, seed):
    """The images that run() gives for this seed, each from the canvas that it shows (its pools read as numbers)."""
    scene = case["scene"]
    rays = case.get("width", 400) * case.get("height", 400) * (2 * case.get("pairs", 0) + case.get("views", 1))
    if SCENES[scene]["steps"] * SCENES[scene]["depth"] * (3e-4 + 5e-10 * rays) > 15.0:  # seconds
        return None
    s = prepare(case, seed)
    run(s)
    if case["kind"] == "session":  # the frame before each stroke shows a canvas that is gone: the last one's is here
        last = _exact_image(*cx.download_octree(), scene, s["cams"])
        return {"frames": [None] * case["strokes"] + [last], "leaves": None, "nodes": None, "size": None}
    image = _exact_image(*cx.download_octree(), scene, s["cams"])
    if case["kind"] == "recolour":
        _canvas["key"] = None
    return {"frames": [image], "leaves": None, "nodes": None, "size": None} if case["kind"] == "paint" else image
