"""Workloads of the renderer, timed through its public entry points.

A case is one call a user's program makes again and again: a frame into device
buffers, a batch of views, frames into host memory, chunks loaded into a scene,
requests to the render server.  Worlds stand for what a program loads once, so
they are built once per process and kept; the camera poses (and which chunks
are loaded) come from the seed.  The open world differs: only the chunks that a
pose needs are resident, so its scene belongs to the state.

Fields: kind (render | tiles | batch | host | load | serve), world (single | city |
open), side (city: voxels per axis), pose (walk: a walker above the ground; far:
the whole world from outside; path: a flight path), w, h, tau (LOD threshold in
pixels), color (colour-block tolerance, -1: raw arrays), views (frames, requests
or chunk LODs of one pass), view_dist (open world).
"""
import functools
import math

from dataclasses import replace

import numpy as np
import torch

import paper_2505_02017_gb300 as aok
import scenegen as sg
from paper_2505_02017_gb300.stream import Streamer


def _case(name, kind, world, w, h, side=0, pose="walk", tau=1.0, color=-1.0, views=1, view_dist=0.0):
    c = {"kind": kind, "world": world, "side": side, "pose": pose, "w": w, "h": h, "tau": tau, "color": color,
         "views": views, "view_dist": view_dist}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one object in one chunk, as a viewer or a thumbnail asks for it: launches and latency count
        _case("object_256", "render", "single", 256, 256, pose="orbit"),
        # a preview, an adaptive-resolution or a probe view of the city: one wave of rays
        _case("city_320x180", "render", "city", 320, 180, side=4096),
        # a window of odd size on the smaller city, below the frame size from which the beam pass runs
        _case("city_1283x717", "render", "city", 1283, 717, side=2048, tau=1.5),
        # the game frame: a walker in the city at 1080p
        _case("city_1080p", "render", "city", 1920, 1080, side=4096),
        # the whole city from outside at 2160p: many LODs, long rays, many misses
        _case("overview_2160p", "render", "city", 3840, 2160, side=4096, pose="far"),
        # open world, 128 x 128 x 2 regions of which those within the view distance are resident
        _case("open_1440p", "render", "open", 2560, 1440, pose="path", view_dist=8192.0),
        # compressed colours (lossy blocks) at 720p
        _case("blocks_720p", "render", "city", 1280, 720, side=4096, color=0.05),
        # the tile-chunk pipeline, a walker's successive frames
        _case("tiles_1080p", "tiles", "city", 1920, 1080, side=4096),
        # many cameras at once, uneven resolutions: a batch of views for a simulator or several players
        _case("batch_24", "batch", "city", 2560, 1440, side=4096, views=24),
        # a frame loop whose frames go to host memory (encoder, remote display): four frames in flight order
        _case("host_4x1080p", "host", "city", 1920, 1080, side=4096, views=4),
        # chunks streamed into a running scene, then a frame of it
        _case("load_32", "load", "city", 640, 360, side=2048, views=32),
        # the render server: requests of mixed sizes submitted together
        _case("serve_16", "serve", "city", 1920, 1080, side=2048, views=16),
    ]


def draw(rng):
    def size(lo, hi):
        w = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        a = rng.choice((16 / 9, 16 / 10, 4 / 3, 1.0, 21 / 9))
        return w, max(1, int(round(w / a)) + rng.randint(-3, 3))

    kind = rng.choice(("render",) * 6 + ("tiles", "batch", "host", "load", "serve"))
    tau = rng.choice((1.0, 1.0, 1.5, 2.0))
    side = rng.choice((1024, 2048, 4096))
    color = rng.choice((-1.0, -1.0, -1.0, 0.0, 0.05))
    if kind == "render":
        world = rng.choice(("single", "city", "city", "city", "open"))
        if world == "single":
            w, h = size(64, 1024)
            return _case(None, kind, world, w, h, pose="orbit", tau=tau)
        if world == "open":
            w, h = size(640, 2560)
            return _case(None, kind, world, w, h, pose="path", tau=tau, view_dist=float(rng.randint(3000, 8192)))
        w, h = size(96, 3000)
        return _case(None, kind, world, w, h, side=side, pose=rng.choice(("walk", "walk", "far")), tau=tau, color=color)
    if kind == "tiles":
        w, h = size(320, 2560)
        return _case(None, kind, "city", w, h, side=side, tau=tau)
    if kind == "batch":
        w, h = size(320, 1920)
        return _case(None, kind, "city", w, h, side=side, tau=tau, color=color, views=rng.randint(2, 24))
    if kind == "host":
        w, h = size(320, 1920)
        return _case(None, kind, "city", w, h, side=side, tau=tau, views=rng.randint(1, 4))
    if kind == "load":
        w, h = size(160, 1280)
        return _case(None, kind, "city", w, h, side=2048, tau=tau, views=rng.randint(1, 48))
    w, h = size(320, 1920)
    return _case(None, kind, "city", w, h, side=side, tau=tau, views=rng.randint(1, 16))


# ---------------------------------------------------------------------------
# worlds, kept for the process
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _world(kind, side, layered, view_dist):
    if kind == "single":
        return sg.World(sg.SINGLE_128)
    if kind == "open":
        return sg.World(replace(sg.OPEN_65536, view_dist=view_dist))
    spec = sg.CITY_4096 if side == 4096 else sg.city(2, side)
    return sg.World(replace(spec, mat_mode=1) if layered else spec)


@functools.lru_cache(maxsize=None)
def _built(kind, side, layered):
    return aok.BuiltWorld(_world(kind, side, layered, 0.0))


@functools.lru_cache(maxsize=None)
def _context():
    return aok.Context(0)


@functools.lru_cache(maxsize=None)
def _scene(kind, side, color):
    layered = color >= 0.0
    return aok.Scene.from_world(_context(), _world(kind, side, layered, 0.0), built=_built(kind, side, layered),
                                color_tol=color if layered else None)


def _pose(case, world, rng, w, h):
    if case["pose"] == "orbit":
        return sg.orbit_camera(world.spec, rng.next(), w, h, radius=160.0, center=(64, 64, 48))
    if case["pose"] == "far":
        return sg.orbit_camera(world.spec, rng.next(), w, h)
    return sg.ground_camera(world, rng.next(), w, h)


def _sizes(case):
    """The resolutions of a case's views: the largest is w x h, the others are steps below it."""
    w, h = case["w"], case["h"]
    if case["kind"] not in ("batch", "serve"):
        return [(w, h)] * (case["views"] if case["kind"] == "host" else 1)
    steps = (1.0, 0.75, 0.5, 0.25, 0.125)
    return [(max(1, int(w * f)), max(1, int(h * f))) for f in (steps[i % 5] for i in range(case["views"]))]


# ---------------------------------------------------------------------------
# a case's state and one pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind, tau = case["kind"], case["tau"]
    rng = sg.Rng(seed * 1000003 + 17)
    s = {"kind": kind, "tau": tau}
    if case["world"] == "open":
        world = _world("open", 0, False, case["view_dist"])
        path = sg.path_cameras(world, rng.next(), 300, case["w"], case["h"])
        s["cam"] = path[rng.randint(0, 299)]
        s["ctx"] = _context()
        s["scene"] = aok.Scene(s["ctx"], world.spec, node_words=24 << 20, leaves=8 << 20, mat_bytes=512 << 20)
        Streamer(s["ctx"], world, s["scene"]).update(s["cam"], tau)
        s["out"] = aok.alloc_frame(case["w"], case["h"])
        return _Open(s)
    world = _world(case["world"], case["side"], case["color"] >= 0.0, 0.0)
    cams = [_pose(case, world, rng, w, h) for w, h in _sizes(case)]
    s["cam"] = cams[0]
    if kind == "load":
        # a scene of its own: its residency changes with every pass
        built = _built("city", case["side"], False)
        s["ctx"] = _context()
        # room in the pools beside what is resident: freed ranges are not all of the sizes wanted next
        s["scene"] = aok.Scene(s["ctx"], world.spec, 2 * built.node_words, 2 * built.leaves, 2 * built.mat_bytes)
        s["scene"].upload_built(built)
        grid, n_lods = s["scene"].grid, world.spec.n_lods
        full = [(i, lod) for i in range(len(built)) for lod in range(n_lods) if built.blob(i, lod)[1].n_node_words]
        s["load"] = []
        for _ in range(min(case["views"], len(full))):
            i, lod = full.pop(rng.randint(0, len(full) - 1))
            c, blob = built.blob(i, lod)
            s["load"].append((c % grid[0], (c // grid[0]) % grid[1], c // (grid[0] * grid[1]), lod, blob))
        s["out"] = aok.alloc_frame(case["w"], case["h"])
        return _Open(s)
    if kind == "serve":
        s["ctx"] = aok.Context(0)
        s["scene"] = aok.Scene.from_world(s["ctx"], world, built=_built("city", case["side"], False))
        s["cams"] = cams
        s["server"] = aok.Server(s["ctx"], max_slots=64, max_batch=32, n_streams=2)
        return _Open(s)
    s["ctx"] = _context()
    s["scene"] = _scene(case["world"], case["side"], case["color"])
    if kind == "batch":
        s["out"] = [aok.alloc_frame(c.W, c.H) for c in cams]
        s["views"] = [aok.make_view(s["scene"], c, tau, *o) for c, o in zip(cams, s["out"])]
    elif kind == "host":
        s["cams"] = cams
        s["out"] = [(torch.empty((c.H, c.W, 4), dtype=torch.int32, pin_memory=True),
                     torch.empty((c.H, c.W), dtype=torch.float32, pin_memory=True)) for c in cams]
    else:
        s["out"] = aok.alloc_frame(case["w"], case["h"])
    return s


class _Open(dict):
    """A state that owns its scene (and server): both go when the state does."""

    def __del__(self):
        if "server" in self:
            self["server"].stop()
        self["scene"].destroy()
        if "server" in self:
            self["ctx"].close()


def run(s):
    kind, ctx, scene = s["kind"], s["ctx"], s["scene"]
    if kind == "render":
        aok.render(ctx, scene, s["cam"], s["tau"], *s["out"])
    elif kind == "tiles":
        aok.render_tiles(ctx, scene, s["cam"], s["tau"], *s["out"])
    elif kind == "batch":
        aok.render_batch(ctx, s["views"])
    elif kind == "host":
        tickets = [aok.render_host_async(ctx, scene, c, s["tau"], *o) for c, o in zip(s["cams"], s["out"])]
        for t in tickets:
            aok.host_frame_wait(ctx, t)
    elif kind == "load":
        for cx, cy, cz, lod, blob in s["load"]:
            scene.evict(cx, cy, cz, lod)
        for cx, cy, cz, lod, blob in s["load"]:
            scene.upload(cx, cy, cz, lod, blob)
        aok.render(ctx, scene, s["cam"], s["tau"], *s["out"])
    else:
        server = s["server"]
        tickets = [server.submit(scene, c, s["tau"]) for c in s["cams"]]
        out = []
        for t in tickets:
            status, frame = server.wait(t)
            aok.check(status, "aok_serve_wait")
            out.append([x.clone() for x in server.result(t, frame)])
        torch.cuda.current_stream().synchronize()  # the server takes the frames back
        for t in tickets:
            server.release(t)
        return out
    return s["out"]


def work(case):
    """Bytes: every pixel's output record (16 + 4) and its material byte, each region's table entry (32) read and
    written, loaded chunks (about 128 KB each) read and written.  Flops: a pixel's ray direction, length and distance
    (24) and, for each level of a chunk's octree, the three mid-plane crossings of one descent (6)."""
    px = sum(w * h for w, h in _sizes(case))
    spec = _world(case["world"], case["side"], case["color"] >= 0.0, case["view_dist"]).spec
    regions = spec.grid[0] * spec.grid[1] * spec.grid[2]
    loaded = 2 * 131072 * case["views"] if case["kind"] == "load" else 0
    return {"bytes": 21 * px + 64 * regions * len(_sizes(case)) + loaded,
            "flops": px * (24 + 6 * int(math.log2(spec.chunk)))}


def exact(case, seed):
    """Hit distances of the one-chunk world from its dense voxels: a voxel walk along every ray in 64 bits."""
    if case["world"] != "single":
        return None
    world = _world("single", 0, False, 0.0)
    n = world.spec.wx
    solid = np.ascontiguousarray(world.dense(0, 0, 0, n, n, n).transpose(2, 1, 0)).astype(bool)
    cam = _pose(case, world, sg.Rng(seed * 1000003 + 17), case["w"], case["h"])
    f = np.float32
    # the ray of a pixel is defined in binary32, one rounding per operation
    u = ((f(2) * np.arange(cam.W, dtype=f) + f(1)) / f(cam.W) - f(1)) * f(cam.tan_half_fovy) * (f(cam.W) / f(cam.H))
    v = (f(1) - (f(2) * np.arange(cam.H, dtype=f) + f(1)) / f(cam.H)) * f(cam.tan_half_fovy)
    R = np.asarray(cam.R, f)
    d = np.stack([(R[i, 0] * u[None, :] + R[i, 1] * v[:, None]) - R[i, 2] for i in range(3)], -1)
    d = d.reshape(-1, 3).astype(np.float64)
    o = np.asarray(cam.origin, np.float64)
    with np.errstate(divide="ignore", invalid="ignore"):
        inv = 1.0 / d
        t0, t1 = (0.0 - o) * inv, (n - o) * inv
    near, far = np.fmin(t0, t1).max(1), np.fmax(t0, t1).min(1)
    t = np.maximum(near, 0.0)
    out = np.full(len(d), np.inf)
    live = np.nonzero(near < far)[0]
    live = live[far[live] > 0.0]
    axis = np.where(near[live] > 0.0, np.fmin(t0, t1)[live].argmax(1), -1)
    p = o + t[live, None] * d[live]
    step = np.where(d[live] > 0, 1, -1)
    cell = np.clip(np.floor(p).astype(np.int64), 0, n - 1)
    face = np.where(step > 0, 0, n - 1)  # the cell entered through the world's face
    for a in range(3):
        cell[axis == a, a] = face[axis == a, a]
    t = t[live]
    while len(live):
        got = solid[cell[:, 0], cell[:, 1], cell[:, 2]]
        out[live[got]] = t[got] * np.linalg.norm(d[live[got]], axis=1)
        live, cell, step = live[~got], cell[~got], step[~got]
        with np.errstate(divide="ignore", invalid="ignore"):
            cross = np.where(d[live] != 0, (cell + (step > 0) - o) / d[live], np.inf)
        a = cross.argmin(1)
        t = cross[np.arange(len(live)), a]
        cell[np.arange(len(live)), a] += step[np.arange(len(live)), a]
        inside = ((cell >= 0) & (cell < n)).all(1)
        live, cell, step, t = live[inside], cell[inside], step[inside], t[inside]
    return [None, torch.from_numpy(out.reshape(cam.H, cam.W))]
