"""State that beam passes share within a context: tags, buffers, the record of
the last pass.  Frames of 1280 x 720 take the pass where it can run, frames of
1600 x 1000 always; each equals the frame without the pass bit for bit."""
import os
import threading
import time
from dataclasses import replace

import pytest

import scenegen as sg
from worlds import MED64

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2505_02017_gb300 as aok  # noqa: E402

OPTIONAL, REQUIRED = (1280, 720), (1600, 1000)


class Setup:
    """A context with its initial settings, a scene of it, and frames without the pass to compare with."""

    def __init__(self, budget=0):
        self.c = aok.Context(0, budget_bytes=budget)
        self.world = sg.World(MED64)
        self.sc = aok.Scene.from_world(self.c, self.world, threads=4)

    def cam(self, k, size=OPTIONAL):
        return sg.ground_camera(self.world, (4, 9, 12)[k % 3], *size, z_lo=4, z_hi=40)

    def ref(self, cam, tau=1.5):
        aok.set_beam(self.c, False)
        out = aok.alloc_frame(cam.W, cam.H)
        aok.render(self.c, self.sc, cam, tau, *out)
        torch.cuda.synchronize()
        aok.set_beam(self.c, True)
        return out

    def close(self):
        self.sc.destroy()
        self.c.close()


def equal(x, y):
    return torch.equal(x[0].cpu(), y[0].cpu()) and torch.equal(x[1].cpu().view(torch.int32), y[1].cpu().view(torch.int32))


def buffers(kind, cam):
    if kind == "host":
        return (torch.empty((cam.H, cam.W, 4), dtype=torch.int32, pin_memory=True),
                torch.empty((cam.H, cam.W), dtype=torch.float32, pin_memory=True))
    return aok.alloc_frame(cam.W, cam.H)


def draw(s, kind, cam, srv=None, out=None, stream=None):
    """The frame of `cam` through one of the calls that run the pass; waits for it (not for other streams when one
    is given)."""
    out = out or (None if kind == "serve" else buffers(kind, cam))
    if kind == "host":
        aok.host_frame_wait(s.c, aok.render_host_async(s.c, s.sc, cam, 1.5, *out))
        return out
    if kind == "serve":
        tk = srv.submit(s.sc, cam, 1.5)
        st, f = srv.wait(tk, 20000)
        assert st == aok.AOK_OK
        with torch.cuda.stream(stream):
            out = tuple(x.clone() for x in srv.result(tk, f))
        torch.cuda.current_stream().synchronize() if stream is None else stream.synchronize()
        assert srv.release(tk) == aok.AOK_OK
        return out
    if kind == "batch":
        aok.render_batch(s.c, [aok.make_view(s.sc, cam, 1.5, *out)], stream=stream)
    elif kind == "tiles":
        aok.render_tiles(s.c, s.sc, cam, 1.5, *out, stream=stream)
    else:
        aok.render(s.c, s.sc, cam, 1.5, *out, stream=stream)
    torch.cuda.synchronize() if stream is None else stream.synchronize()
    return out


@pytest.mark.parametrize("size", [OPTIONAL, REQUIRED], ids=["optional", "required"])
@pytest.mark.parametrize("kind", ["single", "tiles", "host", "batch", "serve"])
def test_tags_start_over(kind, size):
    """Bounds left by the last passes before the tags start over are not read as the new passes'."""
    s = Setup()
    cams = [s.cam(k, size) for k in range(3)]
    refs = [s.ref(m) for m in cams]
    srv = aok.Server(s.c, max_slots=4, max_batch=2, n_streams=1) if kind == "serve" else None
    before = aok.beam_passes(s.c)
    aok.beam_tags_left(s.c, 4)
    for i in range(12):  # (host frames: each of the three slots on both sides)
        assert equal(draw(s, kind, cams[i % 3], srv), refs[i % 3]), i
    assert aok.beam_passes(s.c) == before + 12
    if srv:
        srv.stop()
    s.close()


def test_info_is_of_the_last_view():
    """aok_beam_info reports the last single view's pass, its bounds and its level counts together, also for
    frames that need not take the pass; a batch in between changes neither."""
    s = Setup()
    with pytest.raises(aok.AokError):
        aok.beam_info(s.c)
    seen = {}
    for size in (OPTIONAL, REQUIRED, OPTIONAL):
        cam = s.cam(0, size)
        draw(s, "single", cam)
        b, levels = aok.beam_info(s.c)
        assert b.shape == ((cam.H + 3) // 4, (cam.W + 7) // 8) and levels[0] > 0
        draw(s, "batch", s.cam(1, REQUIRED))
        assert (aok.beam_info(s.c)[0] == b).all() and aok.beam_info(s.c)[1] == levels
        # the same pass by itself (kept, in the buffer of the large frames)
        aok.beam_selected(s.c, s.sc, cam)
        b2, levels2 = aok.beam_info(s.c)
        assert (b2 == b).all() and levels2 == levels
        assert seen.setdefault(size, levels) == levels
    assert seen[OPTIONAL] != seen[REQUIRED]
    aok.beam_selected(s.c, s.sc, s.cam(0, REQUIRED))
    draw(s, "single", s.cam(2))
    assert aok.beam_info(s.c)[0].shape == (180, 160)
    s.close()


def test_two_casts_of_one_selection():
    """Two casts of one selection on two streams, the first held back, and then another frame's pass: it must
    not replace the bounds before both have read them."""
    s = Setup()
    cams = [s.cam(k) for k in range(3)]
    refs = [s.ref(m) for m in cams]
    outs = [aok.alloc_frame(m.W, m.H) for m in cams]
    s1, s2, s3 = (torch.cuda.Stream() for _ in range(3))
    sc3 = aok.Scene.from_world(s.c, s.world, threads=4)  # (its own chunk table)
    aok.select_beam(s.c, s.sc, cams[0], 1.5)
    assert aok.beam_info(s.c)[1][0] > 0
    torch.cuda.synchronize()
    with torch.cuda.stream(s1):
        torch.cuda._sleep(40_000_000)  # about 20 ms
    aok.cast_selected(s.c, s.sc, cams[0], *outs[0], stream=s1)
    aok.cast_selected(s.c, s.sc, cams[0], *outs[1], stream=s2)
    aok.render(s.c, sc3, cams[2], 1.5, *outs[2], stream=s3)
    torch.cuda.synchronize()
    assert equal(outs[0], refs[0]) and equal(outs[1], refs[0]) and equal(outs[2], refs[2])
    sc3.destroy()
    s.close()


@pytest.mark.parametrize("room_kb", range(0, 1200, 200))
def test_server_batch_of_both_kinds_in_a_tight_budget(room_kb):
    """The queues of the large request's pass are the last to fit: what the small request's pass uses must stay."""
    s = Setup()
    used = s.c.memory()[0]
    s.close()
    need = sum(w * h * 20 + ((w * h) >> 2) for w, h in (OPTIONAL, REQUIRED)) + (33 << 20)
    s = Setup(used + need + (room_kb << 10))
    cams = [s.cam(0), s.cam(1, REQUIRED), s.cam(2)]
    refs = [s.ref(m) for m in cams]
    srv = aok.Server(s.c, max_slots=8, max_batch=4, n_streams=1)
    for k in ((0, 1), (1, 2), (2, 1), (0, 1)):
        held = [srv.submit(s.sc, cams[i], 1.5) for i in k]
        for i, tk in zip(k, held):
            st, f = srv.wait(tk, 20000)
            assert st == aok.AOK_OK and equal(srv.result(tk, f), refs[i])
        torch.cuda.synchronize()
        for tk in held:
            assert srv.release(tk) == aok.AOK_OK
    assert aok.beam_passes(s.c) > 0
    srv.stop()
    s.close()


@pytest.mark.parametrize("kind", ["single", "tiles", "host", "batch", "serve"])
@pytest.mark.parametrize("room", [None, 1 << 20])
def test_optional_pass_takes_nothing_from_the_budget(kind, room):
    """The pass runs for frames of 1280 x 720 whatever the budget (room: what it leaves beside the scene and the
    call's own buffers), also after an allocation that failed; the frames change neither the context's charged
    memory nor, from the first one on, the device's free memory."""
    if room is not None:
        s = Setup()
        for _ in range(3 if kind != "serve" else 0):
            draw(s, kind, s.cam(0))
        used = s.c.memory()[0]
        s.close()
    s = Setup(0 if room is None else used + (20 << 20 if kind == "serve" else 0) + room)
    cams = [s.cam(k) for k in range(3)]
    refs = [s.ref(m) for m in cams]
    srv = aok.Server(s.c, max_slots=4, max_batch=2, n_streams=1) if kind == "serve" else None
    aok.set_beam(s.c, False)
    for _ in range(3):  # the call's own buffers (three slots of host frames)
        draw(s, kind, cams[0], srv)
    aok.set_beam(s.c, True)
    mem, free = s.c.memory(), torch.cuda.mem_get_info()[0]
    n = aok.beam_passes(s.c)
    for i in range(2):
        for m, r in zip(cams, refs):
            assert equal(draw(s, kind, m, srv), r)
            n += 1
            assert aok.beam_passes(s.c) == n and s.c.memory() == mem
        assert torch.cuda.mem_get_info()[0] == free
        if room is not None:
            with pytest.raises(aok.AokError):
                aok.Scene(s.c, s.world.spec, node_words=64 << 20, leaves=1, mat_bytes=1)
        free = torch.cuda.mem_get_info()[0]
    if srv:
        srv.stop()
    s.close()


def test_optional_passes_beyond_their_room():
    """Views beyond the block's room are cast without bounds: the last of 30 in a batch, a frame of one row."""
    s = Setup()
    cams = [s.cam(k) for k in range(3)]
    refs = [s.ref(m) for m in cams]
    outs = [aok.alloc_frame(*OPTIONAL) for _ in range(30)]
    n = aok.beam_passes(s.c)
    aok.render_batch(s.c, [aok.make_view(s.sc, cams[i % 3], 1.5, *o) for i, o in enumerate(outs)])
    torch.cuda.synchronize()
    assert all(equal(o, refs[i % 3]) for i, o in enumerate(outs)) and aok.beam_passes(s.c) == n + 1
    row = replace(cams[0], W=900000, H=1)
    ref = s.ref(row)
    for kind in ("single", "tiles", "host"):
        assert equal(draw(s, kind, row), ref)
    assert aok.beam_passes(s.c) == n + 1
    s.close()


def test_frames_without_the_pass_do_not_wait():
    """A large frame's call waits for the device (its buffer grows behind 400 ms of other work); a small frame
    of another scene is enqueued meanwhile by another thread."""
    s = Setup()
    sc2 = aok.Scene.from_world(s.c, s.world, threads=4)
    small, big = s.cam(0, (320, 180)), s.cam(1, (2000, 1200))
    refs = s.ref(small), s.ref(big)
    outs = aok.alloc_frame(320, 180), aok.alloc_frame(2000, 1200)
    draw(s, "single", s.cam(1, REQUIRED))
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    aok.render(s.c, sc2, small, 1.5, *outs[0], stream=s2)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    with torch.cuda.stream(s1):
        torch.cuda._sleep(800_000_000)
    th = threading.Thread(target=lambda: aok.render(s.c, s.sc, big, 1.5, *outs[1], stream=s1))
    th.start()
    time.sleep(0.05)
    t1 = time.perf_counter()
    aok.render(s.c, sc2, small, 1.5, *outs[0], stream=s2)
    t2 = time.perf_counter()
    th.join()
    torch.cuda.synchronize()
    t3 = time.perf_counter()
    assert t3 - t0 > 0.3 and t2 - t1 < 0.1, (t3 - t0, t2 - t1)
    assert equal(outs[0], refs[0]) and equal(outs[1], refs[1])
    sc2.destroy()
    s.close()


def test_threads_with_scenes_of_their_own():
    """Four host threads, each with a scene and a stream, sizes without the pass and with the optional one."""
    s = Setup()
    scenes = [aok.Scene.from_world(s.c, s.world, threads=4) for _ in range(4)]
    cams = [s.cam(k, size) for k in range(3) for size in (OPTIONAL, (320, 180))]
    refs = [s.ref(m) for m in cams]
    bad = []

    def work(i):
        stream = torch.cuda.Stream()
        for k in range(60):
            j = (k + i) % len(cams)
            out = aok.alloc_frame(cams[j].W, cams[j].H)
            aok.render(s.c, scenes[i], cams[j], 1.5, *out, stream=stream)
            stream.synchronize()
            if not equal(out, refs[j]):
                bad.append((i, k))

    torch.cuda.synchronize()
    ths = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for th in ths:
        th.start()
    for th in ths:
        th.join()
    assert not bad
    for sc in scenes:
        sc.destroy()
    s.close()


@pytest.mark.parametrize("kind", ["single", "tiles", "host", "batch", "serve"])
def test_optional_pass_waits_for_no_other_stream(kind):
    """A frame of 1280 x 720 beside a large frame whose stream is held back for 400 ms is there at once, and takes
    the pass again afterwards."""
    s = Setup()
    sc2 = aok.Scene.from_world(s.c, s.world, threads=4)
    cam, big = s.cam(0), s.cam(1, REQUIRED)
    ref, ref2 = s.ref(cam), s.ref(big)
    srv = aok.Server(s.c, max_slots=4, max_batch=2, n_streams=1) if kind == "serve" else None
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    out = None if kind == "serve" else buffers(kind, cam)
    out2 = aok.alloc_frame(big.W, big.H)
    for _ in range(3):
        draw(s, kind, cam, srv, out, s2)
        aok.render(s.c, sc2, big, 1.5, *out2, stream=s1)
    torch.cuda.synchronize()
    with torch.cuda.stream(s1):
        torch.cuda._sleep(800_000_000)
    aok.render(s.c, sc2, big, 1.5, *out2, stream=s1)
    t0 = time.perf_counter()
    got = draw(s, kind, cam, srv, out, s2)
    t1 = time.perf_counter()
    held = not s1.query()
    torch.cuda.synchronize()
    assert held and t1 - t0 < 0.1, t1 - t0
    assert equal(got, ref) and equal(out2, ref2)
    n = aok.beam_passes(s.c)
    assert equal(draw(s, kind, cam, srv, out, s2), ref) and aok.beam_passes(s.c) == n + 1
    if srv:
        srv.stop()
    sc2.destroy()
    s.close()


def test_tune_without_arguments_restores_a_contexts_settings():
    """Levels of the walk and the sizes that take it, after other settings and beam_tune(ctx), are a fresh
    context's (the constants those of aok.h)."""
    hdr = open(os.path.join(os.path.dirname(__file__), "..", "include", "aok.h")).read()
    for name in ("BEAM_REFINE", "BEAM_MIN_PIXELS", "BEAM_MIN_OPTIONAL"):
        assert f"#define AOK_{name} {getattr(aok, name)}\n" in hdr
    s = Setup()
    cams = [s.cam(0, size) for size in ((1000, 799), OPTIONAL, REQUIRED)]

    def walks():
        out = []
        for m in cams:
            n = aok.beam_passes(s.c)
            draw(s, "single", m)
            out.append(aok.beam_info(s.c)[1] if aok.beam_passes(s.c) > n else None)
        return out

    fresh = walks()
    assert fresh[0] is None and fresh[1] and fresh[2]
    aok.beam_tune(s.c, 4, 3, 100000, 64)
    assert walks() != fresh
    aok.beam_tune(s.c)
    assert walks() == fresh
    aok.beam_limits(s.c, 1500000, 1500000)
    assert walks() == [None, None, fresh[2]]
    aok.beam_limits(s.c, 1500000, 790000)
    assert walks()[1:] == fresh[1:] and walks()[0]
    with pytest.raises(aok.AokError):
        aok.beam_limits(s.c, 1, 2)
    s.close()


@pytest.mark.parametrize("k", [-126, -123, -122, -121, -120, -119, -118, -112, -60, -21, -20, 20, 21, 60, 100, 126])
def test_camera_matrix_of_any_scale(k):
    """A matrix scaled by 2^k has the same rays but for their lengths: the frame's hits are those of k = 0 and
    equal with the pass and without, up to the ends of binary32."""
    s = Setup()
    for seed in range(3):
        one = s.cam(seed, (403, 217))
        R = (one.R.astype("float64") * 2.0 ** k).astype("float32")
        cam = replace(one, R=R)
        ref, plain = s.ref(cam), s.ref(one)
        aok.beam_tune(s.c, 16, 2, 0, 0)
        on = draw(s, "single", cam)
        b, _ = aok.beam_info(s.c)
        draw(s, "single", one)
        b1, _ = aok.beam_info(s.c)
        aok.beam_tune(s.c)
        assert equal(on, ref)
        if (R.astype("float64") == one.R * 2.0 ** k).all() and k > -118:
            assert torch.equal(ref[0], plain[0])
            if k < 120:
                assert (b == b1).mean() > 0.99
        assert not (b > 2**31 - 2).all()
    s.close()


def test_optional_passes_beside_a_capture():
    """First frames of 0.8-1.5 M pixels on one stream while another one is captured: the capture lives on."""
    s = Setup()
    sc2 = aok.Scene.from_world(s.c, s.world, threads=4)
    small, cams = s.cam(0, (320, 180)), [s.cam(1), s.cam(2, (1400, 1000)), s.cam(0)]
    refs = [s.ref(m) for m in (small, *cams)]
    outs = [aok.alloc_frame(m.W, m.H) for m in (small, *cams)]
    s1, s2, g = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    n = aok.beam_passes(s.c)
    with torch.cuda.graph(g, stream=s1):
        aok.render(s.c, s.sc, small, 1.5, *outs[0], stream=s1)
        for m, o in zip(cams, outs[1:]):
            aok.render(s.c, sc2, m, 1.5, *o, stream=s2)
    s2.synchronize()
    assert aok.beam_passes(s.c) == n + 3
    g.replay()
    torch.cuda.synchronize()
    assert all(equal(o, r) for o, r in zip(outs, refs))
    sc2.destroy()
    s.close()
