"""The casting kernels' FP32 decisions (view distance, voxel walk) at the
places where they hand over to exact arithmetic."""
import ctypes
from dataclasses import replace

import numpy as np
import pytest

import scenegen as sg
from worlds import HAND32, MED64, MULTI32

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2505_02017_gb300 as aok  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    c = aok.Context(0)
    yield c
    c.close()


def _render(ctx, sc, cam, tau=1.0):
    hit, t = aok.alloc_frame(cam.W, cam.H)
    aok.render(ctx, sc, cam, tau, hit, t)
    torch.cuda.synchronize()
    return hit, t


@pytest.mark.parametrize("rel", [0.0, -2.0 ** -23, 2.0 ** -23, -2.0 ** -18, 2.0 ** -18, -2.0 ** -16, 2.0 ** -16])
def test_view_distance_at_the_limit(ctx, rel):
    # a straight-down ray meets the cube's top after exactly 20.5 voxels
    vd = float(np.float32(20.5 * (1.0 + rel)))
    w = sg.World(replace(HAND32, name=f"limit{rel}", view_dist=vd), boxes=[(4, 4, 4, 8, 8, 8, 0)])
    sc = aok.Scene.from_world(ctx, w, threads=2)
    hit, t = _render(ctx, sc, sg.make_camera((8.25, 8.5, 32.5), (0.0, 0.0, -1.0), 1, 1))
    found = bool((int(hit[0, 0, 3]) >> 19) & 1)
    assert found == (20.5 <= vd)
    assert float(t[0, 0]) == (20.5 if found else np.inf)
    sc.destroy()


# The FP32 walk against the exact march (aok_render_counted runs it), every
# pixel of every record: generic views, and directions and origins on voxel
# and chunk planes, where crossings tie.
WALK_WORLDS = [replace(HAND32, name="chunk8", seed=5, wx=64, wy=64, wz=64, chunk=8, n_lods=1, octaves=3, period0=32,
                       h_min=8, h_max=40, crust=2, n_boxes=12, box_min=2, box_max=9),
               MULTI32, MED64, replace(MULTI32, name="multi32far", view_dist=60.0), sg.city(2, 1024)]
WALK_DIRS = [(1.0, 1.0, -1.0), (-1.0, 2.0, -2.0), (1.0, -1.0, -0.5), (1.0, 0.0, -1.0), (0.0, 0.0, -1.0), (1.0, 1e-6, -0.2)]


def _equal_to_march(ctx, sc, cam, tau):
    hit, t = _render(ctx, sc, cam, tau)
    hit2, t2 = aok.alloc_frame(cam.W, cam.H)
    counts = torch.zeros((cam.H, cam.W, 3), dtype=torch.int32, device="cuda")
    aok.render_counted(ctx, sc, cam, tau, hit2, t2, counts)
    torch.cuda.synchronize()
    assert torch.equal(hit, hit2) and torch.equal(t.view(torch.int32), t2.view(torch.int32))
    return float(((hit[..., 3] >> 19) & 1).float().mean())


@pytest.mark.parametrize("beam", [0, 1])
@pytest.mark.parametrize("spec", WALK_WORLDS, ids=lambda s: s.name)
def test_walk_equals_exact_march(ctx, spec, beam):
    w = sg.World(spec)
    sc = aok.Scene.from_world(ctx, w)
    cams = [sg.orbit_camera(spec, 3 + s, 211 + s, 97 + s, radius=1.3 * spec.wx) for s in range(2)]
    cams += [sg.ground_camera(w, s, 203, 117, z_lo=3, z_hi=max(6, spec.wz // 16)) for s in range(2)]
    for d in WALK_DIRS:
        cams.append(sg.make_camera((spec.wx / 2, spec.wy / 2, spec.wz * 0.75), d, 63, 41))
        cams.append(sg.make_camera((-5.0, spec.wy / 4, spec.wz * 0.75 + 0.25), d, 33, 64))
        cams.append(sg.make_camera((spec.wx * 0.75, spec.wy / 2, spec.wz + 8.0), d, 71, 44))
    aok.beam_tune(ctx, 8, 2, 0 if beam else 1 << 40, 0)
    hits = sum(_equal_to_march(ctx, sc, c, tau) for c in cams for tau in (1.0, 3.0))
    aok.beam_tune(ctx)
    assert hits > 1.0
    sc.destroy()


@pytest.mark.parametrize("scale", [2.0 ** -80, 2.0 ** -41, 2.0 ** 41, 2.0 ** 60])
def test_walk_of_scaled_directions(ctx, scale):
    # only the ratios of a direction's components matter to the walk
    w = sg.World(MED64)
    sc = aok.Scene.from_world(ctx, w)
    cam = sg.ground_camera(w, 4, 160, 90, z_lo=4, z_hi=40)
    want, _ = _render(ctx, sc, cam, 1.5)
    cam.R = (cam.R.astype(np.float64) * np.array([1.0, 1.0, scale])).astype(np.float32)
    cam.tan_half_fovy = np.float32(float(cam.tan_half_fovy) * scale)
    # u and v scale with tan_half_fovy, the view axis with its column: the same rays, longer or shorter
    got, _ = _render(ctx, sc, cam, 1.5 / scale)
    assert torch.equal(want, got)
    _equal_to_march(ctx, sc, cam, 1.5 / scale)
    sc.destroy()


@pytest.mark.parametrize("size", [(1, 1), (3, 2), (61, 79), (64, 76), (139, 70), (139, 71), (278, 140), (278, 141), (399, 390)])
def test_small_frames_at_the_edges_of_the_warp_tiles(ctx, size):
    # frames around the sizes where a warp takes 1, 2, 4, 8, 16 or 32 rays (152 SMs), with ragged edges
    w = sg.World(MED64)
    sc = aok.Scene.from_world(ctx, w, threads=4)
    aok.beam_tune(ctx, 16, 2, 1 << 40, 0)
    for seed in (4, 9):
        _equal_to_march(ctx, sc, sg.ground_camera(w, seed, *size, z_lo=4, z_hi=40), 1.5)
    aok.beam_tune(ctx)
    sc.destroy()


def test_blob_nodes_in_any_order(ctx):
    # a blob's nodes may lie in any order, with unused words between them: the same scene
    w = sg.World(MED64)
    built = aok.BuiltWorld(w)
    spec = MED64
    a = aok.Scene.from_world(ctx, w, built=built)
    b = aok.Scene(ctx, spec, 2 * built.node_words, built.leaves, built.mat_bytes)
    rng = np.random.default_rng(7)
    gx, gy, _ = b.grid
    keep = []
    for i in range(len(built)):
        for lod in range(spec.n_lods):
            c, blob = built.blob(i, lod)
            if blob.n_node_words:
                src = np.ctypeslib.as_array(ctypes.cast(blob.nodes, ctypes.POINTER(ctypes.c_uint32)), (blob.n_node_words,))
                depth, todo = {int(blob.root): 0}, [int(blob.root)]
                last = int(np.log2(spec.chunk >> lod)) - 3  # depth of the nodes above the leaf blocks
                while todo:
                    n = todo.pop()
                    if depth[n] < last:
                        for ch in src[n + 2:n + 2 + int(src[n]).bit_count()]:
                            if int(ch) not in depth:
                                depth[int(ch)] = depth[n] + 1
                                todo.append(int(ch))
                order = rng.permutation(sorted(depth))
                at, pos = {}, 0
                for n in order:
                    at[int(n)] = pos
                    pos += 2 + int(src[n]).bit_count() + int(rng.integers(0, 2))
                dst = np.full(pos + 1, 0xDEADBEEF, np.uint32)
                for n in order:
                    n, k = int(n), int(src[n]).bit_count()
                    dst[at[n]:at[n] + 2] = src[n:n + 2]
                    ch = src[n + 2:n + 2 + k]
                    dst[at[n] + 2:at[n] + 2 + k] = ch if depth[n] == last else [at[int(x)] for x in ch]
                keep.append(dst)
                blob.nodes, blob.n_node_words, blob.root = dst.ctypes.data, len(dst), at[int(blob.root)]
            b.upload(c % gx, (c // gx) % gy, c // (gx * gy), lod, blob)
    for seed in (4, 9):
        cam = sg.ground_camera(w, seed, 203, 117, z_lo=4, z_hi=40)
        x, y = _render(ctx, a, cam, 1.5), _render(ctx, b, cam, 1.5)
        assert torch.equal(x[0], y[0]) and torch.equal(x[1].view(torch.int32), y[1].view(torch.int32))
    a.destroy()
    b.destroy()


def test_small_frame_in_a_cuda_graph(ctx):
    # the selection and the cast that is launched beside it, captured and replayed
    w = sg.World(MED64)
    sc = aok.Scene.from_world(ctx, w, threads=4)
    cam = sg.ground_camera(w, 4, 160, 90, z_lo=4, z_hi=40)
    want = _render(ctx, sc, cam, 1.5)
    hit, t = aok.alloc_frame(cam.W, cam.H)
    s = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s):
        aok.render(ctx, sc, cam, 1.5, hit, t, stream=s)
    for _ in range(3):
        hit.zero_()
        t.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(want[0], hit) and torch.equal(want[1].view(torch.int32), t.view(torch.int32))
    sc.destroy()
