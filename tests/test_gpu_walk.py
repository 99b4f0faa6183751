"""The casting kernels' FP32 decisions (view distance, voxel walk) at the
places where they hand over to exact arithmetic."""
from dataclasses import replace

import numpy as np
import pytest

import oracle as orc
import scenegen as sg
from gpu_util import compare, decode
from worlds import HAND32

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
