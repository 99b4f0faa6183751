"""Chunk upload when host memory runs out: AOK_E_OOM, the pools as before, the
next upload as if nothing had happened.  A preloaded operator new fails the
k-th allocation of an upload, for every k of one in a fresh context."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HOOK = r"""
#include <cstdlib>
#include <new>
static long n, fail;
extern "C" long hook_arm(long k) { long r = n; n = 0; fail = k; return r; }
void* operator new(std::size_t s) {
    n++;
    if (fail && n == fail) throw std::bad_alloc();
    void* p = std::malloc(s ? s : 1);
    if (!p) throw std::bad_alloc();
    return p;
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
"""

SCRIPT = r"""
import ctypes, sys
sys.path[:0] = [sys.argv[1], sys.argv[1] + "/tests"]
import paper_2505_02017_gb300 as aok
import scenegen as sg
from dataclasses import replace
from worlds import MED64
color = float(sys.argv[3])
hook = ctypes.CDLL(sys.argv[2])
hook.hook_arm.restype = ctypes.c_long
w = sg.World(replace(MED64, mat_mode=1) if color >= 0 else MED64)
built = aok.BuiltWorld(w)
c, blob = max((built.blob(i, 0) for i in range(len(built))), key=lambda b: b[1].n_node_words)
L, failed, calls = aok.lib(), 0, 1 << 30
k = 0
while k <= calls:
    ctx = aok.Context(0)
    sc = aok.Scene(ctx, w.spec, built.node_words, built.leaves, built.mat_bytes)
    sc.set_color_blocks(color)
    gx, gy, _ = sc.grid
    args = (ctx.h, sc.id, c % gx, (c // gx) % gy, c // (gx * gy), 0, ctypes.byref(blob))
    empty = sc.usage()
    hook.hook_arm(k)
    st = L.aok_scene_upload_chunk(*args)
    n = hook.hook_arm(0)
    if k == 0:
        assert st == 0
        calls, full = n, sc.usage()
        assert calls >= 5
    else:
        assert st == aok.AOK_E_OOM, (k, st)
        assert sc.usage() == empty, (k, sc.usage())
        failed += 1
        assert L.aok_scene_upload_chunk(*args) == 0 and sc.usage() == full, k
    sc.destroy()
    ctx.close()
    k += 1
print("failed allocations", failed)
"""


@pytest.mark.parametrize("color", [-1.0, 0.05], ids=["raw", "blocks"])
def test_upload_without_host_memory(tmp_path, color):
    src, so, script = tmp_path / "hook.cpp", tmp_path / "hook.so", tmp_path / "run.py"
    src.write_text(HOOK)
    script.write_text(SCRIPT)
    subprocess.check_call(["g++", "-O1", "-shared", "-fPIC", str(src), "-o", str(so)])
    r = subprocess.run([sys.executable, str(script), ROOT, str(so), str(color)], env=dict(os.environ, LD_PRELOAD=str(so)),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert int(r.stdout.split()[-1]) >= 5
