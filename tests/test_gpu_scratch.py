"""Scratch of the fill and the splat where memory is short, and its return.

Shortage is made on the host: a library of two functions that the child process
loads before the CUDA runtime answers one kind of allocation as the runtime does
when there is no memory left.  The scratch is then taken from the device's default
pool, and a context's own allocation is tried again after the kept scratch has gone
back.  A program without a context gives the kept scratch back by a call."""
import os
import subprocess
import sys

import pytest

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#include <dlfcn.h>
#include <stddef.h>
int pool_fails, malloc_fails;   /* calls still to be refused */
static void *real(const char *name) { return dlsym(dlopen("libcudart.so.13", RTLD_LAZY), name); }
int cudaMallocFromPoolAsync(void **p, size_t n, void *pool, void *s) {
    if (pool_fails > 0) { --pool_fails; return 2; }   /* cudaErrorMemoryAllocation */
    return ((int (*)(void **, size_t, void *, void *))real("cudaMallocFromPoolAsync"))(p, n, pool, s);
}
int cudaMalloc(void **p, size_t n) {
    if (malloc_fails > 0) { --malloc_fails; return 2; }
    return ((int (*)(void **, size_t))real("cudaMalloc"))(p, n);
}
"""

CHILD = r"""
import ctypes, sys
shim = ctypes.CDLL(sys.argv[1], ctypes.RTLD_GLOBAL)
import numpy as np
import torch
from paper_2602_01723_gb300 import _lib, scenes
from paper_2602_01723_gb300.sim import Simulator, mcis, render
pool_fails, malloc_fails = (ctypes.c_int.in_dll(shim, k) for k in ("pool_fails", "malloc_fails"))
m = scenes.mcis_case((3000,) * 3, (200_000,) * 3, (500,) * 3)
fill = lambda: mcis(m["surf_off"], m["surf"], m["cand_off"], m["cand"], m["draw_off"], m["u"])
rng = np.random.default_rng(1)
f32 = lambda a: np.asarray(a, np.float32)
splat = lambda: render(f32(P), f32(np.tile([1e-4, 0, 0, 1e-4, 0, 1e-4], (500, 1))), f32(P), f32(np.full(500, 0.5)),
                       scenes.camera(64, 48)[0], *scenes.camera(64, 48)[1:], 64, 48)
P = 0.3 + 0.4 * rng.random((500, 3))
want = [fill()["picked"], splat()[0]]

pool_fails.value = 1
assert torch.equal(fill()["picked"], want[0])
assert pool_fails.value == 0
pool_fails.value = 2
assert torch.equal(splat()[0], want[1])
assert pool_fails.value == 0

fill()
torch.cuda.synchronize()
kept = torch.cuda.mem_get_info()[0]
assert _lib.lib().mpm_release_scratch() == 0
back = torch.cuda.mem_get_info()[0] - kept
assert back >= 16 << 20, back                      # 600,000 candidates take some 40 MB of scratch
assert torch.equal(fill()["picked"], want[0])

sc = scenes.cube_8k()
malloc_fails.value = 1
s = Simulator.from_scene(sc)
assert malloc_fails.value == 0
malloc_fails.value = 1
s.load_scene(sc)
s.step(3)
s.sync()
s.close()
print("fine")
"""


def test_scratch_where_memory_is_short(tmp_path):
    from __graft_entry__ import build
    build()
    src, lib = tmp_path / "shim.c", tmp_path / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(lib), str(src), "-ldl"], check=True)
    r = subprocess.run([sys.executable, "-c", CHILD, str(lib)], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "fine" in r.stdout, r.stdout + r.stderr
