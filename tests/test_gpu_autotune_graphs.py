"""The autotuner's timed passes capture and instantiate no CUDA graph: the warm-up
pass of each setting has done it, the first setting on a fresh context included.

The calls are seen by a library of two functions that the child process loads
before the CUDA runtime, so that libmpm's calls pass through it: each trial records
an event before and after the warm-up pass and the timed one."""
import os
import re
import subprocess
import sys

import pytest

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#include <dlfcn.h>
char seen[4096];
int n_seen;
static void note(char c) { if (n_seen < 4095) seen[n_seen++] = c; }
static void *real(const char *name) { return dlsym(dlopen("libcudart.so.13", RTLD_LAZY), name); }
int cudaEventRecord(void *e, void *s) {
    note('E');
    return ((int (*)(void *, void *))real("cudaEventRecord"))(e, s);
}
int cudaGraphInstantiate(void *ex, void *g, unsigned long long f) {
    note('G');
    return ((int (*)(void *, void *, unsigned long long))real("cudaGraphInstantiate"))(ex, g, f);
}
"""

CHILD = r"""
import ctypes, sys
shim = ctypes.CDLL(sys.argv[1], ctypes.RTLD_GLOBAL)
import torch
from paper_2602_01723_gb300 import scenes
from paper_2602_01723_gb300.sim import Simulator
sc = scenes.cube_8k()
s = Simulator.from_scene(sc)
s.load_scene(sc)
s.sync()
n = ctypes.c_int.in_dll(shim, "n_seen")
n.value = 0
s.autotune(int(sys.argv[2]))
print("seen", ctypes.string_at(ctypes.addressof(ctypes.c_char.in_dll(shim, "seen")), n.value).decode())
s.close()
"""


@pytest.mark.parametrize("n_substeps", [10, 20, 40])
def test_timed_passes_capture_nothing(tmp_path, n_substeps):
    from __graft_entry__ import build
    build()
    src, lib = tmp_path / "shim.c", tmp_path / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(lib), str(src), "-ldl"], check=True)
    r = subprocess.run([sys.executable, "-c", CHILD, str(lib), str(n_substeps)], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr
    calls = r.stdout.split("seen", 1)[1].strip()
    assert "G" in calls
    assert re.fullmatch(r"(EG*EEE){8}", calls), calls
