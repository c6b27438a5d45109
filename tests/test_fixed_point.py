"""Positions to fixed point and back: whole numbers and FP32 values equal to those
that FP64 arithmetic gives, next to ties too.  The functions of the load and the
export are compiled for the host (both are host and device code) and run there.

Inputs: random positions, the ones among them within 2^-12 of a tie many times
over, large and tiny ones, infinities and NaN; grids whose spacing is a power of
two and others."""
import shutil
import subprocess

import numpy as np
import pytest

SRC = r"""
#include <cmath>
#include <cstdio>
#include <vector>
#include "mpm_dev.cuh"
int main() {
    float par[5];   // units per length as a pair, dx, units per cell, cells per unit
    unsigned n[2];
    if (fread(par, 4, 5, stdin) != 5 || fread(n, 4, 2, stdin) != 2) return 1;
    std::vector<float> x(n[0]), w(n[1]);
    std::vector<int> q(n[0]), r(n[1]);
    if (fread(x.data(), 4, n[0], stdin) != n[0] || fread(r.data(), 4, n[1], stdin) != n[1]) return 1;
    for (unsigned i = 0; i < n[0]; ++i) q[i] = mpm::to_fixed(x[i], par[0], par[1], par[2], par[3]);
    for (unsigned i = 0; i < n[1]; ++i) w[i] = mpm::to_world(r[i], par[4] * par[2]);
    fwrite(q.data(), 4, n[0], stdout);
    fwrite(w.data(), 4, n[1], stdout);
    return 0;
}
"""


@pytest.fixture(scope="module")
def prog(tmp_path_factory):
    from paper_2602_01723_gb300 import build as b
    d = tmp_path_factory.mktemp("fixed")
    (d / "m.cu").write_text(SRC)
    assert shutil.which("nvcc") or b._nvcc()
    subprocess.run([b._nvcc(), *b.ARCH, "-O2", "-std=c++17", "-I", b.CSRC, "-o", str(d / "m"), str(d / "m.cu")], check=True)
    return str(d / "m")


@pytest.mark.parametrize("res, qf", [(16, 23), (24, 23), (104, 23), (192, 22), (256, 22), (1000, 20), (4096, 18)])
def test_same_as_fp64(prog, res, qf):
    rng = np.random.default_rng(res)
    dx, cell, unit = np.float32(1.0 / res), np.float32(2.0 ** qf), np.float32(2.0 ** -qf)
    u = float(cell) / float(dx)
    hi = np.float32(u)
    lo = np.float32(u - float(hi))
    x = rng.random(4_000_000).astype(np.float32)
    exact = x.astype(np.float64) / np.float64(dx) * np.float64(cell)
    tie = np.abs(np.abs(exact - np.rint(exact)) - 0.5) < 2.0 ** -12
    odd = np.array([0.0, -0.0, np.nan, np.inf, -np.inf, 3e38, -3e38, 1e-40, 7.0, -7.0], np.float32)
    x = np.concatenate([x[:500_000], x[tie], -x[tie], 3.0 * x[:1000], odd]).astype(np.float32)
    q = np.concatenate([rng.integers(-2 ** 30, 2 ** 30, 500_000), rng.integers(0, 2 ** 25, 100_000),
                        np.arange(2 ** 24 - 50, 2 ** 24 + 50), [0, 1, -1, 2 ** 31 - 1, -2 ** 31 + 1]]).astype(np.int32)
    data = b"".join([np.array([hi, lo, dx, cell, unit], np.float32).tobytes(), np.array([len(x), len(q)], np.uint32).tobytes(),
                     x.tobytes(), q.tobytes()])
    out = subprocess.run([prog], input=data, capture_output=True, check=True).stdout
    got, back = np.frombuffer(out, np.int32, len(x)), np.frombuffer(out, np.float32, len(q), 4 * len(x))
    with np.errstate(all="ignore"):
        v = x.astype(np.float64) / np.float64(dx) * np.float64(cell)
        want = np.where(np.isfinite(v), np.rint(np.clip(v, -2.0 ** 30, 2.0 ** 30)), 0.0)
    np.testing.assert_array_equal(got, want.astype(np.int64))
    np.testing.assert_array_equal(back, (q.astype(np.float64) * (np.float64(unit) * np.float64(dx))).astype(np.float32))
