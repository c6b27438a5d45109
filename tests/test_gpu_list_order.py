"""The direct-binning substeps: every 16th one takes its scatter packets in
(rank, bank) order and lists the particles so, the ones between scatter in
list order.  Runs that end just before, at and after such a substep, replayed
from graphs and launched directly, against the FP64 oracle, at particle counts
around the edges of warps and chunks and for both CTA sizes.

Tolerances, from those of the forward parity tests: positions 1e-4 dx (their
bound for 100 substeps); v 2e-5 of max |v| per substep, C the (6 / dx) |dv|
it inherits, F 2e-5 per substep, each times the number of substeps."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2602_01723_gb300 import scenes  # noqa: E402


def small_scene(n, plastic):
    rng = np.random.default_rng(n)
    R = 16
    x = 0.35 + 0.3 * rng.random((n, 3))
    v = rng.normal(0.0, 0.5, (n, 3))
    F = np.eye(3) + 0.03 * rng.standard_normal((n, 3, 3))
    C = 2.0 * rng.standard_normal((n, 3, 3))
    mats = [scenes.material(0, plastic, 1e4, 0.3, 100.0, yield_stress=3e2)]
    f32 = lambda a: np.ascontiguousarray(a, np.float32)  # noqa: E731
    sc = scenes.Scene("small", R, 1e-4, 0, f32(x), f32(v), np.full(n, (0.5 / R) ** 3, np.float32),
                      np.zeros(n, np.int32), mats)
    return sc, f32(C), f32(F)


@pytest.mark.parametrize("n", [1, 33, 127, 129, 1000])
@pytest.mark.parametrize("chunk", [64, 128])
def test_runs_around_an_ordered_substep(orc, n, chunk):
    from __graft_entry__ import build
    build()
    from paper_2602_01723_gb300.sim import Simulator
    sc, C, F = small_scene(n, n % 3)
    cfg = orc.Cfg(sc.grid_res, sc.dx, sc.dt, sc.gravity)
    mat = orc.Material.from_table(sc.vol, sc.mat_id, sc.materials)
    s = Simulator.from_scene(sc, chunk=chunk)
    for n_sub in (2, 16, 17, 18, 19, 36):
        ref = orc.run(cfg, orc.new_state(sc.x, sc.v, C, F), mat, n_sub)
        vmax = np.abs(ref["v"]).max()
        for graph in (True, False):
            s.set_tuning(scatter=1, chunk=chunk, use_graph=graph)
            s.load(sc.x, sc.vol, sc.mat_id, v=sc.v, C=C, F=F)
            s.step(n_sub)
            s.sync()
            got = {k: a.double().cpu().numpy() for k, a in s.get().items()}
            err = {k: np.abs(got[k] - ref[k]).max() for k in got}
            assert err["x"] < 1e-4 * sc.dx, (n_sub, graph, err)
            assert err["v"] < n_sub * 2e-5 * vmax, (n_sub, graph, err)
            assert err["C"] < n_sub * 2e-5 * vmax * 6.0 / sc.dx, (n_sub, graph, err)
            assert err["F"] < n_sub * 2e-5, (n_sub, graph, err)
    s.close()
