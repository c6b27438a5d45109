"""The key frame's substep gives its signals from the P2G and G2P kernels and
writes no new state: particle counts around the edges of warps and chunks, both
CTA sizes, every scatter strategy, the common and the further material models,
with and without the signals as outputs, against the FP64 oracle; the key frames
and the current state are left as they were.

Tolerances: those of the full-size tests, g_tau 1e-4 relative, delta 6e-5, G 2e-4
(log E 1e-5 more)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2602_01723_gb300 import scenes  # noqa: E402


@pytest.mark.parametrize("n", [1, 33, 127, 129, 1000])
@pytest.mark.parametrize("scatter,chunk,elastic", [(1, 64, 0), (1, 128, 0), (0, 128, 1), (2, 128, 0), (1, 128, 2)])
def test_signals_from_the_substep_kernels(orc, n, scatter, chunk, elastic):
    from __graft_entry__ import build
    build()
    from paper_2602_01723_gb300.sim import Simulator
    rng = np.random.default_rng(200 + n)
    R = 16
    f32 = lambda a: np.ascontiguousarray(a, np.float32)  # noqa: E731
    x, v = f32(0.35 + 0.3 * rng.random((n, 3))), f32(rng.normal(0.0, 0.5, (n, 3)))
    sc = scenes.Scene("small", R, 1e-4, 0, x, v, np.full(n, (0.5 / R) ** 3, np.float32), np.zeros(n, np.int32),
                      [scenes.material(elastic, 0, 1e4, 0.3, 100.0)])
    keys = [(v, f32(2.0 * rng.standard_normal((n, 3, 3))), f32(np.eye(3) + 0.03 * rng.standard_normal((n, 3, 3))))
            for _ in range(2)]
    cfg = orc.Cfg(sc.grid_res, sc.dx, sc.dt, sc.gravity)
    mat = orc.Material.from_table(sc.vol, sc.mat_id, sc.materials)
    ref = orc.bgdo(cfg, [orc.new_state(x, *k) for k in keys], mat, label=sc.mat_id)
    s = Simulator.from_scene(sc, chunk=chunk)
    s.set_tuning(scatter=scatter, chunk=chunk, use_graph=True)
    for k, (vk, C, F) in enumerate(keys):
        s.load(x, sc.vol, sc.mat_id, v=vk, C=C, F=F)
        s.snapshot(k)
    before = {k: a.clone() for k, a in s.get().items()}
    outs = [s.bgdo([0, 1], signals=sig) for sig in (True, False, True)]
    for k, a in s.get().items():
        assert torch.equal(a, before[k]), k
    s.step(1)
    assert s.stats()["device_error"] == 0
    for out in outs:
        got = {k: a.double().cpu().numpy() for k, a in out.items()}
        assert np.abs(got["G"] - ref["G"]).max() < 2e-4
        assert np.abs(got["log_E"] - ref["log_E"]).max() < 2e-4 + 1e-5
        if "g_tau" in got:
            scale = np.abs(ref["g_tau"]).max()
            assert np.all(np.abs(got["g_tau"] - ref["g_tau"]) <= 1e-4 * np.abs(ref["g_tau"]) + 1e-6 * scale)
            assert np.abs(got["delta"] - ref["delta"]).max() < 6e-5
    s.close()
