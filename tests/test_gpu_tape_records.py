"""The recompute of the reverse pass writes each state's records straight into
the tape and takes its scatter packets in (rank, bank) order every 8th substep
of a segment, in list order between.  Gradients with segments of one substep,
of just that period and around it, at particle counts around the edges of warps
and chunks, for both CTA sizes and for the common and the further material
models, against the FP64 oracle's reverse pass.

Tolerance: that of the adjoint tests, 1e-3 relative per parameter kind.  (One
particle alone does not move by its own stress, so the counts start at 33.)"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2602_01723_gb300 import scenes  # noqa: E402


def small_scene(n, elastic):
    rng = np.random.default_rng(100 + n)
    R = 16
    x = 0.35 + 0.3 * rng.random((n, 3))
    v = rng.normal(0.0, 0.5, (n, 3))
    F = np.eye(3) + 0.03 * rng.standard_normal((n, 3, 3))
    C = 2.0 * rng.standard_normal((n, 3, 3))
    f32 = lambda a: np.ascontiguousarray(a, np.float32)  # noqa: E731
    sc = scenes.Scene("small", R, 1e-4, 0, f32(x), f32(v), np.full(n, (0.5 / R) ** 3, np.float32),
                      np.zeros(n, np.int32), [scenes.material(elastic, 0, 1e4, 0.3, 100.0)])
    cot = rng.standard_normal((2, n, 3)).astype(np.float32)
    return sc, f32(C), f32(F), cot


@pytest.mark.parametrize("n", [33, 127, 129, 1000])
@pytest.mark.parametrize("chunk,elastic", [(64, 0), (128, 0), (128, 2)])
def test_gradients_around_an_ordered_substep(orc, n, chunk, elastic):
    from __graft_entry__ import build
    build()
    from paper_2602_01723_gb300.sim import Simulator
    sc, C, F, cot = small_scene(n, elastic)
    n_sub, frames = 21, [12, 21]
    cfg = orc.Cfg(sc.grid_res, sc.dx, sc.dt, sc.gravity)
    mat = orc.Material.from_table(sc.vol, sc.mat_id, sc.materials)
    _, tape = orc.run(cfg, orc.new_state(sc.x, sc.v, C, F), mat, n_sub, tape=True)
    _, ref = orc.backward(cfg, mat, tape, frames, cot.astype(np.float64))
    for every in (1, 8, 9, 17):
        s = Simulator.from_scene(sc, chunk=chunk, ckpt_every=every)
        s.load(sc.x, sc.vol, sc.mat_id, v=sc.v, C=C, F=F)
        s.step(n_sub, record=True)
        g = s.backward(frames, torch.as_tensor(cot)).double().cpu().numpy()
        s.close()
        for j in range(2):   # log E, nu
            err = np.linalg.norm(g[:, j] - ref[:, j]) / np.linalg.norm(ref[:, j])
            assert err < 1e-3, (every, j, err)
