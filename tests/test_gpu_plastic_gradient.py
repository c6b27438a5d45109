"""Gradients through one return map, for tables with plasticity, at particle counts
around the edges of warps and chunks: two substeps, a loss on the positions after
the second, which the first return map alone reaches.  Tables with von Mises and
Drucker-Prager beside elastic particles, and with the volume-based plasticities as
well (the two instances of the reverse G2P with a second pass over the nodes).

No particle's trial state is near a kink of its return map: at the yield surface
the gradient jumps, and rounding decides the side (two runs of the same inputs
then differ there).  The distance is checked in FP64, on the trial states of the
oracle without plasticity.

Tolerance 1e-4 relative per parameter kind: some 200 FP32 roundings in a chain are
1.2e-5, the SVD's adjoint enlarges them by the spread of the singular values over
their gaps, about ten in the mean of these states."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2602_01723_gb300 import scenes  # noqa: E402

R, E, NU, YIELD, PHI = 16, 1e4, 0.3, 60.0, 30.0
TABLES = {"common": [(0, 0), (0, 1), (0, 2), (1, 0)], "all": [(0, 1), (0, 2), (4, 3), (3, 0), (0, 4)]}


def distance_to_kink(F, plastic):
    """|delta gamma| of the trial state, and |tr eps| for Drucker-Prager; infinite where there is no return map;
    for the clamp of J the distance from its bounds."""
    s = np.linalg.svd(F, compute_uv=False)
    s[:, 2] *= np.sign(np.linalg.det(F))
    if plastic in (0, 3):
        return np.full(len(F), np.inf)
    if plastic == 4:
        J = np.linalg.det(F)
        return np.minimum(np.abs(J - 0.05), np.abs(J - 1.2))
    eps = np.log(np.maximum(s, 1e-4))
    tr = eps.sum(1)
    h = np.linalg.norm(eps - tr[:, None] / 3.0, axis=1)
    mu, lam = E / (2 * (1 + NU)), E * NU / ((1 + NU) * (1 - 2 * NU))
    if plastic == 1:
        return np.abs(h - YIELD / (2 * mu))
    a = np.sqrt(2.0 / 3.0) * 2.0 * np.sin(np.radians(PHI)) / (3.0 - np.sin(np.radians(PHI)))
    dg = h + (3 * lam + 2 * mu) / (2 * mu) * tr * a
    return np.where(tr > 0, tr, np.minimum(np.abs(dg), np.abs(tr)))


@pytest.mark.parametrize("n", [33, 129, 1000])
@pytest.mark.parametrize("table", list(TABLES))
@pytest.mark.parametrize("chunk", [64, 128])
def test_gradient_through_one_return_map(orc, n, table, chunk):
    from __graft_entry__ import build
    build()
    from paper_2602_01723_gb300.sim import Simulator
    rng = np.random.default_rng(700 + n)
    f32 = lambda a: np.ascontiguousarray(a, np.float32)  # noqa: E731
    models = TABLES[table]
    ids = rng.integers(0, len(models), n).astype(np.int32)
    mats = lambda plastic: [scenes.material(e, p if plastic else 0, E, NU, 100.0, yield_stress=YIELD,  # noqa: E731
                                            friction_angle_deg=PHI) for e, p in models]
    x, v = f32(0.35 + 0.3 * rng.random((n, 3))), f32(rng.normal(0.0, 0.5, (n, 3)))
    C, F = f32(2.0 * rng.standard_normal((n, 3, 3))), f32(np.eye(3) + 0.08 * rng.standard_normal((n, 3, 3)))
    vol = np.full(n, (0.5 / R) ** 3, np.float32)
    cot = rng.standard_normal((1, n, 3)).astype(np.float32)
    sc = scenes.Scene("small", R, 1e-4, 0, x, v, vol, ids, mats(True))
    cfg = orc.Cfg(sc.grid_res, sc.dx, sc.dt, sc.gravity)
    # states close to a kink are replaced by a rotation-free stretch far from it
    far = np.diag([1.06, 0.9, 0.95]).astype(np.float32)
    for _ in range(2):
        trial = orc.run(cfg, orc.new_state(x, v, C, F), orc.Material.from_table(vol, ids, mats(False)), 1)["F"].reshape(n, 3, 3)
        d = np.array([distance_to_kink(trial[i:i + 1], models[ids[i]][1])[0] for i in range(n)])
        F[d < 2e-3] = far
    assert d.min() > 1e-3
    mat = orc.Material.from_table(vol, ids, sc.materials)
    _, tape = orc.run(cfg, orc.new_state(x, v, C, F), mat, 2, tape=True)
    _, ref = orc.backward(cfg, mat, tape, [2], cot.astype(np.float64))
    s = Simulator.from_scene(sc, chunk=chunk)
    s.load(x, vol, ids, v=v, C=C, F=F)
    s.step(2, record=True)
    g = s.backward([2], torch.as_tensor(cot)).double().cpu().numpy()
    s.close()
    for j in range(3):   # log E, nu, yield stress
        norm = np.linalg.norm(ref[:, j])
        assert norm > 0
        err = np.linalg.norm(g[:, j] - ref[:, j]) / norm
        assert err < 1e-4, (j, err)
