"""The nearest-surface search of the fill sampling where its cells, groups and
cut-off meet their edges: few and many candidates (one to eight of them a
warp), coarse and halved cells, cut-offs from a cell of the finest grid to many
times the cube, repeated and equidistant surface points (settled in FP64),
coordinates outside the cube, objects of one point and of none.

Tolerances as in the fill sampling's parity test: distances below the cut-off
1e-15 relative, weights 1e-14, draws the inverse CDF of the weights."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS = 1e-6


def shells(rng, n, kind):
    """Surface points of one object, (n, 3)."""
    d = rng.standard_normal((n, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    p = 0.5 + 0.09 * d
    if kind == "repeated":      # every point four times
        p = np.repeat(p[: max(1, n // 4)], 4, axis=0)
    elif kind == "outside":     # a plane across the cube's face
        p = np.stack([1.0 + 0.02 * rng.standard_normal(n), rng.random(n), rng.random(n)], 1)
    elif kind == "grid":        # a lattice: many equal distances
        p = 0.4 + 0.2 * rng.integers(0, 9, (n, 3)) / 8.0
    return p.astype(np.float32)


@pytest.mark.parametrize("kind", ["sphere", "repeated", "outside", "grid"])
@pytest.mark.parametrize("n_surf, n_cand", [(1, 5), (60, 33), (2500, 700), (2500, 31000)])
@pytest.mark.parametrize("sigma", [0.02, 0.0015, 0.4, 3.0])
def test_search_matches_the_oracle(orc, kind, n_surf, n_cand, sigma):
    from __graft_entry__ import build
    build()
    from paper_2602_01723_gb300.sim import mcis
    rng = np.random.default_rng(n_surf + n_cand)
    surf = [shells(rng, n_surf, kind), shells(rng, max(1, n_surf // 2), "sphere"), np.zeros((0, 3), np.float32)]
    cand = [(0.5 + 0.11 * rng.uniform(-1, 1, (n_cand, 3))), rng.uniform(-0.05, 1.05, (max(1, n_cand // 10), 3)),
            rng.random((4, 3))]
    cand[0][0] = surf[0][0]     # on a surface point
    cand[0][-1] = 0.5           # the centre
    cand = [c.astype(np.float32) for c in cand]
    off = lambda parts: np.concatenate([[0], np.cumsum([len(a) for a in parts])]).astype(np.int64)  # noqa: E731
    so, co, do = off(surf), off(cand), np.array([0, 50, 80, 90], np.int64)
    S, Q, u = np.concatenate(surf), np.concatenate(cand), rng.random(90)
    ref = orc.mcis(so, S, co, Q, do, u, sigma, EPS)
    got = {k: v.cpu().numpy() for k, v in mcis(so, S, co, Q, do, u, sigma, EPS).items()}
    near = ref["d"] < sigma * math.sqrt(2 * math.log(1 / EPS))
    np.testing.assert_allclose(got["d"][near], ref["d"][near], rtol=1e-15, atol=0)
    assert np.all(got["d"][~near] >= ref["d"][~near] * (1 - 1e-15))
    np.testing.assert_allclose(got["w"], ref["w"], rtol=1e-14, atol=0)
    for k in range(3):
        cum = np.cumsum(np.floor(got["w"][co[k]:co[k + 1]] * 2.0 ** 40 + 0.5).astype(np.int64))
        t = np.floor(u[do[k]:do[k + 1]] * float(cum[-1])).astype(np.int64)
        np.testing.assert_array_equal(got["picked"][do[k]:do[k + 1]],
                                      co[k] + np.minimum(np.searchsorted(cum, t, side="right"), len(cum) - 1))
