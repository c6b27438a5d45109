"""The fill on both sides of the line from which the cells of the surface points are
halved (24,000 points an object), near and beyond the cut-off, against a direct FP64
search: distances below the cut-off 1e-15 relative, weights 1e-14, and the same
infinite or finite distances beyond (the nearest point of the coarse cells up to six
away)."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS, RINGS = 1e-6, 6


@pytest.mark.parametrize("n_surf", [23_999, 24_000])
@pytest.mark.parametrize("sigma, r", [(0.02, 0.09), (0.02, 0.2), (0.05, 0.3), (0.004, 0.05)])
def test_either_side_of_the_line(n_surf, sigma, r):
    from __graft_entry__ import build
    build()
    from paper_2602_01723_gb300.sim import mcis
    rng = np.random.default_rng(n_surf)
    d = rng.standard_normal((n_surf, 3))
    S = (0.5 + r * d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32)
    S[1::9] = S[::9][: len(S[1::9])]                          # repeated points
    S[2::9] = S[::9][: len(S[2::9])]
    Q = (0.5 + 1.1 * r * rng.uniform(-1, 1, (500, 3))).astype(np.float32)
    cut = sigma * math.sqrt(2.0 * math.log(1.0 / EPS))
    G = min(256, max(1, int(math.floor(RINGS / cut))))
    cell = lambda x: np.clip(np.floor(x * np.float32(G)), 0, G - 1).astype(int)  # noqa: E731
    cs, cq = cell(S), cell(Q)
    want = np.full(len(Q), np.inf)
    for i in range(len(Q)):
        near = (np.abs(cs - cq[i]) <= RINGS).all(1)
        if near.any():
            want[i] = math.sqrt(((Q[i].astype(np.float64) - S[near].astype(np.float64)) ** 2).sum(1).min())
    off = lambda n: np.array([0, n], np.int64)  # noqa: E731
    got = {k: v.cpu().numpy() for k, v in mcis(off(n_surf), S, off(len(Q)), Q, off(8), rng.random(8), sigma, EPS).items()}
    np.testing.assert_array_equal(np.isinf(got["d"]), np.isinf(want))
    fin = np.isfinite(want)
    np.testing.assert_allclose(got["d"][fin], want[fin], rtol=1e-15, atol=0)
    w = np.maximum(np.exp(-np.minimum(want, 1e3) ** 2 / (2.0 * sigma ** 2)), EPS)
    np.testing.assert_allclose(got["w"], w, rtol=1e-14, atol=0)
