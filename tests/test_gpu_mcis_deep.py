"""Fill candidates deeper than the cut-off, and surface points given several times:
both leave the search by warps for a second kernel.

Beyond the cut-off a candidate's weight is eps, and its distance that to the nearest
surface point in the coarse cells up to six away from its own (infinite where they
hold none): against a direct FP64 search over those cells, 1e-15 relative.  Cells of
the coarse size and halved (from 2,000 surface points an object on), candidates
close together and far apart, points that are not finite beside others, a candidate
that is not finite.

A fill with deep candidates may take six times as long as one without: it took 17
times as long with one lane per deep candidate, and takes about as long now."""
import math
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS, RINGS = 1e-6, 6


@pytest.fixture(scope="module")
def mcis():
    from __graft_entry__ import build
    build()
    from paper_2602_01723_gb300.sim import mcis
    return mcis


def cells(x, G):
    with np.errstate(invalid="ignore"):
        c = np.floor(x.astype(np.float32) * np.float32(G))
    return np.clip(np.where(np.isnan(c), 0, c), 0, G - 1).astype(int)


def direct(S, Q, sigma):
    cut = sigma * math.sqrt(2.0 * math.log(1.0 / EPS))
    G = min(256, max(1, int(math.floor(RINGS / cut))))
    cs, cq = cells(S, G), cells(Q, G)
    out = np.full(len(Q), np.inf)
    for i in range(len(Q)):
        near = (np.abs(cs - cq[i]) <= RINGS).all(1) & np.isfinite(S).all(1)
        if near.any() and np.isfinite(Q[i]).all():
            out[i] = ((Q[i].astype(np.float64) - S[near].astype(np.float64)) ** 2).sum(1).min()
    return np.sqrt(out)


def sphere(rng, n, r):
    d = rng.standard_normal((n, 3))
    return 0.5 + r * d / np.linalg.norm(d, axis=1, keepdims=True)


@pytest.mark.parametrize("n_surf", [40, 1999, 2000, 9000])
@pytest.mark.parametrize("sigma, r", [(0.02, 0.22), (0.01, 0.1), (0.004, 0.3)])
@pytest.mark.parametrize("odd", [False, True])
def test_beyond_the_cut_off(mcis, n_surf, sigma, r, odd):
    rng = np.random.default_rng(n_surf)
    S = sphere(rng, n_surf, r)
    Q = np.concatenate([0.5 + 0.6 * r * rng.uniform(-1, 1, (400, 3)), 0.5 + 0.03 * rng.uniform(-1, 1, (150, 3)),
                        rng.uniform(-0.1, 1.1, (60, 3))])
    S, Q = S.astype(np.float32), Q.astype(np.float32)
    if odd:
        S[::7, 1] = np.nan
        S[3::11, 2] = np.inf
        S[5::13, 0] = -np.inf
        Q[5] = np.nan
        Q[77, 2] = np.inf
    d = direct(S, Q, sigma)
    off = lambda n: np.array([0, n], np.int64)  # noqa: E731
    got = mcis(off(n_surf), S, off(len(Q)), Q, off(8), rng.random(8), sigma, EPS)["d"].cpu().numpy()
    assert (d > sigma * math.sqrt(2.0 * math.log(1.0 / EPS))).any()
    np.testing.assert_array_equal(np.isinf(got), np.isinf(d))
    np.testing.assert_allclose(got[np.isfinite(d)], d[np.isfinite(d)], rtol=1e-15, atol=0)


def test_deep_candidates_take_about_as_long(mcis):
    rng = np.random.default_rng(1)

    def fill_time(r):
        n, nc = 36_000, 250_000
        q = 0.5 + r * rng.uniform(-1, 1, (3 * nc, 3))
        q = q[((q - 0.5) ** 2).sum(1) < r * r][:nc]
        S, Q = (torch.tensor(a.astype(np.float32), device="cuda") for a in (sphere(rng, n, r), q))
        u, off = torch.rand(1000, dtype=torch.float64, device="cuda"), lambda m: np.array([0, m], np.int64)
        took = []
        for _ in range(7):
            torch.cuda.synchronize()
            t = time.perf_counter()
            mcis(off(n), S, off(nc), Q, off(1000), u)
            torch.cuda.synchronize()
            took.append(time.perf_counter() - t)
        return min(took)

    assert fill_time(0.3) < 6.0 * fill_time(0.1)
