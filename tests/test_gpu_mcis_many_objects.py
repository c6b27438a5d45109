"""The fill sampling with so many objects that their occupancy masks together
pass 2^27 words (a cell's number, word and bit, then no longer fits 32 bits
unless it is counted within the object): the first and the last objects hold
points and candidates, the others are empty.  Against a direct search in FP64,
tolerances as in the fill sampling's parity test (distances 1e-15 relative,
weights 1e-14)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIGMA, EPS = 0.25, 1e-6   # cut-off 1.31: four cells per axis, 32 mask words an object


@pytest.mark.parametrize("n_obj", [4_194_300, 4_194_309])   # 2^27 words are 4,194,304 objects
def test_masks_beyond_2_27_words(n_obj):
    from __graft_entry__ import build
    build()
    from paper_2602_01723_gb300.sim import mcis
    rng = np.random.default_rng(n_obj)
    held = [0, 1, n_obj - 2, n_obj - 1]
    ns, nc = [7, 300, 5, 400], [40, 33, 60, 50]

    def offsets(counts):
        c = np.zeros(n_obj, np.int64)
        c[held] = counts
        return np.concatenate([[0], np.cumsum(c)])

    so, co, do = offsets(ns), offsets(nc), offsets([3, 4, 5, 6])
    S, Q = rng.random((sum(ns), 3)).astype(np.float32), rng.random((sum(nc), 3)).astype(np.float32)
    u = rng.random(18)
    got = {k: v.cpu().numpy() for k, v in mcis(so, S, co, Q, do, u, SIGMA, EPS).items()}
    for k in held:
        s, q = S[so[k]:so[k + 1]].astype(np.float64), Q[co[k]:co[k + 1]].astype(np.float64)
        d2 = ((q[:, None] - s[None]) ** 2).sum(2).min(1)
        np.testing.assert_allclose(got["d"][co[k]:co[k + 1]], np.sqrt(d2), rtol=1e-15, atol=0)
        w = np.maximum(np.exp(-d2 / (2 * SIGMA ** 2)), EPS)
        np.testing.assert_allclose(got["w"][co[k]:co[k + 1]], w, rtol=1e-14, atol=0)
        picked = got["picked"][do[k]:do[k + 1]]
        assert ((picked >= co[k]) & (picked < co[k + 1])).all()
