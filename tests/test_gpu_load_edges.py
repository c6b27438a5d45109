"""Loading and export through shared memory: particle counts around the edges of
warps and CTAs, device arrays that start on a 4-byte but no 16-byte boundary, host
arrays, subsets of the outputs, and a state out of the domain or with a value that
is not finite, which is still reported.

The records keep v, C and F in float32 as they were given, so these come back bit
for bit.  Positions are kept in fixed point, 23 fraction bits of a cell on this
grid, and come back within one unit and a float32 rounding: dx 2^-23 + 2^-24."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2602_01723_gb300 import scenes  # noqa: E402

R, DX = 16, 1.0 / 16


@pytest.fixture(scope="module")
def sim_mod():
    from __graft_entry__ import build
    build()
    from paper_2602_01723_gb300 import sim
    return sim


def arrays(n):
    rng = np.random.default_rng(300 + n)
    f32 = lambda a: np.ascontiguousarray(a, np.float32)  # noqa: E731
    return dict(x=f32(0.3 + 0.4 * rng.random((n, 3))), v=f32(rng.normal(0.0, 0.5, (n, 3))),
                C=f32(rng.standard_normal((n, 3, 3))), F=f32(np.eye(3) + 0.03 * rng.standard_normal((n, 3, 3))))


def simulator(sim_mod, n, a):
    sc = scenes.Scene("small", R, 1e-4, 0, a["x"], a["v"], np.full(n, (0.5 / R) ** 3, np.float32),
                      np.zeros(n, np.int32), [scenes.material(0, 0, 1e4, 0.3, 100.0)])
    return sc, sim_mod.Simulator.from_scene(sc)


def shifted(a):
    """the array on the device, one float behind a 256-byte boundary"""
    t = torch.empty(a.size + 1, dtype=torch.float32, device="cuda")
    t[1:] = torch.as_tensor(a.reshape(-1), device="cuda")
    return t[1:].view(a.shape)


@pytest.mark.parametrize("n", [1, 31, 127, 128, 129, 257, 1000])
@pytest.mark.parametrize("where", ["host", "device", "shifted"])
def test_load_and_get_round_trip(sim_mod, n, where):
    a = arrays(n)
    sc, s = simulator(sim_mod, n, a)
    put = {"host": lambda t: t, "device": lambda t: torch.as_tensor(t, device="cuda"), "shifted": shifted}[where]
    s.load(put(a["x"]), put(sc.vol), sc.mat_id if where == "host" else torch.as_tensor(sc.mat_id, device="cuda"),
           v=put(a["v"]), C=put(a["C"]), F=put(a["F"]))
    got = {k: t.cpu().numpy() for k, t in s.get().items()}
    for k in "vCF":
        assert np.array_equal(got[k].reshape(a[k].shape), a[k]), k
    assert np.abs(got["x"].astype(np.float64) - a["x"]).max() <= DX * 2.0 ** -23 + 2.0 ** -24
    assert np.array_equal(s.positions().cpu().numpy(), got["x"])
    s.step(3)                                              # (the load's binning is usable)
    assert s.stats()["device_error"] == 0
    s.close()


@pytest.mark.parametrize("n", [1, 129])
@pytest.mark.parametrize("bad", ["domain", "nan", "inf"])
def test_bad_states_are_still_reported(sim_mod, n, bad):
    a = arrays(n)
    sc, s = simulator(sim_mod, n, a)
    if bad == "domain":
        a["x"][n - 1, 1] = 1.5
    else:
        a["F"][n - 1, 2, 1] = {"nan": np.nan, "inf": np.inf}[bad]
    with pytest.raises(Exception):
        s.load(a["x"], sc.vol, sc.mat_id, v=a["v"], C=a["C"], F=a["F"])
        s.sync()
    s.close()
