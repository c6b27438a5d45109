"""What the load says of a bad value, by the array it is in: a position, velocity,
affine velocity, deformation gradient, volume or parameter that is not finite is
non-finite, a position off the grid or a material or instance that does not exist
out of the domain.  The bad particle is the only one, the last of a full block of
the load, or in its last partial one; a valid load afterwards is accepted."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2602_01723_gb300 import scenes  # noqa: E402

R = 16
DOMAIN, NONFINITE = "MPM_ERR_OUT_OF_DOMAIN", "MPM_ERR_NONFINITE"
BAD = [("x", (2,), np.nan), ("x", (0,), np.inf), ("v", (1,), np.nan), ("v", (2,), -np.inf), ("C", (0, 0), np.nan),
       ("C", (2, 2), np.inf), ("F", (0, 0), np.nan), ("F", (1, 2), np.inf), ("F", (2, 2), np.nan), ("vol", (), np.nan),
       ("params", (0,), np.nan), ("params", (0,), 200.0), ("params", (1,), np.inf), ("params", (2,), np.nan),
       ("x", (0,), -0.2), ("x", (1,), 1.5), ("x", (2,), 3e38), ("mat", (), 1), ("mat", (), -1)]


@pytest.mark.parametrize("n", [1, 128, 300])
@pytest.mark.parametrize("name, at, value", BAD)
def test_status_of_a_bad_value(n, name, at, value):
    from __graft_entry__ import build
    build()
    from paper_2602_01723_gb300 import _lib
    from paper_2602_01723_gb300.sim import Simulator
    rng = np.random.default_rng(n)
    f32 = lambda a: np.ascontiguousarray(a, np.float32)  # noqa: E731
    good = dict(x=f32(0.3 + 0.4 * rng.random((n, 3))), v=f32(rng.normal(0.0, 0.5, (n, 3))),
                C=f32(rng.standard_normal((n, 3, 3))), F=f32(np.eye(3) + 0.03 * rng.standard_normal((n, 3, 3))),
                vol=np.full(n, (0.5 / R) ** 3, np.float32), params=f32(np.tile([9.0, 0.3, 0.0], (n, 1))),
                mat=np.zeros(n, np.int32))

    def load(a):
        s.load(a["x"], a["vol"], a["mat"], v=a["v"], C=a["C"], F=a["F"], params=a["params"])
        s.sync()

    s = Simulator(R, 1.0 / R, 1e-4, (0.0, -9.8, 0.0), [scenes.material(0, 0, 1e4, 0.3, 100.0)])
    bad = {k: a.copy() for k, a in good.items()}
    bad[name][(n - 1,) + at] = value
    with pytest.raises(_lib.MpmError) as e:
        load(bad)
    # (what has no place on the grid may be out of the domain as well)
    want = (DOMAIN,) if np.isfinite(value) and name != "params" else (NONFINITE,) if name != "x" else (NONFINITE, DOMAIN)
    assert str(e.value).startswith(want), str(e.value)
    load(good)
    s.step(2)
    s.sync()
    s.close()
