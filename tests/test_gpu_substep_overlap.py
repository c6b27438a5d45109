"""mpm_substep_noalloc, whose kernels start before the one ahead has ended: particle
counts around the edges of its CTAs, outputs in the inputs' place, ten calls in a
row against ten oracle substeps, and a bad particle that is reported by its call and
not by the next.

Tolerances, those of the entry point's other tests for one substep (positions 1e-4
dx, v and C 1e-5 relative, F 2e-5), times the number of substeps."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2602_01723_gb300 import scenes  # noqa: E402

R, DX, DT, G = 16, 1.0 / 16, 1e-4, (0.0, 0.0, -9.8)


def call(L, table, arrays, out):
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    return L.lib().mpm_substep_noalloc(
        (ctypes.c_int32 * 3)(R, R, R), DX, DT, (ctypes.c_float * 3)(*G), table, len(table), None, len(arrays["vol"]),
        *[p(arrays[k]) for k in ("x", "v", "C", "F", "vol", "mat")], *[p(out[k]) for k in "xvCF"],
        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))


@pytest.mark.parametrize("n", [1, 31, 63, 64, 65, 129, 3000])
@pytest.mark.parametrize("in_place", [False, True])
def test_ten_calls_in_a_row(orc, n, in_place):
    from __graft_entry__ import build
    build()
    from paper_2602_01723_gb300 import _lib as L
    rng = np.random.default_rng(400 + n)
    f32 = lambda a: np.ascontiguousarray(a, np.float32)  # noqa: E731
    x, v = f32(0.35 + 0.3 * rng.random((n, 3))), f32(rng.normal(0.0, 0.5, (n, 3)))
    C, F = f32(2.0 * rng.standard_normal((n, 3, 3))), f32(np.eye(3) + 0.03 * rng.standard_normal((n, 3, 3)))
    vol, mat = np.full(n, (0.5 / R) ** 3, np.float32), (np.arange(n) % 3).astype(np.int32)
    mats = [scenes.material(0, 0, 1e4, 0.3, 100.0), scenes.material(1, 0, 1e4, 0.3, 100.0),
            scenes.material(0, 1, 1e4, 0.3, 100.0, yield_stress=3e2)]
    table = (L.mpm_material * len(mats))(*[L.mpm_material(m["elastic"], m["plastic"], m["E"], m["nu"], m["rho"],
                                                         m["yield_stress"], m["friction_angle_deg"]) for m in mats])
    dev = lambda a: torch.as_tensor(a, device="cuda").contiguous().clone()  # noqa: E731
    a = dict(x=dev(x), v=dev(v), C=dev(C), F=dev(F), vol=dev(vol), mat=dev(mat))
    b = a if in_place else dict(a, **{k: torch.empty_like(a[k]) for k in "xvCF"})
    bad = dict(a, x=a["x"].clone())
    bad["x"][n - 1, 1] = 1.5
    other = {k: torch.empty_like(a[k]) for k in "xvCF"}
    for step in range(10):
        if step == 4:
            assert call(L, table, bad, other) != 0
        assert call(L, table, a, b) == 0
        a, b = b, a
    ref = orc.run(orc.Cfg(R, DX, DT, G), orc.new_state(x, v, C, F), orc.Material.from_table(vol, mat, mats), 10)
    err = {k: np.abs(a[k].double().cpu().numpy().reshape(ref[k].shape) - ref[k]).max() for k in "xvCF"}
    assert err["x"] < 10 * 1e-4 * DX, err
    assert err["v"] < 10 * 1e-5 * np.abs(ref["v"]).max(), err
    assert err["C"] < 10 * 1e-5 * np.abs(ref["C"]).max(), err
    assert err["F"] < 10 * 2e-5, err
