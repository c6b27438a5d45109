"""Forward runs on both sides of the particle count up to which the kernels of a
substep are dependent launches (65,536): launched directly, replayed from graphs,
captured in the caller's graph, and recorded with a state copy after every third
substep, against the FP64 oracle.

Tolerances: positions 1e-4 dx (the forward tests' bound for 100 substeps), F 2e-5
per substep."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2602_01723_gb300 import scenes  # noqa: E402

N_SUB = 20


@pytest.mark.parametrize("n", [500, 65536, 65537])
def test_both_sides_of_the_line(orc, n):
    from __graft_entry__ import build
    build()
    from paper_2602_01723_gb300.sim import Simulator
    rng = np.random.default_rng(500 + n)
    R = 16 if n < 1000 else 48
    f32 = lambda a: np.ascontiguousarray(a, np.float32)  # noqa: E731
    x, v = f32(0.3 + 0.4 * rng.random((n, 3))), f32(rng.normal(0.0, 0.5, (n, 3)))
    F = f32(np.eye(3) + 0.03 * rng.standard_normal((n, 3, 3)))
    C = f32(rng.standard_normal((n, 3, 3)))
    sc = scenes.Scene("line", R, 1e-4, 0, x, v, np.full(n, (0.5 / R) ** 3, np.float32), np.zeros(n, np.int32),
                      [scenes.material(0, 0, 1e4, 0.3, 100.0)])
    ref = orc.run(orc.Cfg(R, sc.dx, sc.dt, sc.gravity), orc.new_state(x, v, C, F),
                  orc.Material.from_table(sc.vol, sc.mat_id, sc.materials), N_SUB)
    s = Simulator.from_scene(sc, ckpt_every=3)
    a = [torch.as_tensor(t, device="cuda") for t in (x, sc.vol, sc.mat_id, v, C, F)]

    def load():
        s.load(a[0], a[1], a[2], v=a[3], C=a[4], F=a[5])

    def check(what):
        got = s.get()
        assert s.stats()["device_error"] == 0, what
        ex = np.abs(got["x"].double().cpu().numpy() - ref["x"]).max()
        ef = np.abs(got["F"].double().cpu().numpy().reshape(ref["F"].shape) - ref["F"]).max()
        assert ex < 1e-4 * sc.dx and ef < N_SUB * 2e-5, (what, ex, ef)

    for graph in (False, True):
        s.set_tuning(scatter=1, chunk=128, use_graph=graph)
        for record in (False, True):
            load()
            s.step(N_SUB, record=record)
            check((graph, record))
    load()
    s.step(N_SUB)                 # (a run outside the capture allocates what it needs)
    load()
    s.sync()
    st = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        s.step(N_SUB)
    g.replay()
    torch.cuda.synchronize()
    check("captured")
    s.close()


@pytest.mark.parametrize("n", [500, 65536, 65537])
def test_gradients_on_both_sides_of_the_line(n):
    """The reverse pass from the grid tape (dependent launches up to the line)
    against the one that rebuilds each state (ordinary launches), replayed from
    graphs and launched directly: within the adjoint tests' 1e-3 relative."""
    from __graft_entry__ import build
    build()
    from paper_2602_01723_gb300.sim import Simulator
    rng = np.random.default_rng(600 + n)
    R = 16 if n < 1000 else 48
    f32 = lambda a: np.ascontiguousarray(a, np.float32)  # noqa: E731
    x, v = f32(0.3 + 0.4 * rng.random((n, 3))), f32(rng.normal(0.0, 0.5, (n, 3)))
    F = f32(np.eye(3) + 0.03 * rng.standard_normal((n, 3, 3)))
    cot = torch.as_tensor(f32(rng.standard_normal((2, n, 3))))
    sc = scenes.Scene("line", R, 1e-4, 0, x, v, np.full(n, (0.5 / R) ** 3, np.float32), np.zeros(n, np.int32),
                      [scenes.material(0, 0, 1e4, 0.3, 100.0)])
    out = {}
    for tape_grid, graph in ((1, False), (0, False), (0, True)):
        s = Simulator.from_scene(sc, ckpt_every=6, tape_grid=tape_grid)
        s.set_tuning(scatter=1, chunk=128, use_graph=graph)
        s.load(x, sc.vol, sc.mat_id, v=v, F=F)
        s.step(N_SUB, record=True)
        out[tape_grid, graph] = s.backward([9, N_SUB], cot).double().cpu().numpy()
        assert s.stats()["device_error"] == 0
        s.close()
    ref = out[1, False]
    for k, g in out.items():
        for j in range(2):
            assert np.linalg.norm(g[:, j] - ref[:, j]) < 1e-3 * np.linalg.norm(ref[:, j]), (k, j)
