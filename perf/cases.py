"""The calls whose speed is watched: what a program that uses this framework has it do, over the range of
sizes and options it is used at.

A case is a dict of plain values.  ``prepare`` draws its inputs from the seed and makes the handle a program
keeps (a ``Simulator`` with its options); ``run`` is one pass through the public entry points; ``work`` states
the bytes and operations the pass cannot do without; ``exact`` is the same pass in 64 bits, in plain torch.

Kinds:
  substep  one substep through the allocation-free C entry point (latency-critical callers)
  frame    load a state, advance it, read the state back (a simulated frame, or one candidate of a sweep)
  grad     a trajectory loss and its gradient with respect to per-particle material parameters
  bgdo     stage 2 of the material optimisation, from stored key frames
  splat    a rendered frame: positions, deformed covariances, splatting into an image
  mcis     interior fill sampling

The particle states are those of the middle of a run: objects that move, spin and touch the floor, with a
smooth strain and a little particle-to-particle noise in F.
"""
import ctypes
import math
import types

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2602_01723_gb300 import _lib, scenes
from paper_2602_01723_gb300.sim import Simulator, mcis, render, trajectory

GRAVITY = (0.0, -9.8, 0.0)
BOUND = 3
# faces x-, x+, y-, y+, z-, z+: sticky floor, the others slip (the library's defaults)
WALLS = (1, 1, 2, 1, 1, 1)
RHO = 100.0


def listed():
    return [
        # the smallest call: one substep of the 8,192-particle cube's size, where launches and the wait count
        dict(name="substep_8k", kind="substep", n=8192, res=32, ry=32, mix="basic"),
        # a small elastic body, 100 substeps: the plain forward workload at its smallest
        dict(name="cube_8k", kind="frame", n=8192, objects=1, instances=1, res=32, ry=32, steps=100, mix="elastic"),
        # the paper-like scene (elastic, plasticine and sand): the main forward workload
        dict(name="objects_300k", kind="frame", n=300_000, objects=3, instances=1, res=128, ry=128, steps=100,
             mix="basic"),
        # the further constitutive models (StVK, Hencky, fluid, volume), an odd count, a grid that is not a cube
        dict(name="models_77k", kind="frame", n=77_777, objects=3, instances=1, res=104, ry=60, steps=60, mix="more"),
        # the largest scene: a block-sparse 256^3 grid
        dict(name="objects_2m", kind="frame", n=2_000_000, objects=8, instances=1, res=256, ry=256, steps=30,
             mix="basic"),
        # a batched parameter sweep: 64 uneven objects, each on its own grid
        dict(name="sweep_64", kind="frame", n=1_350_000, objects=1, instances=64, res=64, ry=64, steps=40,
             mix="sweep"),
        # the gradient at the size of a finite-difference check
        dict(name="grad_512", kind="grad", n=512, objects=1, instances=1, res=16, ry=16, steps=40, every=20,
             frames=10, mix="elastic"),
        # the differentiable ball: per-particle log E and nu from an observed trajectory
        dict(name="grad_50k", kind="grad", n=50_000, objects=1, instances=1, res=64, ry=64, steps=100, every=20,
             frames=10, mix="elastic"),
        # the gradient of a batched sweep, with every common model and a sum per candidate
        dict(name="grad_sweep_64", kind="grad", n=1_350_000, objects=1, instances=64, res=64, ry=64, steps=40,
             every=20, frames=5, mix="sweep"),
        # the material optimisation's second stage on the paper-like scene
        dict(name="bgdo_300k", kind="bgdo", n=300_000, objects=3, instances=1, res=128, ry=128, keys=3, mix="basic"),
        # an image of the paper-like scene
        dict(name="splat_300k", kind="splat", n=300_000, objects=3, instances=1, res=128, ry=128, width=1024,
             height=768, mix="basic"),
        # the fill sampling of its three objects
        dict(name="mcis_750k", kind="mcis", surface=36_000, candidates=250_000, draws=64_000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# object layouts: (centres in x and z, largest horizontal extent)
_LAYOUT = {1: ([(0.5, 0.5)], 0.6), 3: ([(0.2, 0.5), (0.5, 0.5), (0.8, 0.5)], 0.3),
           8: ([(0.2 + 0.2 * (b % 4), 0.3 + 0.4 * (b // 4)) for b in range(8)], 0.21)}


def _least_res(n_object, objects):
    """The coarsest grid on which objects of n_object particles fit their layout (a torus is the widest:
    0.83 n^(1/3) cells across, and twice that of small counts for the shell)."""
    return (0.83 * n_object ** (1.0 / 3.0) + 3.0) / _LAYOUT[objects][1]


def _grid_for(rng, n, objects, instances, most):
    per = n / (objects * instances)
    if instances > 1:
        per *= 2.0
    least = max(16.0, _least_res(per, objects))
    res = min(most, 4 * math.ceil(least * rng.uniform(1.0, 1.5) / 4))
    ry = 4 * math.ceil(max(16.0, res * rng.choice((0.6, 0.75, 1.0))) / 4)
    return res, min(res, ry) if res >= 32 else res


def draw(rng):
    kind = rng.choice(("substep", "frame", "frame", "frame", "grad", "grad", "bgdo", "splat", "mcis"))
    if kind == "mcis":
        return dict(kind=kind, surface=_log_int(rng, 500, 36_000), candidates=_log_int(rng, 1_000, 250_000),
                    draws=_log_int(rng, 100, 64_000))
    if kind == "substep":
        # at most 64^3 nodes
        n = _log_int(rng, 300, 60_000)
        res, ry = _grid_for(rng, n, 1, 1, 64)
        return dict(kind=kind, n=n, res=res, ry=ry, mix=rng.choice(("basic", "elastic")))
    objects, instances = rng.choice(((1, 1), (3, 1), (8, 1), (1, 0)))
    if kind in ("bgdo", "splat") and instances == 0:
        instances = 1
    if instances == 0:
        instances = rng.randint(2, 64)
        n, most = instances * _log_int(rng, 300, 20_000), 64
    elif objects == 8:
        n, most = _log_int(rng, 8_000, 1_900_000 if kind == "frame" else 300_000), 256
    elif objects == 3:
        n, most = _log_int(rng, 1_500, 290_000), 192
    else:
        n, most = _log_int(rng, 500, 200_000), 128
    res, ry = _grid_for(rng, n, objects, instances, most)
    mix = "sweep" if instances > 1 else rng.choice(("basic", "elastic", "sweep"))
    case = dict(kind=kind, n=n, objects=objects, instances=instances, res=res, ry=ry, mix=mix)
    if kind == "frame":
        if instances == 1 and rng.random() < 0.25:
            case["mix"] = "more"
        case["steps"] = min(rng.randint(1, 100), max(1, 50_000_000 // n))
    elif kind == "grad":
        case["steps"] = min(rng.randint(2, 80), max(2, 50_000_000 // n))
        case["every"] = rng.randint(4, 25)
        case["frames"] = rng.randint(1, min(10, case["steps"]))
    elif kind == "bgdo":
        case["keys"] = rng.randint(1, 4)
    else:
        case["height"] = rng.randint(120, 768)
        case["width"] = rng.randint(160, 1024)
    return case


# ---------------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------------

def _materials(mix, count, rng):
    """One table entry per object or instance."""
    out, first = [], int(rng.integers(0, 3))
    for b in range(count):
        E, nu = float(np.exp(rng.uniform(np.log(1e3), np.log(1e5)))), float(rng.uniform(0.2, 0.4))
        ys = float(np.exp(rng.uniform(np.log(3e2), np.log(3e3))))
        if mix == "elastic":
            el, pl, E, nu = 0, 0, 5e3, 0.3
        elif mix == "basic":        # elastic, plasticine, sand
            el, pl = 0, (first + b) % 3
        elif mix == "sweep":        # and Neo-Hookean
            el, pl = ((0, 0), (1, 0), (0, 1), (0, 2))[int(rng.integers(0, 4))]
        else:                       # Hencky sand, fluid, StVK, volume, Hencky
            el, pl = ((3, 2), (4, 3), (2, 0), (5, 4), (3, 0))[b % 5]
        out.append(scenes.material(el, pl, E, nu, RHO, yield_stress=ys, friction_angle_deg=30.0))
    return out


def _shape(b, n, dx, centre, floor):
    """Sphere, torus or box whose half-cell lattice holds about 65% of n particles, its bottom on `floor`."""
    vol = 0.65 * n * (dx / 2) ** 3
    c = (centre[0], 0.0, centre[1])
    if b % 3 == 0:
        s = scenes.Sphere(c, (vol * 3 / (4 * math.pi)) ** (1 / 3))
    elif b % 3 == 1:
        r = (vol / (2 * math.pi ** 2 * 2.5)) ** (1 / 3)
        s = scenes.Torus(c, 2.5 * r, r)
    else:
        s = scenes.Box(c, 0.5 * vol ** (1 / 3))
    s.c = s.c + np.array([0.0, floor - s.bbox()[0][1], 0.0])
    return s


def _state(case, seed):
    """Numpy inputs of one scene: float32 arrays as the library takes them."""
    rng = np.random.Generator(np.random.PCG64([seed, case["n"], case["res"]]))
    B, K, n, dx = case.get("instances", 1), case.get("objects", 1), case["n"], 1.0 / case["res"]
    parts = B * K
    share = rng.uniform(0.1, 1.9, parts) if B > 1 else np.full(parts, 1.0)
    counts = np.maximum(1, np.floor(n * share / share.sum()).astype(int))
    counts[int(np.argmax(counts))] += n - counts.sum()
    xs, vs, Cs, Fs, objs = [], [], [], [], []
    for b in range(parts):
        centre = _LAYOUT[K][0][b % K]
        s = _shape(b, counts[b], dx, centre, 3.3 * dx)
        p, _ = scenes.shell_plus_interior([s], int(counts[b]), dx, rng)
        m = len(p)
        w = rng.normal(0.0, 2.0, 3)
        spin = np.array([[0, -w[2], w[1]], [w[2], 0, -w[0]], [-w[1], w[0], 0]])
        d = p - s.c
        # a smooth strain of a few per cent over the object, and noise of half a per cent
        k = rng.uniform(-1.0, 1.0, (3, 9)) * (2 * math.pi / np.ptp(p, axis=0).max())
        F = np.eye(3).reshape(1, 9) + 0.04 * np.sin(d @ k + rng.uniform(0, 2 * math.pi, 9))
        F += 0.005 * rng.standard_normal((m, 9), dtype=np.float32)
        xs.append(p)
        vs.append(np.array([0.0, -1.0, 0.0]) + d @ spin.T + 0.05 * np.sin(d @ k[:, :3]))
        Cs.append(spin.reshape(1, 9) + 0.5 * np.sin(d @ k))
        Fs.append(F)
        objs.append(np.full(m, b, np.int32))
    x, obj = np.concatenate(xs), np.concatenate(objs)
    f32 = lambda a: np.ascontiguousarray(a, dtype=np.float32)  # noqa: E731
    S = dict(x=f32(x), v=f32(np.concatenate(vs)), C=f32(np.concatenate(Cs)), F=f32(np.concatenate(Fs)),
             vol=np.full(n, (0.5 * dx) ** 3, np.float32), mat_id=obj,
             instance=obj if B > 1 else None, materials=_materials(case["mix"], parts, rng),
             grid=(case["res"], case["ry"], case["res"]), dx=dx)
    # well inside the stability limit of the stiffest material of the range
    S["dt"] = min(1e-4, 5e-5 * 128 / case["res"])
    S["params"] = None
    if case["mix"] == "elastic" and case["kind"] != "substep":    # that entry point takes the table's
        S["params"] = f32(np.stack([rng.normal(math.log(5e3), 0.5, n).clip(6.5, 10.5), rng.uniform(0.2, 0.4, n),
                                    np.zeros(n)], 1))
    if case["kind"] == "grad":
        if S["params"] is None:
            t = S["materials"]
            S["params"] = f32(np.stack([[math.log(m["E"]) for m in t], [m["nu"] for m in t],
                                        [m["yield_stress"] for m in t]], 1)[obj])
        last = case["steps"]
        S["frame_sub"] = [int(round(last * (f + 1) / case["frames"])) for f in range(case["frames"])]
        # the observed trajectory: another body's, a few millimetres to centimetres away
        t = np.array(S["frame_sub"])[:, None, None] * S["dt"]
        S["target"] = f32(x + t * S["v"] + 0.02 * np.sin(7.0 * x) + 0.005 * rng.standard_normal((1, 3)))
    return S


def _keys(case, seed, S):
    """Key frames of a scene: the loaded state and later ones of the same kind (v, C, F)."""
    rng = np.random.Generator(np.random.PCG64([seed, case["n"], 1]))
    out = []
    for k in range(case["keys"]):
        th = 0.2 * k
        R = np.array([[math.cos(th), -math.sin(th), 0.0], [math.sin(th), math.cos(th), 0.0], [0, 0, 1.0]])
        F = np.einsum("ij,njk->nik", R, S["F"].reshape(-1, 3, 3)).reshape(-1, 9)
        F = F + 0.01 * rng.standard_normal(F.shape, dtype=np.float32)
        out.append((S["v"] + np.float32(0.1 * k), S["C"] * np.float32(1.0 + 0.2 * k), F.astype(np.float32)))
    return out


def _dev(a, device="cuda"):
    return None if a is None else torch.from_numpy(np.ascontiguousarray(a)).to(device)


def _splat_inputs(case, seed, S):
    cov = scenes.gaussian_covariances(types.SimpleNamespace(n=case["n"], dx=S["dx"]), k_seed=seed)
    col, op = scenes.gaussian_appearance(types.SimpleNamespace(n=case["n"]), k_seed=seed + 1)
    return cov, col, op, scenes.camera(case["width"], case["height"])


def _mcis_inputs(case, seed):
    return scenes.mcis_case((case["surface"],) * 3, (case["candidates"],) * 3, (case["draws"],) * 3, k_seed=seed)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "mcis":
        m = _mcis_inputs(case, seed)
        return dict(case=case, surf_off=m["surf_off"], cand_off=m["cand_off"], draw_off=m["draw_off"],
                    surf=_dev(m["surf"]), cand=_dev(m["cand"]), u=_dev(m["u"]))
    S = _state(case, seed)
    st = dict(case=case, scene=S)
    st["init"] = {k: _dev(S[k]) for k in ("x", "v", "C", "F", "vol", "mat_id", "instance")}
    st["params"] = _dev(S["params"])
    if kind == "substep":
        n = case["n"]
        st["out"] = {k: torch.empty((n, w), device="cuda") for k, w in (("x", 3), ("v", 3), ("C", 9), ("F", 9))}
        t = S["materials"]
        st["table"] = (_lib.mpm_material * len(t))(*[
            _lib.mpm_material(m["elastic"], m["plastic"], m["E"], m["nu"], m["rho"], m["yield_stress"],
                              m["friction_angle_deg"]) for m in t])
        st["grid"] = (ctypes.c_int32 * 3)(*S["grid"])
        st["g"] = (ctypes.c_float * 3)(*GRAVITY)
        return st
    st["sim"] = Simulator(S["grid"], S["dx"], S["dt"], GRAVITY, S["materials"], n_instances=case["instances"],
                          ckpt_every=case.get("every", 20))
    if kind == "grad":
        st["target"] = _dev(S["target"])
    elif kind == "bgdo":
        i = st["init"]
        for slot, (v, C, F) in enumerate(_keys(case, seed, S)):
            st["sim"].load(i["x"], i["vol"], i["mat_id"], v=_dev(v), C=_dev(C), F=_dev(F), params=st["params"])
            st["sim"].snapshot(slot)
        torch.cuda.synchronize()
    elif kind == "splat":
        i = st["init"]
        cov, col, op, cam = _splat_inputs(case, seed, S)
        st["sim"].load(i["x"], i["vol"], i["mat_id"], v=i["v"], C=i["C"], F=i["F"], params=st["params"])
        st["sim"].load_covariance(_dev(cov))
        st.update(color=_dev(col), opacity=_dev(op), camera=cam)
    return st


# ---------------------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------------------

def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "mcis":
        return mcis(state["surf_off"], state["surf"], state["cand_off"], state["cand"], state["draw_off"], state["u"])
    if kind == "substep":
        S, i, o = state["scene"], state["init"], state["out"]
        p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
        _lib.check(_lib.lib().mpm_substep_noalloc(
            state["grid"], S["dx"], S["dt"], state["g"], state["table"], len(state["table"]), None, case["n"],
            p(i["x"]), p(i["v"]), p(i["C"]), p(i["F"]), p(i["vol"]), p(i["mat_id"]), p(o["x"]), p(o["v"]), p(o["C"]),
            p(o["F"]), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
        return o
    sim, i = state["sim"], state["init"]
    if kind == "frame":
        sim.load(i["x"], i["vol"], i["mat_id"], v=i["v"], C=i["C"], F=i["F"], instance=i["instance"],
                 params=state["params"])
        sim.step(case["steps"])
        return sim.get()
    if kind == "grad":
        params = state["params"].clone().requires_grad_(True)
        frames = trajectory(params, sim, i, state["scene"]["frame_sub"])
        d = frames - state["target"]
        loss = (d * d).sum() / (frames.shape[0] * frames.shape[1])
        loss.backward()
        out = dict(frames=frames.detach(), grad=params.grad)
        if case["instances"] > 1:
            out["per_candidate"] = sim.reduce_by_material(params.grad)
        return out
    if kind == "bgdo":
        return sim.bgdo(list(range(case["keys"])), signals=True)
    x, cov = sim.positions(), sim.covariance()
    view, fx, fy, cx, cy = state["camera"]
    img, trans = render(x, cov, state["color"], state["opacity"], view, fx, fy, cx, cy, case["width"], case["height"])
    return dict(x=x, cov=cov, image=img, trans=trans)


# ---------------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------------------

# one particle-substep: the state (x v C F, 96 B) read and written once, its material word; about 0.19 active
# nodes per particle, 32 B each.  Operations: 27 nodes x (12 gathered + 16 scattered) and some 600 for the
# F update, the SVD, the return map and the stress.
STEP_BYTES, STEP_FLOPS = 200, 1400
# a recorded forward, its recompute and the reverse of one substep
GRAD_BYTES, GRAD_FLOPS = 880, 5600


def work(case):
    kind = case["kind"]
    if kind == "mcis":
        s, c, d = 3 * case["surface"], 3 * case["candidates"], 3 * case["draws"]
        # points in, distance and weight out; uniform in, index out; some tens of surface points per candidate
        return dict(bytes=12 * s + 28 * c + 16 * d, flops=8 * 64 * c)
    n = case["n"]
    if kind == "substep":
        return dict(bytes=STEP_BYTES * n, flops=STEP_FLOPS * n)
    if kind == "frame":
        return dict(bytes=n * (200 + STEP_BYTES * case["steps"]), flops=n * STEP_FLOPS * case["steps"])
    if kind == "grad":
        return dict(bytes=n * (24 * case["frames"] + GRAD_BYTES * case["steps"]), flops=n * GRAD_FLOPS * case["steps"])
    if kind == "bgdo":
        return dict(bytes=n * (288 * case["keys"] + 8), flops=n * (STEP_FLOPS + 400) * case["keys"])
    pix = case["width"] * case["height"]
    # state, covariance, colour and opacity in; positions, covariances and the image out; a few pixels a Gaussian
    return dict(bytes=n * (48 + 24 + 16 + 36) + 16 * pix, flops=n * 400 + 20 * 40 * pix)


# ---------------------------------------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------------------------------------

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


class _Eigh(torch.autograd.Function):
    """Eigenvalues (n, 3) and eigenvectors (n, 3, 3, columns) of symmetric 3x3 matrices by cyclic Jacobi."""

    @staticmethod
    def forward(ctx, B):
        a = {(i, j): B[:, i, j].clone() for i in range(3) for j in range(i, 3)}
        V = torch.eye(3, dtype=B.dtype, device=B.device).expand_as(B).clone()
        for _ in range(7):
            for p, q, r in ((0, 1, 2), (0, 2, 1), (1, 2, 0)):
                pr, qr = (min(p, r), max(p, r)), (min(q, r), max(q, r))
                apq, app, aqq = a[p, q], a[p, p], a[q, q]
                th = (aqq - app) / torch.where(apq == 0, 1.0, 2.0 * apq)
                t = torch.where(th >= 0, 1.0, -1.0) / (th.abs() + torch.sqrt(th * th + 1.0))
                t = torch.where(apq == 0, 0.0, t)
                c = torch.rsqrt(t * t + 1.0)
                s = t * c
                a[p, p], a[q, q], a[p, q] = app - t * apq, aqq + t * apq, torch.zeros_like(apq)
                a[pr], a[qr] = c * a[pr] - s * a[qr], s * a[pr] + c * a[qr]
                vp, vq = V[:, :, p].clone(), V[:, :, q].clone()
                V[:, :, p], V[:, :, q] = c[:, None] * vp - s[:, None] * vq, s[:, None] * vp + c[:, None] * vq
        lam = torch.stack([a[0, 0], a[1, 1], a[2, 2]], 1)
        ctx.save_for_backward(lam, V)
        return lam, V

    @staticmethod
    def backward(ctx, glam, gV):
        lam, V = ctx.saved_tensors
        gap = lam[:, None, :] - lam[:, :, None]
        K = torch.where(gap.abs() < 1e-13, 0.0, 1.0 / torch.where(gap == 0, 1.0, gap))
        M = torch.diag_embed(glam) + (V.transpose(1, 2) @ gV) * K
        G = V @ M @ V.transpose(1, 2)
        return 0.5 * (G + G.transpose(1, 2))


class _Mpm64:
    """The substep of the library's header (MLS-MPM, quadratic B-spline, APIC) in 64 bits, on dense grids."""

    def __init__(self, S, instances, device):
        t64 = lambda a: torch.as_tensor(a, dtype=torch.float64, device=device)  # noqa: E731
        self.device = device
        self.R = S["grid"]
        self.dx, self.dt = float(np.float32(S["dx"])), float(np.float32(S["dt"]))
        self.g = t64(np.asarray(GRAVITY, np.float32))
        ids = torch.as_tensor(S["mat_id"], dtype=torch.int64, device=device)
        col = lambda k: t64(np.array([np.float32(m[k]) for m in S["materials"]], np.float64))[ids]  # noqa: E731
        self.elastic, self.plastic = col("elastic").long(), col("plastic").long()
        self.models = sorted({m["elastic"] for m in S["materials"]}), sorted({m["plastic"] for m in S["materials"]})
        self.vol = t64(S["vol"])
        self.mass = col("rho") * self.vol
        phi = torch.sin(col("friction_angle_deg") * (math.pi / 180.0))
        self.alpha = math.sqrt(2.0 / 3.0) * 2.0 * phi / (3.0 - phi)
        self.params = torch.stack([torch.log(col("E")), col("nu"), col("yield_stress")], 1)
        if S["params"] is not None:
            self.params = t64(S["params"])
        n = len(S["x"])
        self.state = (t64(S["x"]), t64(S["v"]), t64(S["C"]).reshape(n, 3, 3), t64(S["F"]).reshape(n, 3, 3))
        self.instances = instances
        self.inst = 0 if S["instance"] is None else torch.as_tensor(S["instance"], dtype=torch.int64, device=device)
        self.open, self.block = self._walls()

    def _walls(self):
        idx = torch.stack(torch.meshgrid(*[torch.arange(r, device=self.device) for r in self.R], indexing="ij"), -1)
        idx = idx.reshape(-1, 3)
        res = torch.tensor(self.R, device=self.device)
        lo, hi = idx < BOUND, idx >= res - BOUND
        w = torch.tensor(WALLS, device=self.device).reshape(3, 2)
        sticky = ((lo & (w[:, 0] == 2)) | (hi & (w[:, 1] == 2))).any(1, keepdim=True)
        return ~sticky, (lo & (w[:, 0] == 1), hi & (w[:, 1] == 1))

    def lame(self, params):
        E, nu = torch.exp(params[:, 0]), params[:, 1]
        return E / (2.0 * (1.0 + nu)), E * nu / ((1.0 + nu) * (1.0 - 2.0 * nu))

    def svd(self, F):
        lam, V = _Eigh.apply(F.transpose(1, 2) @ F)
        s = torch.sqrt(lam)
        return (F @ V) / s[:, None, :], s, V

    def stress(self, F, mu, lam):
        """Kirchhoff stress of every particle's model."""
        eye = torch.eye(3, dtype=F.dtype, device=F.device)
        J = torch.linalg.det(F)
        out = torch.zeros_like(F)
        iso = lambda a: a[:, None, None] * eye  # noqa: E731
        for m in self.models[0]:
            if m in (0, 3):
                U, s, _ = self.svd(F)
            if m == 0:
                t = (U * (2.0 * mu[:, None] * (s - 1.0) * s)[:, None, :]) @ U.transpose(1, 2) + iso(lam * J * (J - 1.0))
            elif m == 1:
                t = mu[:, None, None] * (F @ F.transpose(1, 2) - eye) + iso(lam * torch.log(J))
            elif m == 2:
                E = 0.5 * (F.transpose(1, 2) @ F - eye)
                t = 2.0 * mu[:, None, None] * (F @ E @ F.transpose(1, 2)) + iso(lam * J * (J - 1.0))
            elif m == 3:
                eps = torch.log(s.clamp_min(1e-4))
                t = (U * (2.0 * mu[:, None] * eps + (lam * eps.sum(1))[:, None])[:, None, :]) @ U.transpose(1, 2)
            elif m == 4:
                t = iso(lam * J * (J - 1.0))
            else:
                t = iso((2.0 * mu / 3.0 + lam) * (J - 1.0 / J))
            out = torch.where((self.elastic == m)[:, None, None], t, out)
        return out

    def return_map(self, F, mu, lam, ys):
        for m in self.models[1]:
            if m == 0:
                continue
            if m in (1, 2):
                U, s, V = self.svd(F)
                eps = torch.log(s.clamp_min(1e-4))
                tr = eps.sum(1)
                h = eps - tr[:, None] / 3.0
                nrm = torch.sqrt((h * h).sum(1))
                dg = nrm - ys / (2.0 * mu) if m == 1 else nrm + (3.0 * lam + 2.0 * mu) / (2.0 * mu) * tr * self.alpha
                z = torch.exp(eps - (dg / nrm)[:, None] * h)
                changed = dg > 0.0
                if m == 2:
                    z = torch.where((tr > 0.0)[:, None], 1.0, z)
                    changed = changed | (tr > 0.0)
                new = torch.where(changed[:, None, None], (U * z[:, None, :]) @ V.transpose(1, 2), F)
            else:
                J = torch.linalg.det(F)
                J = J.clamp(0.05, 1.2) if m == 4 else J
                c = torch.sign(J) * J.abs() ** (1.0 / 3.0)
                new = c[:, None, None] * torch.eye(3, dtype=F.dtype, device=F.device)
            F = torch.where((self.plastic == m)[:, None, None], new, F)
        return F

    def substep(self, x, v, C, F, params):
        mu, lam = self.lame(params)
        X = x / self.dx
        base = torch.floor(X - 0.5)
        f = X - base
        w = (0.5 * (1.5 - f) ** 2, 0.75 - (f - 1.0) ** 2, 0.5 * (f - 0.5) ** 2)
        b = base.long()
        k = (4.0 * self.dt / self.dx ** 2) * self.vol
        A = self.mass[:, None, None] * C - k[:, None, None] * self.stress(F, mu, lam)
        Pm = self.mass[:, None] * v
        nodes = self.R[0] * self.R[1] * self.R[2]

        def stencil():
            for o in range(27):
                i, j, l = o // 9, (o // 3) % 3, o % 3
                node = ((b[:, 0] + i) * self.R[1] + b[:, 1] + j) * self.R[2] + b[:, 2] + l + self.inst * nodes
                d = torch.tensor([i, j, l], dtype=x.dtype, device=x.device) - f
                yield node, w[i][:, 0] * w[j][:, 1] * w[l][:, 2], d * self.dx

        grid = torch.zeros((self.instances * nodes, 4), dtype=x.dtype, device=x.device)
        for node, wt, d in stencil():
            q = torch.cat([Pm + (A @ d[:, :, None])[:, :, 0], self.mass[:, None]], 1)
            grid = grid.index_add(0, node, wt[:, None] * q) if grid.requires_grad or q.requires_grad else \
                grid.index_add_(0, node, wt[:, None] * q)
        m = grid[:, 3:]
        u = torch.where(m > 0, grid[:, :3] / torch.where(m > 0, m, 1.0) + self.dt * self.g, 0.0)
        u = u.reshape(self.instances, nodes, 3)
        u = torch.where(self.open, u, 0.0)
        u = torch.where(self.block[0] & (u < 0), 0.0, u)
        u = torch.where(self.block[1] & (u > 0), 0.0, u).reshape(-1, 3)
        vn, Cn = torch.zeros_like(v), torch.zeros_like(C)
        for node, wt, d in stencil():
            a = wt[:, None] * u[node]
            vn = vn + a
            Cn = Cn + a[:, :, None] * d[:, None, :]
        Cn = Cn * (4.0 / self.dx ** 2)
        Fn = F + self.dt * (Cn @ F)
        return x + self.dt * vn, vn, Cn, self.return_map(Fn, mu, lam, params[:, 2])


def _exact_frame(case, seed, instances=None, steps=None):
    S = _state(case, seed)
    M = _Mpm64(S, instances or case["instances"], _device())
    st = M.state
    for _ in range(steps if steps is not None else case["steps"]):
        st = M.substep(*st, M.params)
    return dict(zip(("x", "v", "C", "F"), st))


def _exact_grad(case, seed):
    S = _state(case, seed)
    M = _Mpm64(S, case["instances"], _device())
    with_grad = case["n"] * case["steps"] <= 8_000_000
    params = M.params.clone().requires_grad_(with_grad)
    st, frames, done = M.state, [], 0
    for sub in S["frame_sub"]:
        for _ in range(sub - done):
            st = checkpoint(M.substep, *st, params, use_reentrant=False) if with_grad else M.substep(*st, params)
        done = sub
        frames.append(st[0])
    x = torch.stack(frames)
    out = dict(frames=x.detach(), grad=None)
    if with_grad:
        d = x - torch.as_tensor(S["target"], dtype=torch.float64, device=x.device)
        ((d * d).sum() / (x.shape[0] * x.shape[1])).backward()
        out["grad"] = params.grad
    if case["instances"] > 1:
        out["per_candidate"] = None
        if with_grad:
            sums = torch.zeros((len(S["materials"]), 3), dtype=torch.float64, device=x.device)
            out["per_candidate"] = sums.index_add(0, torch.as_tensor(S["mat_id"], device=x.device).long(), params.grad)
    return out


def _exact_bgdo(case, seed):
    S = _state(case, seed)
    M = _Mpm64(S, 1, _device())
    mu, lam = M.lame(M.params)
    logE = M.params[:, 0]
    eta = (0.1 * torch.log1p(torch.exp(logE))).clamp_max(1.0)
    G, gs, ds = 0.0, [], []
    eye = torch.eye(3, dtype=torch.float64, device=M.device)
    for v, C, F in _keys(case, seed, S):
        v, C, F = (torch.as_tensor(a, dtype=torch.float64, device=M.device) for a in (v, C, F))
        C, F = C.reshape(-1, 3, 3), F.reshape(-1, 3, 3)
        g = torch.linalg.matrix_norm(M.stress(F, mu, lam))
        d = torch.linalg.matrix_norm(M.substep(M.state[0], v, C, F, M.params)[3] - eye)
        G = G + (eta * torch.log1p(g) - (1.0 - eta) * (d - float(np.float32(0.1)))) / case["keys"]
        gs.append(g)
        ds.append(d)
    return dict(G=G, log_E=logE - G, g_tau=torch.stack(gs), delta=torch.stack(ds))


def _exact_splat(case, seed):
    S = _state(case, seed)
    dv = _device()
    t64 = lambda a: torch.as_tensor(a, dtype=torch.float64, device=dv)  # noqa: E731
    cov, col, op, (view, fx, fy, cx, cy) = _splat_inputs(case, seed, S)
    x, F, c0, col, op = t64(S["x"]), t64(S["F"]).reshape(-1, 3, 3), t64(cov), t64(col), t64(op)
    view = t64(np.asarray(view, np.float32)).reshape(3, 4)
    fx, fy, cx, cy = (float(np.float32(a)) for a in (fx, fy, cx, cy))
    pick = torch.tensor([0, 1, 2, 1, 3, 4, 2, 4, 5], device=dv)
    Sg = F @ c0[:, pick].reshape(-1, 3, 3) @ F.transpose(1, 2)
    W, H = case["width"], case["height"]
    t = x @ view[:, :3].T + view[:, 3]
    keep = t[:, 2] > 0.2
    t, col, op, Sc = t[keep], col[keep], op[keep], (view[:, :3] @ Sg @ view[:, :3].T)[keep]
    z, zero = t[:, 2], torch.zeros_like(t[:, 2])
    Jm = torch.stack([fx / z, zero, -fx * t[:, 0] / z ** 2, zero, fy / z, -fy * t[:, 1] / z ** 2], 1).reshape(-1, 2, 3)
    P = Jm @ Sc @ Jm.transpose(1, 2) + 0.3 * torch.eye(2, dtype=torch.float64, device=dv)
    a, b, d = P[:, 0, 0], P[:, 0, 1], P[:, 1, 1]
    det, mid = a * d - b * b, 0.5 * (a + d)
    rad = torch.ceil(3.0 * torch.sqrt(mid + torch.sqrt((mid * mid - det).clamp_min(0.1))))
    u, v = fx * t[:, 0] / z + cx, fy * t[:, 1] / z + cy
    gx, gy = (W + 15) // 16, (H + 15) // 16
    x0, x1 = torch.floor((u - rad) / 16).clamp(0, gx), torch.floor((u + rad + 15) / 16).clamp(0, gx)
    y0, y1 = torch.floor((v - rad) / 16).clamp(0, gy), torch.floor((v + rad + 15) / 16).clamp(0, gy)
    order = torch.sort(z, stable=True)[1]
    u, v, a, b, d, det, op, col, x0, x1, y0, y1 = (q[order] for q in (u, v, a, b, d, det, op, col, x0, x1, y0, y1))
    img = torch.zeros((H, W, 3), dtype=torch.float64, device=dv)
    tr = torch.ones((H, W), dtype=torch.float64, device=dv)
    for ty in range(gy):
        row = torch.nonzero((y0 <= ty) & (ty < y1))[:, 0]
        for tx in range(gx):
            i = row[(x0[row] <= tx) & (tx < x1[row])]
            px = torch.arange(16 * tx, min(W, 16 * tx + 16), device=dv) + 0.5
            py = torch.arange(16 * ty, min(H, 16 * ty + 16), device=dv) + 0.5
            ex, ey = px[None, None, :] - u[i, None, None], py[None, :, None] - v[i, None, None]
            A, B, D = (q[i, None, None] for q in (d / det, -b / det, a / det))
            power = -0.5 * (A * ex * ex + D * ey * ey) - B * ex * ey
            al = (op[i, None, None] * torch.exp(power)).clamp_max(0.99)
            al = torch.where((power > 0) | (al < 1.0 / 255.0), 0.0, al)
            T = torch.cumprod(1.0 - al, 0)
            seen = T >= 1e-4
            before = torch.cat([torch.ones_like(T[:1]), T[:-1]]) if len(i) else T
            c = torch.einsum("kyx,kc->yxc", torch.where(seen, al * before, 0.0), col[i])
            sl = (slice(16 * ty, 16 * ty + len(py)), slice(16 * tx, 16 * tx + len(px)))
            img[sl] = c
            if len(i):
                tr[sl] = torch.where(seen, T, 1.0).amin(0)
    return dict(x=x, cov=Sg.reshape(-1, 9)[:, [0, 1, 2, 4, 5, 8]], image=img, trans=tr)


def _exact_mcis(case, seed):
    m, dv = _mcis_inputs(case, seed), _device()
    surf, cand = (torch.as_tensor(m[k], dtype=torch.float64, device=dv) for k in ("surf", "cand"))
    out = []
    for k in range(3):
        s = surf[m["surf_off"][k]:m["surf_off"][k + 1]]
        for q in torch.split(cand[m["cand_off"][k]:m["cand_off"][k + 1]], max(1, 400_000_000 // len(s))):
            d2 = (q[:, None, 0] - s[None, :, 0]) ** 2
            for a in (1, 2):
                d2 += (q[:, None, a] - s[None, :, a]) ** 2
            out.append(d2.amin(1))
    d2 = torch.cat(out)
    w = torch.exp(-d2 / (2.0 * 0.02 ** 2)).clamp_min(1e-6)
    # beyond the cut-off the distance may be larger than the true one
    within = bool((d2 <= 2.0 * 0.02 ** 2 * math.log(1e6)).all())
    return dict(d=torch.sqrt(d2) if within else None, w=w, picked=None)


def exact(case, seed):
    kind = case["kind"]
    # on the host alone the larger ones would take minutes
    if _device() == "cpu" and (kind in ("splat", "mcis") or case["n"] * case.get("steps", 1) > 200_000):
        return None
    if kind == "substep":
        S = _exact_frame(dict(case, objects=1, instances=1), seed, steps=1)
        n = case["n"]
        return dict(S, C=S["C"].reshape(n, 9), F=S["F"].reshape(n, 9))
    with torch.no_grad():
        if kind == "frame":
            return _exact_frame(case, seed)
        if kind == "bgdo":
            return _exact_bgdo(case, seed)
        if kind == "splat":
            return _exact_splat(case, seed)
        if kind == "mcis":
            return _exact_mcis(case, seed)
    return _exact_grad(case, seed)
