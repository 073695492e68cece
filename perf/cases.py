"""The solver's workloads as cases to be timed and compared: what each stands for, its inputs, one pass of it through
the public entry points, the work it cannot do without, and the same answer in 64 bits from plain torch.

A case is a dict of plain values: `kind` names the entry point, `shape` the scene and `a`, `b`, `c` its sizes (cells per
axis, or bodies and cells), `dtype` the solver's form (f32: SIM_FP32_MIXED, f64: SIM_FP64).  Scenes are the ones of
paper_2405_08001_gb300.scenes, moved by seeded deformations into the states that the solver meets in a run: strained,
twisted, and in contact.

Every step case starts from a given state (sim_set_state, as a program does that resumes a run, tries several controls
from one state, or resets an episode), advances one time step and reads the state back.  The method is chaotic: a
difference of rounding grows by about a factor of ten every five iterations once contacts or the step cap are active
(measured on two runs of the same inputs, whose atomic sums come in another order), so that in float the contact cases
run as many iterations as leave the two runs comparable: a real-time program's counts, not the configurations' 50.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2405_08001_gb300 import binding as B
from paper_2405_08001_gb300 import diff
from paper_2405_08001_gb300 import scenes as S

MODELS = {"nh": B.SIM_MAT_NH, "snh": B.SIM_MAT_SNH, "fcr": B.SIM_MAT_FCR, "arap": B.SIM_MAT_ARAP}


# ----------------------------------------------------------------------------------------------------- the cases

def _case(name, kind, shape, a, b, c, dtype, iters=0, model="nh", beta="pr", split=0):
    return {"name": name, "kind": kind, "shape": shape, "a": a, "b": b, "c": c, "dtype": dtype, "iters": iters,
            "model": model, "beta": beta, "split": split}


def listed():
    return [
        # the smallest step: two blocks of 3^3 cells meeting corner first, as in an interactive scene or a unit test of
        # a program that uses the solver: latency alone
        _case("step blocks f64", "step", "blocks", 3, 3, 3, "f64", iters=20),
        # the drop of 8^3 cells onto a plane (the framework's first configuration), 50 iterations, in contact
        _case("step drop f32", "step", "cube", 8, 8, 8, "f32", iters=50),
        # the benchmark's twisted bar, 98,304 tets, about two turns between its ends: self-contact candidates
        _case("step bar f32", "step", "bar", 16, 16, 64, "f32", iters=25),
        # the same bar in the plain form: a user who needs 64 bits throughout
        _case("step bar f64", "step", "bar", 16, 16, 64, "f64", iters=50),
        # the largest: ten bars stacked crosswise within the barrier's reach, 983,040 tets, tens of thousands of pairs
        _case("step stack f32", "step", "stack", 10, 16, 64, "f32", iters=15),
        # independent scenes in one handle (learning, parameter sweeps), 64 cubes of 4^3 to 16^3 cells at the plane
        _case("step batch f32", "step", "batch", 64, 4, 16, "f32", iters=15),
        # bodies that touch, each with its own step size (split objects), odd sizes
        _case("step objects f32", "step", "stack", 4, 5, 19, "f32", iters=12, split=1),
        # one evaluation at given positions from host arrays (a line search, a monitor, another optimiser): ragged bar
        _case("gradient bar f32", "gradient", "bar", 15, 17, 61, "f32"),
        # Hessian times vector on the device (a Newton-Krylov or eigenvalue program), the 24^3 cube
        _case("hvp cube f64", "hvp", "cube", 24, 24, 24, "f64"),
        # the reverse of one time step of the same cube (the differentiation configuration)
        _case("adjoint cube f64", "adjoint", "cube", 24, 24, 24, "f64", iters=2000),
        # the allocation-free p^T H p on caller-owned device buffers, a large mesh
        _case("php noalloc large", "noalloc", "cube", 55, 55, 55, "f64"),
        # fitting per-tet moduli and initial velocities through two time steps of a small cube, forward and backward
        _case("train cube f64", "train", "cube", 5, 4, 6, "f64", iters=400),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box(rng, cells_lo, cells_hi):
    """Odd cell counts of a box of about the drawn number of cells."""
    n = _log_int(rng, cells_lo, cells_hi)
    s = n ** (1.0 / 3.0)
    a = max(2, round(s * rng.uniform(0.7, 1.3)))
    b = max(2, round(s * rng.uniform(0.7, 1.3)))
    return a, b, max(2, round(n / (a * b)))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "gradient", "energy", "php", "hvp", "adjoint", "noalloc", "train"])
    dtype = rng.choice(["f32", "f32", "f64"])
    model = rng.choice(["nh", "nh", "nh", "snh", "fcr", "arap"])
    if kind == "step":
        shape = rng.choice(["blocks", "cube", "bar", "stack", "batch"])
        beta, split = rng.choice(["pr", "pr", "dk"]), 0
        iters = rng.randint(10, 50) if dtype == "f64" else rng.randint(10, 30) if shape == "cube" else rng.randint(5, 16)
        if shape == "blocks":
            a = b = c = rng.randint(2, 6)
        elif shape == "cube":
            a, b, c = _box(rng, 27, 20000 if dtype == "f32" else 8000)
        elif shape == "bar":
            a, b = rng.randint(4, 20), rng.randint(4, 20)
            c = rng.randint(3, 4) * max(a, b)
            model = rng.choice(["nh", "nh", "snh"])
        elif shape == "stack":
            a, b = rng.randint(2, 8), rng.randint(3, 12)
            c, model, split = 4 * b - rng.randint(0, 3), "nh", rng.choice([0, 0, 1])
        else:
            a, b = _log_int(rng, 2, 60), rng.randint(2, 5)
            c, model, dtype, iters = b + rng.randint(0, 8), "nh", "f32", rng.randint(5, 16)
        return _case("", kind, shape, a, b, c, dtype, iters, model, beta, split)
    if kind == "noalloc":
        return _case("", kind, "cube", *_box(rng, 8, 150000), "f64")
    if kind == "train":
        return _case("", kind, "cube", *_box(rng, 27, 300), "f64", iters=400)
    if kind == "adjoint":
        return _case("", kind, "cube", *_box(rng, 27, 12000), "f64", iters=2000, model=rng.choice(["nh", "snh"]))
    if kind == "hvp":
        return _case("", kind, "cube", *_box(rng, 27, 30000), dtype, model=model)
    if rng.random() < 0.5:
        a, b = rng.randint(4, 20), rng.randint(4, 20)
        return _case("", kind, "bar", a, b, 4 * max(a, b), dtype, model=rng.choice(["nh", "snh"]))
    return _case("", kind, "cube", *_box(rng, 27, 30000), dtype, model=model)


# ----------------------------------------------------------------------------------------------------- inputs

def _waves(X, rng, strain):
    """A seeded smooth displacement of about the given strain: a few long sine waves."""
    size = float((X.max(0) - X.min(0)).max())
    u = np.zeros_like(X)
    for _ in range(3):
        k = rng.normal(size=3) * (2.0 / size)
        d = rng.normal(size=3)
        u += np.sin(X @ k + rng.uniform(0.0, 2.0 * math.pi))[:, None] * d / (np.linalg.norm(k) * np.linalg.norm(d))
    return strain * u


def _inputs(case, seed):
    """The scene with its state (scene.x0, scene.v0), the targets of the kinematic vertices and a generator."""
    rng = np.random.default_rng([int(seed), 77])
    shape, a, b, c = case["shape"], case["a"], case["b"], case["c"]
    targets = None
    if shape == "blocks":
        sc = S.two_blocks(int(seed) % 100003, n=a, side=0.01 * a, iters=case["iters"])
        sc.x0 = sc.x0 + _waves(sc.x0, rng, 0.002)
    elif shape == "cube":
        # a strained box whose lowest vertices are inside the plane barrier's reach; flying clear of it where steps have
        # to converge and where the barrier's curvature would hide the elastic part of the output
        sc = S.cube_drop(n=max(a, b, c), cells=(a, b, c), iters=max(case["iters"], 1), drop=0.0)
        clear = case["kind"] in ("train", "hvp", "php")
        x = sc.rest_x + _waves(sc.rest_x, rng, 0.01)
        x = x + rng.normal(scale=1e-3 * 0.1 / max(a, b, c), size=x.shape)
        x[:, 2] += -x[:, 2].min() + (0.02 if clear else rng.uniform(0.4, 0.7) * sc.dhat)
        sc.x0 = x
        sc.v0 = _waves(sc.rest_x, rng, 0.5) + rng.normal(scale=0.2, size=3)
        if not clear:
            sc.v0[:, 2] = -0.05 * rng.random() + 0.1 * sc.v0[:, 2]
    elif shape == "bar":
        # pure torsion by the angle that the caps have reached, between one and two turns apart, in rotation
        h = 0.1 / max(a, b)
        sc = S.twisted_bar(a, b, c, size=(a * h, b * h, c * h), iters=max(case["iters"], 1))
        L, axis = c * h, np.array([0.5 * a * h, 0.5 * b * h, 0.0])
        th = rng.uniform(4.0, 7.0) * (L / 0.4)
        q = 2.0 * sc.rest_x[:, 2] / L - 1.0
        u = sc.rest_x + _waves(sc.rest_x, rng, 0.004) * (1.0 - q * q)[:, None]
        u = u + rng.normal(scale=1e-3 * h, size=u.shape) * (sc.fixed == 0)[:, None]
        co, si, r = np.cos(th * q), np.sin(th * q), u - axis
        sc.x0 = np.stack([co * r[:, 0] - si * r[:, 1], si * r[:, 0] + co * r[:, 1], r[:, 2]], 1) + axis
        w = 2.0 * q
        sc.v0 = np.stack([-w * (sc.x0[:, 1] - axis[1]), w * (sc.x0[:, 0] - axis[0]), 0.0 * w], 1)
        f = np.nonzero(sc.fixed)[0]
        d = 2.0 * sc.dt * np.sign(q[f])
        r = sc.x0[f] - axis
        targets = np.stack([np.cos(d) * r[:, 0] - np.sin(d) * r[:, 1], np.sin(d) * r[:, 0] + np.cos(d) * r[:, 1], r[:, 2]], 1) + axis
    elif shape == "stack":
        # bars of b x b x c cells laid crosswise, their faces half the barrier's reach apart, pressed together
        h = 0.1 / b
        sc = S.pile(a, cells=(b, b, c), size=(0.1, 0.1, c * h), seed=int(seed) % 100003, gap=0.6, iters=case["iters"])
        n = sc.n_verts // a
        sc.x0 = sc.rest_x + rng.normal(scale=0.02 * sc.dhat, size=sc.rest_x.shape)
        sc.v0 = np.repeat(rng.normal(scale=0.01, size=(a, 3)) + np.array([0.0, 0.0, -0.01]), n, 0)
        if case["split"]:
            sc.scene_of_vert = np.repeat(np.arange(a), n).astype(np.int32)
    else:
        # the sizes and orientations belong to the case, the stiffnesses, heights and speeds to the seed
        sc = S.batched(a, seed=1000 * b + c, n_min=b, n_max=c, iters=case["iters"])
        sc.youngs_per_tet = rng.uniform(5e4, 5e5, size=a)[sc.scene_of_vert[sc.tets[:, 0]]]
        low = np.full(a, np.inf)
        np.minimum.at(low, sc.scene_of_vert, sc.x0[:, 2])
        drop = low - rng.uniform(0.3, 0.9, size=a) * sc.dhat
        sc.x0 = sc.x0 - drop[sc.scene_of_vert][:, None] * np.array([0.0, 0.0, 1.0])
        sc.v0 = np.array([0.0, 0.0, -0.1]) * rng.random(a)[sc.scene_of_vert][:, None]
    return sc, targets, rng


def _vectors(case, sc, rng):
    """The further vectors of the evaluation and differentiation cases: a direction, a prediction, loss gradients."""
    n = sc.x0.shape
    p = 1e-3 * (rng.normal(size=n) + 3.0 * _waves(sc.rest_x, rng, 1.0) / 0.1)
    xt = sc.x0 + sc.dt * sc.v0 + rng.normal(scale=1e-6, size=n)
    return p, xt, rng.normal(size=n), 0.02 * rng.normal(size=n)


def _lumped(sc):
    """Lumped masses: a quarter of each tet's rest mass to each corner."""
    X = sc.rest_x[sc.tets]
    vol = np.linalg.det(X[:, 1:] - X[:, :1]) / 6.0
    m = np.zeros(sc.n_verts)
    np.add.at(m, sc.tets.reshape(-1), np.repeat(sc.density * vol / 4.0, 4))
    return m


def prepare(case, seed):
    sc, targets, rng = _inputs(case, seed)
    p, xt, ax, av = _vectors(case, sc, rng)
    kind = case["kind"]

    def dev(v, t=torch.float64):
        return torch.as_tensor(np.ascontiguousarray(v), dtype=t).cuda()

    st = {"kind": kind, "scene": sc}
    if kind == "train":
        st["E"] = dev(sc.youngs * (1.0 + 0.2 * rng.random(sc.n_tets)))
        st["v0"], st["x_goal"] = dev(sc.v0), dev(sc.x0 + 2.0 * sc.dt * sc.v0 + 0.01 * rng.normal(size=3))
        return st
    if kind == "noalloc":
        st.update(x=dev(sc.x0), p=dev(p), X=dev(sc.rest_x), tets=dev(sc.tets, torch.int32), mass=dev(_lumped(sc)))
        return st
    # the handle's work goes to a stream of the program's own, as its tensors' does
    st["stream"] = torch.cuda.Stream()
    st["sim"] = B.Sim(sc, precision=B.SIM_FP32_MIXED if case["dtype"] == "f32" else B.SIM_FP64, model=MODELS[case["model"]],
                      beta=B.SIM_BETA_DK if case["beta"] == "dk" else B.SIM_BETA_PR_PLUS, split_objects=case["split"],
                      cuda_stream=st["stream"].cuda_stream)
    if kind in ("gradient", "energy", "php"):
        st.update(x=sc.x0.copy(), xt=xt, p=p)
    elif kind == "step":
        st.update(x=dev(sc.x0), v=dev(sc.v0), x_out=dev(0 * sc.x0), v_out=dev(0 * sc.x0),
                  targets=None if targets is None else dev(targets))
    elif kind == "hvp":
        st.update(x=dev(sc.x0), p=dev(p), out=dev(0 * p))
    else:
        st.update(x=dev(sc.x0), ax=dev(ax), av=dev(av), ax0=dev(0 * ax), av0=dev(0 * ax), dE=dev(np.zeros(sc.n_tets)),
                  iters=case["iters"])
    torch.cuda.synchronize()
    return st


def run(st):
    kind = st["kind"]
    if kind == "train":
        E, v0 = st["E"].clone().requires_grad_(), st["v0"].clone().requires_grad_()
        x = diff.simulate(E, v0, st["scene"], 2, tol=1e-10, max_iters=2000)
        loss = ((x - st["x_goal"]) ** 2).sum()
        loss.backward()
        return x.detach(), E.grad, v0.grad
    if kind == "noalloc":
        sc = st["scene"]
        out = torch.empty(1, dtype=torch.float64, device="cuda")
        B.sim_pHp_noalloc(st["x"], st["p"], st["X"], st["tets"], st["mass"], sc.youngs, sc.poisson, sc.dt, out,
                          torch.cuda.current_stream())
        return out
    h = st["sim"].h
    if kind == "step":
        B.sim_set_state(h, st["x"], st["v"])
        B.sim_step(h, 1, st["targets"])
        x, v, _ = B.sim_get_state(h, st["x_out"], st["v_out"])
        return x, v
    if kind == "gradient":
        return B.sim_eval_gradient(h, st["x"], st["xt"])
    if kind == "energy":
        e, parts = B.sim_eval_energy(h, st["x"], st["xt"])
        return e, parts
    if kind == "php":
        return B.sim_eval_pHp(h, st["x"], st["p"])
    if kind == "hvp":
        return B.sim_eval_hvp(h, st["x"], st["p"], st["out"])
    with torch.cuda.stream(st["stream"]):
        st["dE"].zero_()
        ax0, av0, _, _ = B.sim_adjoint_step(h, st["x"], st["ax"], st["av"], dE=st["dE"], tol=1e-10, max_iters=st["iters"],
                                            ax0=st["ax0"], av0=st["av0"])
    return ax0, av0, st["dE"]


# ----------------------------------------------------------------------------------------------------- accounting

def _counts(case):
    """About how many vertices and tets the case has (a batch: by its mean cell count)."""
    a, b, c = case["a"], case["b"], case["c"]
    if case["shape"] == "blocks":
        return 2 * (a + 1) ** 3, 12 * a ** 3
    if case["shape"] == "stack":
        return a * (b + 1) ** 2 * (c + 1), 6 * a * b * b * c
    if case["shape"] == "batch":
        n = range(b, c + 1)
        return a * sum((k + 1) ** 3 for k in n) // len(n), a * sum(6 * k ** 3 for k in n) // len(n)
    return (a + 1) * (b + 1) * (c + 1), 6 * a * b * c


def work(case):
    """Inputs read once and outputs written once; the arithmetic of the method per tet: gradient and diagonal about 220
    operations, the curvature along a direction about 110, a Hessian-vector product about 200; a vertex about 60 for
    each iteration.  A step cannot do without its iterations' arithmetic; its state and mesh fit L2 or not."""
    nv, nt = _counts(case)
    w = 4 if case["dtype"] == "f32" else 8
    mesh = nt * (16 + 10 * w)          # indices, D_m^-1 and the volume
    k = case["kind"]
    if k == "step":
        return {"bytes": mesh + 96 * nv, "flops": case["iters"] * (330 * nt + 60 * nv)}
    if k == "gradient":
        return {"bytes": mesh + 96 * nv, "flops": 220 * nt + 20 * nv}
    if k in ("energy", "php"):
        return {"bytes": mesh + 48 * nv, "flops": 110 * nt + 20 * nv}
    if k == "hvp":
        return {"bytes": mesh + 72 * nv, "flops": 200 * nt + 10 * nv}
    if k == "noalloc":
        return {"bytes": 16 * nt + 80 * nv, "flops": 200 * nt + 10 * nv}
    its = 150 if k == "adjoint" else 2 * (case["iters"] + 100)   # conjugate-gradient iterations of such a solve
    return {"bytes": mesh + 120 * nv + 8 * nt, "flops": its * (200 * nt + 60 * nv)}


def tolerance(case):
    """About four times what two runs of the same inputs, or a run and the 64-bit value, were seen to differ by over a
    few seeds of each kind, rounded up."""
    f32 = case["dtype"] == "f32"
    rel = {"step": 3e-3 if f32 else 1e-5, "gradient": 3e-6 if f32 else 1e-9, "energy": 1e-5 if f32 else 1e-10,
           "php": 1e-5 if f32 else 1e-10, "hvp": 1e-5 if f32 else 1e-10, "adjoint": 1e-8, "noalloc": 1e-11,
           "train": 1e-5}[case["kind"]]
    return {"rel": rel, "max": min(0.5, 100 * rel)}


# ----------------------------------------------------------------------------------------------------- 64 bits

def _cross(a, b):
    return torch.linalg.cross(a, b, dim=-1)


def _dot(a, b):
    return (a * b).sum(-1)


def _cof(F):
    """The derivative of det F: columns f1 x f2, f2 x f0, f0 x f1."""
    f = F.unbind(-1)
    return torch.stack([_cross(f[1], f[2]), _cross(f[2], f[0]), _cross(f[0], f[1])], -1)


def _dcof(F, G):
    f, g = F.unbind(-1), G.unbind(-1)
    return torch.stack([_cross(g[i], f[j]) + _cross(f[i], g[j]) for i, j in ((1, 2), (2, 0), (0, 1))], -1)


def _axial(K):
    return torch.stack([K[:, 2, 1] - K[:, 1, 2], K[:, 0, 2] - K[:, 2, 0], K[:, 1, 0] - K[:, 0, 1]], -1)


def _skew(b):
    z = torch.zeros_like(b[:, 0])
    return torch.stack([z, -b[:, 2], b[:, 1], b[:, 2], z, -b[:, 0], -b[:, 1], b[:, 0], z], -1).reshape(-1, 3, 3)


def _on_segment(q, a, b):
    ab = b - a
    L2 = _dot(ab, ab)
    u = torch.where(L2 > 0, _dot(q - a, ab) / L2.clamp_min(1e-300), torch.zeros_like(L2)).clamp(0.0, 1.0)
    r = q - a - u[:, None] * ab
    return _dot(r, r), u


def _pick(best, c, d2, cand):
    m = d2 < best
    return torch.where(m, d2, best), torch.where(m[:, None], torch.stack(cand, -1), c)


def _pt(x, v):
    """Closest-point coefficients of point v0 and triangle v1 v2 v3 (first of the clamped edges wins ties)."""
    x0, x1, x2, x3 = (x[v[:, k]] for k in range(4))
    r, e1, e2 = x0 - x1, x2 - x1, x3 - x1
    a, b, q = _dot(e1, e1), _dot(e1, e2), _dot(e2, e2)
    det = a * q - b * b
    s, t = _dot(r, e1), _dot(r, e2)
    be, ga = (q * s - b * t) / det.clamp_min(1e-300), (a * t - b * s) / det.clamp_min(1e-300)
    inside = (det > 1e-12 * a * q) & (be >= 0) & (ga >= 0) & (be + ga <= 1)
    one, zero = torch.ones_like(be), torch.zeros_like(be)
    best, u = _on_segment(x0, x1, x2)
    c = torch.stack([one, u - 1, -u, zero], -1)
    d2, u = _on_segment(x0, x2, x3)
    best, c = _pick(best, c, d2, [one, zero, u - 1, -u])
    d2, u = _on_segment(x0, x3, x1)
    best, c = _pick(best, c, d2, [one, -u, zero, u - 1])
    return torch.where(inside[:, None], torch.stack([one, be + ga - 1, -be, -ga], -1), c)


def _ee(x, v):
    x0, x1, x2, x3 = (x[v[:, k]] for k in range(4))
    e0, e1, r = x1 - x0, x3 - x2, x0 - x2
    a, b, q, d, e = _dot(e0, e0), _dot(e0, e1), _dot(e1, e1), _dot(e0, r), _dot(e1, r)
    det = a * q - b * b
    s, t = (b * e - q * d) / det.clamp_min(1e-300), (a * e - b * d) / det.clamp_min(1e-300)
    inside = (det > 1e-12 * a * q) & (s >= 0) & (s <= 1) & (t >= 0) & (t <= 1)
    one, zero = torch.ones_like(s), torch.zeros_like(s)
    best, u = _on_segment(x0, x2, x3)
    c = torch.stack([one, zero, u - 1, -u], -1)
    d2, u = _on_segment(x1, x2, x3)
    best, c = _pick(best, c, d2, [zero, one, u - 1, -u])
    d2, u = _on_segment(x2, x0, x1)
    best, c = _pick(best, c, d2, [1 - u, u, -one, zero])
    d2, u = _on_segment(x3, x0, x1)
    best, c = _pick(best, c, d2, [1 - u, u, zero, -one])
    return torch.where(inside[:, None], torch.stack([1 - s, s, t - 1, -t], -1), c)


class _Exact:
    """The incremental potential of a scene in float64 on the GPU: E(x) = 1/2 |x - xt|_M^2 + h^2 Psi(x) + kappa sum b(d),
    with its gradient, diagonal, curvature and Hessian products (closest points frozen), and the solver's iteration."""

    def __init__(self, sc, case, youngs=None):
        self.sc, self.case, self.dev = sc, case, "cuda"

        def t(v, k=torch.float64):
            return torch.as_tensor(np.ascontiguousarray(v), dtype=k, device=self.dev)

        self.t = t
        X, self.tet = t(sc.rest_x), t(sc.tets, torch.int64)
        D = (X[self.tet[:, 1:]] - X[self.tet[:, :1]]).transpose(1, 2)
        self.W = torch.linalg.inv(D)
        self.hv = sc.dt ** 2 * torch.linalg.det(D) / 6.0
        E = sc.youngs_per_tet if sc.youngs_per_tet is not None else np.full(sc.n_tets, sc.youngs)
        E = t(E) if youngs is None else youngs
        self.mu = E / (2 * (1 + sc.poisson))
        self.lam = E * sc.poisson / ((1 + sc.poisson) * (1 - 2 * sc.poisson))
        self.w = torch.cat([-self.W.sum(1, keepdim=True), self.W], 1)      # [T, corner, 3]
        self.mass = t(_lumped(sc))
        self.free = t(np.ones(sc.n_verts) if sc.fixed is None else 1 - sc.fixed)[:, None]
        self.plane = None if sc.plane is None else (t(sc.plane[0]), sc.plane[1])
        # surface: faces of one tet, their edges and vertices; the object of each is the bar, block or scene it is in
        f = sc.tets[:, [[1, 2, 3], [0, 3, 2], [0, 1, 3], [0, 2, 1]]].reshape(-1, 3)
        s, n = np.sort(f, 1).astype(np.int64), sc.n_verts
        _, first, times = np.unique((s[:, 0] * n + s[:, 1]) * n + s[:, 2], return_index=True, return_counts=True)
        f = f[first[times == 1]]
        s = np.sort(f[:, [[0, 1], [1, 2], [2, 0]]].reshape(-1, 2), 1).astype(np.int64)
        e = np.unique(s[:, 0] * n + s[:, 1])
        self.tri, self.edge, self.pts = t(f, torch.int64), t(np.stack([e // n, e % n], 1), torch.int64), t(np.unique(f), torch.int64)
        g = np.zeros(sc.n_verts) if sc.scene_of_vert is None else sc.scene_of_vert
        self.grp = t(g, torch.int64)
        self.ng = int(np.max(g)) + 1
        self.apart = sc.scene_of_vert is not None and not case["split"]    # no pairs between two scenes
        self.pairs_at, self.reach = None, 12.0 * sc.dhat

    def _near(self, x, a, b):
        """Index pairs (i, j) of primitives a and b whose boxes are within reach of each other."""
        lo_a, hi_a = x[a].amin(1).float(), x[a].amax(1).float()
        lo_b, hi_b = x[b].amin(1).float(), x[b].amax(1).float()
        r, got = 1.01 * self.reach, []
        step = max(1, 60_000_000 // max(1, len(b)))
        for s in range(0, len(a), step):
            m = None
            for k in range(3):
                n = (lo_a[s:s + step, k, None] - r <= hi_b[None, :, k]) & (lo_b[None, :, k] - r <= hi_a[s:s + step, k, None])
                m = n if m is None else m.logical_and_(n)
            ij = m.nonzero()
            ij[:, 0] += s
            got.append(ij)
        return torch.cat(got)

    def _candidates(self, x):
        """All surface pairs that can come within dhat before some vertex has moved by half the rest of the reach."""
        if self.pairs_at is not None and float((x - self.pairs_at).norm(dim=1).max()) < 0.49 * (self.reach - self.sc.dhat):
            return
        self.pairs_at = x.clone()
        ij = self._near(x, self.pts[:, None], self.tri)
        v, f = self.pts[ij[:, 0]], self.tri[ij[:, 1]]
        keep = (f != v[:, None]).all(1)
        pt = torch.cat([v[:, None], f], 1)[keep]
        ij = self._near(x, self.edge, self.edge)
        ij = ij[ij[:, 0] < ij[:, 1]]
        a, b = self.edge[ij[:, 0]], self.edge[ij[:, 1]]
        ee = torch.cat([a, b], 1)[(a[:, :, None] != b[:, None, :]).flatten(1).all(1)]
        if self.apart:
            pt, ee = pt[self.grp[pt[:, 0]] == self.grp[pt[:, 1]]], ee[self.grp[ee[:, 0]] == self.grp[ee[:, 2]]]
        self.cand = (pt, ee)

    def contacts(self, x):
        self._candidates(x)
        pt, ee = self.cand
        self.v = torch.cat([pt, ee])
        c = torch.cat([_pt(x, pt), _ee(x, ee)])
        t = (c[:, :, None] * x[self.v]).sum(1)
        d = t.norm(dim=1)
        m = d < self.sc.dhat
        self.v, self.c, self.tt, d = self.v[m], c[m], t[m], d[m]
        b1, b2 = self._barrier(d)
        self.A, self.Bc = self.sc.kappa * (b2 / d ** 2 - b1 / d ** 3), self.sc.kappa * b1 / d
        self.d = d
        if self.plane is not None:
            n, o = self.plane
            d = x @ n - o
            b1, b2 = self._barrier(torch.where(d < self.sc.dhat, d, torch.full_like(d, self.sc.dhat)))
            self.k1, self.k2, self.dp = self.sc.kappa * b1, self.sc.kappa * b2, d

    def _barrier(self, d):
        h = self.sc.dhat
        r, L = d - h, torch.log1p((d - h) / h)
        return -2 * r * L - r * r / d, -2 * L - 4 * r / d + (r / d) ** 2

    def element(self, x):
        """Deformation gradients and the density's derivatives at x."""
        self.F = (x[self.tet[:, 1:]] - x[self.tet[:, :1]]).transpose(1, 2) @ self.W
        self.cof = _cof(self.F)
        J = (self.F[:, :, 0] * self.cof[:, :, 0]).sum(1)
        self.J, mu, lam, m = J, self.mu, self.lam, self.case["model"]
        self.p1, self.c2 = torch.zeros_like(mu), mu.clone()
        if m == "nh":
            L = J.log()
            self.p3, self.p33 = (lam * L - mu) / J, (mu + lam * (1 - L)) / J ** 2
        elif m == "snh":
            self.p3, self.p33 = lam * (J - 1) - mu, lam
        else:
            if m == "arap":
                lam = torch.zeros_like(lam)
            self.p1, self.c2, self.p3, self.p33 = -2 * mu, 2 * mu, lam * (J - 1), lam
            R = self.F                                    # the polar factor by Newton's iteration
            for _ in range(30):
                C = _cof(R)
                inv_t = C / (R[:, :, 0] * C[:, :, 0]).sum(1)[:, None, None]
                R = 0.5 * (R + inv_t)
            self.R = R
            U = R.transpose(1, 2) @ self.F
            self.trU = U.diagonal(dim1=1, dim2=2).sum(1)
            self.Mi = torch.linalg.inv(self.trU[:, None, None] * torch.eye(3, dtype=U.dtype, device=U.device) - 0.5 * (U + U.transpose(1, 2)))
        self.rotated = m in ("fcr", "arap")

    def _scatter(self, idx, val, n):
        out = torch.zeros((n,) + val.shape[1:], dtype=val.dtype, device=self.dev)
        return out.index_add_(0, idx, val)

    def stress(self):
        P = self.c2[:, None, None] * self.F + self.p3[:, None, None] * self.cof
        if self.rotated:
            P = P + self.p1[:, None, None] * self.R
        return P

    def gradient(self, x, xt, mass):
        nv = len(x)
        self.element(x)
        self.contacts(x)
        g, dg = mass[:, None] * (x - xt), mass[:, None].expand(-1, 3).clone()
        f = torch.einsum("tab,tib->tia", self.hv[:, None, None] * self.stress(), self.w)
        cw = torch.einsum("tab,tib->tia", self.cof, self.w)
        h = self.c2[:, None, None] * (self.w ** 2).sum(-1, keepdim=True) + self.p33[:, None, None] * cw ** 2
        if self.rotated:
            for i in range(4):
                for a in range(3):
                    ax = _axial(self.R[:, a, :, None] * self.w[:, i, None, :])
                    h[:, i, a] += self.p1 * torch.einsum("ta,tab,tb->t", ax, self.Mi, ax)
        g = g + self._scatter(self.tet.reshape(-1), f.reshape(-1, 3), nv)
        dg = dg + self._scatter(self.tet.reshape(-1), (self.hv[:, None, None] * h).reshape(-1, 3), nv)
        ct = self.c[:, :, None] * self.tt[:, None, :]
        g = g + self._scatter(self.v.reshape(-1), (self.Bc[:, None, None] * ct).reshape(-1, 3), nv)
        dg = dg + self._scatter(self.v.reshape(-1), (self.A[:, None, None] * ct ** 2 + (self.Bc[:, None] * self.c ** 2)[:, :, None]).reshape(-1, 3), nv)
        if self.plane is not None:
            n = self.plane[0]
            g, dg = g + self.k1[:, None] * n, dg + self.k2[:, None] * n ** 2
        return g, dg

    def energy(self, x, xt, mass):
        self.element(x)
        self.contacts(x)
        I2, J, mu, lam = (self.F ** 2).sum((1, 2)), self.J, self.mu, self.lam
        m = self.case["model"]
        if m == "nh":
            psi = mu / 2 * (I2 - 3) - mu * J.log() + lam / 2 * J.log() ** 2
        elif m == "snh":
            psi = mu / 2 * (I2 - 3) - mu * (J - 1) + lam / 2 * (J - 1) ** 2
        else:
            psi = mu * (I2 - 2 * self.trU + 3) + (lam / 2 * (J - 1) ** 2 if m == "fcr" else 0)
        h = self.sc.dhat

        def b(d):
            return -(d - h) ** 2 * torch.log1p((d - h) / h)

        plane = 0.0 if self.plane is None else float(self.sc.kappa * b(self.dp[self.dp < h]).sum())
        return [float(0.5 * (mass[:, None] * (x - xt) ** 2).sum()), float((self.hv * psi).sum()),
                float(self.sc.kappa * b(self.d).sum()), plane]

    def curvature(self, p, mass):
        """p^T H p at the last gradient, per group, the other groups' entries of p taken as zero."""
        q = self._scatter(self.grp, mass * _dot(p, p), self.ng)
        if self.plane is not None:
            q = q + self._scatter(self.grp, self.k2 * (p @ self.plane[0]) ** 2, self.ng)
        dF = (p[self.tet[:, 1:]] - p[self.tet[:, :1]]).transpose(1, 2) @ self.W
        e = self.c2 * (dF ** 2).sum((1, 2)) + self.p33 * (self.cof * dF).sum((1, 2)) ** 2
        e = e + self.p3 * (_dcof(self.F, dF) * dF).sum((1, 2))
        if self.rotated:
            ax = _axial(self.R.transpose(1, 2) @ dF)
            e = e + self.p1 * torch.einsum("ta,tab,tb->t", ax, self.Mi, ax)
        q = q + self._scatter(self.grp[self.tet[:, 0]], self.hv * e, self.ng)
        if len(self.v):
            gv, pv = self.grp[self.v], p[self.v] * self.c[:, :, None]
            for k in (0, 3):                               # the first and the last vertex are of the two primitives
                w = (pv * (gv == gv[:, k:k + 1])[:, :, None]).sum(1)
                one = (gv[:, 0] == gv[:, 3]).to(w.dtype) * 0.5 + (gv[:, 0] != gv[:, 3]).to(w.dtype)
                q = q + self._scatter(gv[:, k], one * (self.A * _dot(w, self.tt) ** 2 + self.Bc * _dot(w, w)), self.ng)
        return q

    def product(self, p, mass):
        """H p at the last gradient."""
        nv = len(p)
        dF = (p[self.tet[:, 1:]] - p[self.tet[:, :1]]).transpose(1, 2) @ self.W
        dP = self.c2[:, None, None] * dF + self.p3[:, None, None] * _dcof(self.F, dF)
        dP = dP + (self.p33 * (self.cof * dF).sum((1, 2)))[:, None, None] * self.cof
        if self.rotated:
            b = torch.einsum("tab,tb->ta", self.Mi, _axial(self.R.transpose(1, 2) @ dF))
            dP = dP + self.p1[:, None, None] * (self.R @ _skew(b))
        out = mass[:, None] * p
        f = torch.einsum("tab,tib->tia", self.hv[:, None, None] * dP, self.w)
        out = out + self._scatter(self.tet.reshape(-1), f.reshape(-1, 3), nv)
        w = (self.c[:, :, None] * p[self.v]).sum(1)
        f = (self.A * _dot(w, self.tt))[:, None] * self.tt + self.Bc[:, None] * w
        out = out + self._scatter(self.v.reshape(-1), (self.c[:, :, None] * f[:, None, :]).reshape(-1, 3), nv)
        if self.plane is not None:
            out = out + (self.k2 * (p @ self.plane[0]))[:, None] * self.plane[0]
        return out

    def jacobi(self, dg):
        m = self.mass[:, None]
        return self.free / torch.where(dg > 1e-3 * m, dg, m.expand_as(dg))

    def step(self, x, v, targets, iters):
        sc = self.sc
        x0, xt = x, x + sc.dt * v + sc.dt ** 2 * self.t(sc.gravity)
        if targets is not None:
            f = self.free[:, 0] == 0
            x = x.clone()
            x[f] = self.t(targets)
            xt = torch.where(f[:, None], x, xt)
        mass = self.mass * self.free[:, 0]
        p = g0 = gPg0 = None
        each = lambda a, b: self._scatter(self.grp, _dot(a, b), self.ng)  # noqa: E731
        for k in range(iters):
            g, dg = self.gradient(x, xt, mass)
            g = g * self.free
            P = self.jacobi(dg)
            if k == 0:
                beta = torch.zeros(self.ng, dtype=x.dtype, device=self.dev)
                gPg, p = each(g, P * g), torch.zeros_like(x)
            else:
                y, gPg = g - g0, each(g, P * g)
                if self.case["beta"] == "pr":
                    beta = torch.where(gPg0 > 0, each(g, P * y) / gPg0, torch.zeros_like(gPg0)).clamp_min(0.0)
                else:
                    yp = each(y, p)
                    beta = torch.where(yp.abs() < 1e-30, torch.zeros_like(yp), each(g, P * y) / yp - each(y, P * y) / yp * each(p, g) / yp)
                beta = torch.where(-gPg + beta * each(g, p) >= 0, torch.zeros_like(beta), beta)
            p = -P * g + beta[self.grp][:, None] * p
            gp, pHp = each(g, p), self.curvature(p, mass)
            big = torch.zeros(self.ng, dtype=x.dtype, device=self.dev).scatter_reduce_(0, self.grp, p.norm(dim=1), "amax")
            cap = torch.where(big > 0, sc.dhat / (2 * big), torch.zeros_like(big))
            newton = -gp / pHp
            al = torch.where((pHp > 0) & newton.isfinite(), torch.minimum(newton, cap), cap)
            x = x + al[self.grp][:, None] * p
            g0, gPg0 = g, gPg
        return x, (x - x0) / sc.dt

    def adjoint(self, x, ax, av):
        """lambda from H lambda = ax + av / h by conjugate gradients to 1e-13; the step's three gradients."""
        sc, m = self.sc, self.mass
        _, dg = self.gradient(x, x, m)
        P = self.jacobi(dg)
        b = ax + av / sc.dt
        lam, r = torch.zeros_like(b), b.clone()
        z = P * r
        p, rz = z, (r * z).sum()
        for _ in range(4000):
            q = self.product(p, m)
            a = rz / (p * q).sum()
            lam, r = lam + a * p, r - a * q
            if float(r.norm()) <= 1e-13 * float(b.norm()):
                break
            z = P * r
            new = (r * z).sum()
            p, rz = z + new / rz * p, new
        ml = m[:, None] * lam
        E = self.mu * (2 * (1 + sc.poisson))
        f = torch.einsum("tab,tib->tia", (self.hv / E)[:, None, None] * self.stress(), self.w)
        return ml - av / sc.dt, sc.dt * ml, -(f * lam[self.tet]).sum((1, 2))


def exact(case, seed):
    sc, targets, rng = _inputs(case, seed)
    p, xt, ax, av = _vectors(case, sc, rng)
    kind = case["kind"]
    if kind == "train":
        E = torch.as_tensor(sc.youngs * (1.0 + 0.2 * rng.random(sc.n_tets)), device="cuda")
        goal = sc.x0 + 2.0 * sc.dt * sc.v0 + 0.01 * rng.normal(size=3)
        X = _Exact(sc, case, E)
        goal, xs, v = X.t(goal), [X.t(sc.x0)], X.t(sc.v0)
        for _ in range(2):
            x, v = X.step(xs[-1], v, None, 600)
            xs.append(x)
        ax, av, dE = 2.0 * (xs[-1] - goal), torch.zeros_like(goal), torch.zeros_like(E)
        for x in (xs[2], xs[1]):
            ax, av, d = X.adjoint(x, ax, av)
            dE = dE + d
        return xs[-1], dE, av
    X = _Exact(sc, case)
    x, p, xt, m = X.t(sc.x0), X.t(p), X.t(xt), X.mass
    if kind == "step":
        x, v = X.step(x, X.t(sc.v0), targets, case["iters"])
        # the velocity of a float step is the difference of two positions over dt: what is left of its digits after
        # the iterations' growth of rounding varies with the order of the atomic sums, and measures that alone
        return x, (v if case["dtype"] == "f64" else None)
    if kind == "adjoint":
        return X.adjoint(x, X.t(ax), X.t(av))
    if kind == "energy":
        parts = X.energy(x, xt, m)
        return sum(parts), np.array(parts)
    if kind == "noalloc":                                  # inertia and elasticity alone
        X.plane, X.v = None, ()
        X.element(x)
        return X.curvature(p, m)
    g, dg = X.gradient(x, xt, m)
    if kind == "gradient":
        return g.cpu().numpy(), dg.cpu().numpy()
    if kind == "hvp":
        return X.product(p, m)
    return float(X.curvature(p, m).sum())
