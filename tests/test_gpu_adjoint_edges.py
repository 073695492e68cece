"""The differentiation calls at the edges of what they accept."""
import dataclasses
import math

import numpy as np
import pytest

from paper_2405_08001_gb300 import scenes as S
from test_gpu_parity import B, O  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


def strained(cells, seed):
    sc = S.cube_drop(n=max(cells), cells=cells, drop=0.05)
    rng = np.random.default_rng(seed)
    c = sc.x0.mean(axis=0)
    A = np.array([[1.03, 0.02, 0.0], [0.0, 0.99, 0.015], [0.0, 0.0, 1.0]])
    return sc, (sc.x0 - c) @ A.T + c + 2e-5 * rng.normal(size=sc.x0.shape), rng


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("model", [0, 1, 2, 3])
@pytest.mark.parametrize("uniform", [False, True])
def test_zero_moduli(B, O, uniform, model, prec):  # noqa: F811
    """dL/dE_e of tets with E_e = 0 (some of them, or all by youngs = 0) is finite and equals the oracle's with a modulus
    of 1e-11 in their place (whose Hessian is about 1e-12 of the mass: lambda and the gradient change by no more than that).
    The FP32 product's error is below 1e-5 (its hvp tests) and H's condition number here about 1e3."""
    sc, x, rng = strained((3, 3, 3), 7)
    E = np.full(sc.n_tets, 0.0 if uniform else 1e5)
    E[::3] = 0.0
    tiny = np.where(E == 0.0, 1e-11, E)
    if uniform:
        sim = B.Sim(dataclasses.replace(sc, youngs=0.0), precision=prec, model=model)
    else:
        sim = B.Sim(dataclasses.replace(sc, youngs=1.0, youngs_per_tet=E), precision=prec, model=model)
    o = O.Oracle.from_scene(dataclasses.replace(sc, youngs=1.0, youngs_per_tet=tiny), model=model)
    ax, av = rng.normal(size=x.shape), rng.normal(size=x.shape)
    dE, dEo = np.zeros(sc.n_tets), np.zeros(sc.n_tets)
    a, v, _, _ = B.sim_adjoint_step(sim.h, x, ax, av, dE=dE, tol=1e-13 if prec == 0 else 1e-9, max_iters=5000)
    ao, vo, _, _ = o.adjoint_step(x, ax, av, dE=dEo, tol=1e-13, max_iters=5000)
    assert np.isfinite(dE).all()
    tol = 1e-9 if prec == 0 else 1e-2
    for g, r in ((a, ao), (v, vo), (dE, dEo), (dE[::3], dEo[::3])):
        assert np.linalg.norm(g - r) <= tol * np.linalg.norm(r)
    sim.close()


# 432 tets: one cluster; 8,640: the whole grid in both precisions
@pytest.mark.parametrize("cells", [(3, 3, 8), (12, 12, 10)])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("model", [0, 2])
def test_kinematic_rows_and_columns_are_dropped(B, O, model, prec, cells):  # noqa: F811
    """H v and the reverse step on a bar whose two end caps are kinematic, against the oracle, which drops their rows and
    columns: their entries of H v are 0, their ax0 is -av1 / h and their av0 is 0, all exactly."""
    sc = S.twisted_bar(*cells)
    fx = sc.fixed.astype(bool)
    rng = np.random.default_rng(17)
    x = sc.x0 + 1e-4 * rng.normal(size=sc.x0.shape)
    sim = B.Sim(sc, precision=prec, model=model)
    o = O.Oracle.from_scene(sc, model=model)
    v = rng.normal(size=x.shape)
    hv, ref = B.sim_eval_hvp(sim.h, x, v), o.hvp(x, v)
    assert (hv[fx] == 0.0).all()
    assert np.linalg.norm(hv - ref) <= (1e-10 if prec == 0 else 1e-5) * np.linalg.norm(ref)
    ax, av = rng.normal(size=x.shape), 1e-2 * rng.normal(size=x.shape)
    dE, dEo = np.zeros(sc.n_tets), np.zeros(sc.n_tets)
    a, b, _, _ = B.sim_adjoint_step(sim.h, x, ax, av, dE=dE, tol=1e-13 if prec == 0 else 1e-9, max_iters=20000)
    ao, bo, _, _ = o.adjoint_step(x, ax, av, dE=dEo, tol=1e-13, max_iters=20000)
    assert (b[fx] == 0.0).all() and np.array_equal(a[fx], -av[fx] / sc.dt)
    tol = 1e-9 if prec == 0 else 1e-2       # FP32: the product's 1e-5 at most, times H's condition number of about 1e3
    for g, r in ((a, ao), (b, bo), (dE, dEo)):
        assert np.linalg.norm(g - r) <= tol * np.linalg.norm(r), np.linalg.norm(g - r) / np.linalg.norm(r)
    # the state's own flags are as they were: the next step holds the caps at their targets
    t = sc.targets(0)
    sim.step(1, t)
    assert np.abs(sim.state()[0][fx] - t).max() < 1e-12
    sim.close()


def free_bytes():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_hvp_needs_no_solver_memory(B):  # noqa: F811
    """The first sim_eval_hvp of a handle allocates two vectors of 32 bytes a vertex, and none of the reverse step's (160
    bytes a tet among them)."""
    sc, x, rng = strained((30, 30, 30), 3)
    v = rng.normal(size=x.shape)
    used = []
    for _ in range(2):                          # the first handle loads the kernels
        sim = B.Sim(sc, precision=0)
        f = free_bytes()
        B.sim_eval_hvp(sim.h, x, v)
        used.append(f - free_bytes())
        sim.close()
    assert used[1] <= 2 * 32 * sc.n_verts + (4 << 20), used   # and the driver's 2 MB pages


def test_reverse_step_without_room_for_the_record(B):  # noqa: F811
    """Where the device has no room for the tets' record (160 bytes each) the solve runs without it: the same result
    within the solver's tolerance, no SIM_ERR_OOM."""
    import torch
    sc, x, rng = strained((30, 30, 30), 5)      # 162,000 tets: 26 MB of record, 9 MB of vectors
    ax, av = rng.normal(size=x.shape), np.zeros_like(x)
    out = []
    for full in (False, True):
        sim = B.Sim(sc, precision=0)
        torch.cuda.empty_cache()
        hog = torch.empty(free_bytes() - (20 << 20), dtype=torch.uint8, device="cuda") if full else None
        a, v, it, res = B.sim_adjoint_step(sim.h, x, ax, av, tol=1e-11, max_iters=5000)
        assert res <= 1e-11
        out.append((a, v))
        del hog
        torch.cuda.empty_cache()
        sim.close()
    for p, q in zip(*out):
        assert np.linalg.norm(p - q) <= 1e-8 * np.linalg.norm(q)   # 1e-11 times the condition number of about 1e3


@pytest.mark.parametrize("cells", [(9, 11, 13), (20, 20, 20)])   # one cluster; the whole grid
def test_fp32_step_length_is_summed_in_double(B, O, cells):  # noqa: F811
    """One CG iteration: lambda = alpha P r with alpha = r.P r / p.H p.  H p is the FP32 form's (sim_eval_hvp), and alpha
    the quotient of sums in double over it, whatever the order: N u of a sum of N positive terms, 30,000 u < 1e-11.  The
    segmented scatter makes P the same from call to call."""
    sc, x, rng = strained(cells, 23)
    sim = B.Sim(sc, precision=1, scatter=B.SIM_SCATTER_SEGMENTED)
    _, d = B.sim_eval_gradient(sim.h, x, x)
    P = (np.float32(1.0) / d.astype(np.float32)).astype(np.float64)
    r = rng.normal(size=x.shape)
    p = P * r
    q = B.sim_eval_hvp(sim.h, x, p)
    alpha = math.fsum((r * p).ravel()) / math.fsum((p * q).ravel())
    _, av, it, _ = B.sim_adjoint_step(sim.h, x, r, np.zeros_like(r), tol=1e-30, max_iters=1)
    assert it == 1
    lam = av / (sc.dt * O.Oracle.from_scene(sc).mass()[:, None])
    got = np.median(lam / p)
    assert abs(got / alpha - 1.0) < 1e-11, got / alpha - 1.0
    sim.close()
