"""The gradient pass passes over candidates that cannot have come within dhat since the candidate build (their distance there,
less twice the largest displacement since).  A time step in one launch, which does so, against the same step one iteration
per launch, which cannot know the displacement and looks at every candidate: the same active pairs at every iteration and
the same positions, on blocks that fall onto one another with the slack r from small (many builds) to large (none)."""
import numpy as np
import pytest

from paper_2405_08001_gb300 import scenes as S
from test_gpu_parity import B  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [(0, 1e-9), (1, 1e-3)])   # rounding grows by up to 1e4 over these iterations
@pytest.mark.parametrize("pad", [0.5, 2.0, 8.0])
@pytest.mark.parametrize("make", [lambda: S.two_blocks(0, gap=0.9, speed=0.4), lambda: S.two_blocks(3, gap=1.3, speed=1.0),
                                  lambda: S.pile(3, cells=(5, 4, 9), size=(0.05, 0.04, 0.09), gap=0.98, iters=12)])
def test_one_launch_equals_single_iterations(B, make, pad, prec, tol):  # noqa: F811
    sc = make()
    n = 10
    a, b = (B.Sim(sc, precision=prec, iters=n, pad_r=pad * sc.dhat) for _ in range(2))
    a.step(1)
    B.sim_begin_step(b.h)
    active = []
    for _ in range(n):
        B.sim_iterate(b.h, 1)
        active.append(B.sim_get_iterate(b.h)[5]["n_active"])
    B.sim_end_step(b.h)
    xa, xb = a.state()[0], b.state()[0]
    trace = B.sim_get_trace(a.h)
    assert max(active) > 0
    assert trace[:, B.TRACE_COLUMNS.index("n_active")].astype(int).tolist() == active
    assert np.abs(xa - xb).max() <= tol * np.abs(xb - sc.x0).max()
    a.close()
    b.close()


def close_pairs(ratio, kind, rng, n, dhat=1e-3):
    """n pairs of separate tets that meet, less than dhat apart, at two nearly parallel edges (kind "ee") or where a vertex of
    one stands over a sliver face of the other ("pt"): sin^2 of the angle 1e-5 to 1.2e-5, where a float's closest points come
    from a determinant of a hundred roundings; edges of up to ratio dhat, and no larger extent than theirs."""
    L = ratio * dhat
    X, T = [], []
    for k in range(n):
        th, d, l2 = np.sqrt(1e-5 * 1.2 ** rng.uniform()), rng.uniform(0.8, 0.98) * dhat, L * rng.uniform(0.5, 1.0)
        u = np.array([np.cos(th), np.sin(th), 0.0])
        if kind == "ee":      # edges along x and u, crossing at c and c2 of their lengths
            c, c2 = rng.uniform(0.05, 0.95, 2)
            a = np.array([[-c * L, 0, 0], [(1 - c) * L, 0, 0], [(0.5 - c) * L, -0.2 * L, -0.3 * L], [(0.5 - c) * L, 0.2 * L, -0.3 * L]])
            m = (0.5 - c2) * l2 * u
            b = np.array([-c2 * l2 * u, (1 - c2) * l2 * u, m + [0, -0.2 * L, 0.3 * L], m + [0, 0.2 * L, 0.3 * L]]) + [0, 0, d]
        else:                 # a point over the inside of the face 0, L x, l2 u
            f = np.array([[0, 0, 0], [L, 0, 0], l2 * u])
            q = rng.dirichlet(np.ones(3)) @ f + [0, 0, d]
            a = np.concatenate([f, [[0.5 * L, 0.1 * L, -0.3 * L]]])
            b = q + np.array([[0, 0, 0], [0.2 * L, 0, 0.3 * L], [-0.1 * L, 0.2 * L, 0.3 * L], [-0.1 * L, -0.2 * L, 0.3 * L]])
        R = S.random_rotation(rng)
        o = 4 * L * np.array([k % 128, k // 128, 0])
        for t in (a, b):
            if np.linalg.det(t[1:] - t[0]) < 0:
                t = t[[0, 2, 1, 3]]
            X.append(t @ R.T + o)
            T.append(np.arange(4) + 4 * len(T))
    X = np.ascontiguousarray(np.concatenate(X))
    return S.Scene(name="close_pairs", rest_x=X, tets=np.array(T, np.int32), x0=X, v0=np.zeros_like(X), youngs=1e5, poisson=0.4,
                   density=1000.0, dt=1.0 / 60.0, dhat=dhat, kappa=1e4, iters=1, steps=1)


@pytest.mark.parametrize("kind", ["ee", "pt"])
@pytest.mark.parametrize("ratio", [50, 100])     # (beyond, the list itself, by the float distance, depends on the edges' order)
def test_nearly_parallel_pairs_are_not_passed_over(B, ratio, kind):  # noqa: F811
    """The same on nearly parallel edges and sliver faces that are long for dhat, whose float distance at the build is far
    above the true one for some: the first iteration of a whole step finds the pairs that a single iteration finds.  (FP64:
    the FP32 form's own float filter depends on which edge of a pair comes first.)"""
    sc = close_pairs(ratio, kind, np.random.default_rng(ratio), 16384)
    a, b = (B.Sim(sc, precision=0) for _ in range(2))
    a.step(1)
    B.sim_begin_step(b.h)
    B.sim_iterate(b.h, 1)
    n = B.sim_get_iterate(b.h)[5]["n_active"]
    assert n >= 16000
    assert int(B.sim_get_trace(a.h)[0, B.TRACE_COLUMNS.index("n_active")]) == n
    a.close()
    b.close()


@pytest.mark.parametrize("far", [150.0, 1000.0, 5000.0])
def test_fp32_far_from_the_origin(B, far):  # noqa: F811
    """The FP32 form measures displacements between float heads, whose rounding grows with the distance from the origin.  Two
    tets there come 0.84 units of the heads' last place closer and within dhat, each by less than half a unit, so that
    no head moves: the pair that a single iteration finds is found in a whole step.  (No stiffness: the first iteration
    ends at x~.)"""
    u = float(np.spacing(np.float32(far)))
    d0 = round(1e-3 / u) * u
    dhat = d0 - 0.6 * u
    a = 0.1 * np.array([[0, 0, 0], [0.1, 0, 0], [0, 0.1, 0], [0.03, 0.03, -0.1]])
    b = 0.1 * np.array([[0.03, 0.03, 0], [0.13, 0.03, 0.1], [0.03, 0.13, 0.1], [-0.07, -0.07, 0.1]])
    b[:, 2] += d0
    X = np.concatenate([a, b]) + [0, 0, far]
    X[:, 2] = np.round(X[:, 2] / u) * u
    v = np.zeros_like(X)
    v[:4, 2], v[4:, 2] = 0.42 * u * 60, -0.42 * u * 60
    T = np.array([[0, 2, 1, 3], [4, 5, 6, 7]], np.int32)
    for t in T:
        if np.linalg.det(X[t[1:]] - X[t[0]]) < 0:
            t[[1, 2]] = t[[2, 1]]
    sc = S.Scene(name="far", rest_x=X, tets=T, x0=X, v0=v, youngs=0.0, poisson=0.4, density=1000.0, dt=1.0 / 60.0, dhat=dhat, kappa=1e4,
                 iters=3, steps=1)
    s, w = (B.Sim(sc, precision=1, pad_r=2 * dhat) for _ in range(2))
    B.sim_begin_step(s.h)
    active = []
    for _ in range(sc.iters):
        B.sim_iterate(s.h, 1)
        active.append(B.sim_get_iterate(s.h)[5]["n_active"])
    assert active[0] == 0 and max(active) > 0, active
    w.step(1)
    assert B.sim_get_trace(w.h)[:, B.TRACE_COLUMNS.index("n_active")].astype(int).tolist() == active
    s.close()
    w.close()


def test_a_scene_near_the_grids_limit(B):  # noqa: F811
    """Cells are numbered up to 2^20 from the origin.  A tet so far out that the triangles' cells are within that and the
    edges' smaller ones would not be: the step runs."""
    X = np.array([[0.0, 0.0, 0.0], [1.0, 0.0, 0.0], [0.0, 1.0, 0.0], [0.0, 0.0, 1.0]])
    x0 = X + np.array([3.2e6, 0.0, 0.0])
    sc = S.Scene(name="far", rest_x=X, tets=np.array([[0, 1, 2, 3]], np.int32), x0=x0, v0=np.zeros_like(X), youngs=1e3, poisson=0.4,
                 density=1000.0, dt=1.0 / 60.0, dhat=1.0, kappa=1e4, iters=2)
    sim = B.Sim(sc, precision=0, pad_r=1.0)
    sim.step(1)
    assert np.abs(sim.state()[0] - x0).max() < 1e-6
    sim.close()


def test_fp32_pairs_below_the_line_are_evaluated_in_double(B):  # noqa: F811
    """Below 1e-3 dhat the FP32 form evaluates a pair in double (n_near_fp64 counts them): also where the float
    filter's distance lies above the line and the float-float one below.  Crossed edges 1e-6 to 1e-2 of the line below it."""
    rng = np.random.default_rng(31)
    dhat, L, X, T = 1e-3, 0.1, [], []
    for k in range(512):
        f = 1.0 - 10.0 ** rng.uniform(-6, -2)      # (1e-6 of the line is 1e-12 m; x is rounded to 1e-15)
        th = rng.uniform(0.3, 1.2)
        u = np.array([np.cos(th), np.sin(th), 0.0])
        a = np.array([[-0.4 * L, 0, 0], [0.6 * L, 0, 0], [0.1 * L, -0.2 * L, -0.3 * L], [0.1 * L, 0.2 * L, -0.3 * L]])
        b = np.array([-0.5 * L * u, 0.5 * L * u, [0, -0.2 * L, 0.3 * L], [0, 0.2 * L, 0.3 * L]]) + [0, 0, 1e-3 * f * dhat]
        R, o = S.random_rotation(rng), 0.4 * np.array([k % 32, k // 32, 0])
        for t in (a, b):
            if np.linalg.det(t[1:] - t[0]) < 0:
                t = t[[0, 2, 1, 3]]
            X.append(t @ R.T + o)
            T.append(np.arange(4) + 4 * len(T))
    X = np.ascontiguousarray(np.concatenate(X))
    sc = S.Scene(name="near", rest_x=X, tets=np.array(T, np.int32), x0=X, v0=np.zeros_like(X), youngs=1e5, poisson=0.4, density=1000.0,
                 dt=1.0 / 60.0, dhat=dhat, kappa=1e-3, iters=1, steps=1)
    sim = B.Sim(sc, precision=1)
    B.sim_eval_gradient(sim.h, X, X)
    assert sim.state()[2]["n_near_fp64"] == 512
    sim.close()


@pytest.mark.parametrize("prec", [0, 1])
def test_an_evaluation_at_nan_leaves_the_skip_as_it_was(B, prec):  # noqa: F811
    """An evaluation that fails on a non-finite position does not reach the next step's candidates."""
    sc = S.two_blocks(0)
    active = []
    for bad in (False, True):
        sim = B.Sim(sc, precision=prec, iters=4)
        if bad:
            x = sc.x0.copy()
            x[5] = np.nan
            with pytest.raises(B.SimError):
                B.sim_eval_gradient(sim.h, x, x)
        sim.step(1)
        active.append(B.sim_get_trace(sim.h)[:, B.TRACE_COLUMNS.index("n_active")].astype(int).tolist())
        sim.close()
    assert active[0] == active[1] and max(active[0]) > 0, active
