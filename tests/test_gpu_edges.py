"""The element passes work on a tet's edge vectors Ds and on M = Dm^-1 Dm^-T, the FP64 form with a logarithm of its own.
Separate tets against the oracle, tet by tet: aspect ratios up to 1000, stretched and turned, with det F at the edges of
the logarithm's table (1, its first cells on both sides, the halves between cells, powers of two) and far out.

With u the unit roundoff, every entry is a sum of products of a few rounded factors, so its error is at most C u times
the sum of the products' magnitudes; C = 16 covers a chain's accumulated roundings and the oracle's own (a chain is about 30 operations,
half an ulp each), 4 times that the FP32 form, which has J as 1 + (J - 1) (J = 0.02 loses 1 / J).  A flat tet's
cofactors and determinant cancel, so their products' magnitudes count, not theirs, and J's error goes on into the terms that
depend on J.  The FP32 form sums with tails: there u = 2^-24 applies to the metric change G = Ds^T Ds - Dm^T Dm after the
cancellation, whose own error is below 2^-44 of its terms."""
import numpy as np
import pytest

from paper_2405_08001_gb300 import scenes as S
from test_gpu_parity import B, O  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu

J_EDGE = [1.0, 1 - 2.0**-9, 1 - 2.0**-9 - 1e-9, 1 + 2.0**-8, 1 + 2.0**-8 + 1e-9, 1 + 1e-7, 1 - 1e-7, 1 + 3.5 / 128,
          1 + 126.5 / 128, 0.5, 0.75, 2.0, 0.02, 40.0]
E, NU = 1e5, 0.4
MU, LAM = E / (2 * (1 + NU)), E * NU / ((1 + NU) * (1 - 2 * NU))


def cof(s):
    return np.stack([np.cross(s[:, 1], s[:, 2]), np.cross(s[:, 2], s[:, 0]), np.cross(s[:, 0], s[:, 1])], axis=1)


def separate_tets(aspect, rng):
    X, x = [], []
    for n, J in enumerate(J_EDGE):
        Dm = 0.01 * (np.eye(3) + 0.2 * rng.normal(size=(3, 3)))
        Dm[2] /= aspect                                                   # flat
        if np.linalg.det(Dm) < 0:
            Dm = Dm[:, [1, 0, 2]]
        Q = np.linalg.qr(rng.normal(size=(3, 3)))[0]
        Q *= np.sign(np.linalg.det(Q))
        st = np.exp(0.05 * rng.normal(size=3))
        F = Q @ np.diag(st * (J / st.prod()) ** (1 / 3)) if J != 1.0 else Q
        o = np.array([0.15 * (n % 4), 0.15 * (n // 4), 0.0])
        for out, D in ((X, Dm), (x, F @ Dm)):
            out.append(np.concatenate([[o], o + D.T]))
    X, x = (np.ascontiguousarray(np.concatenate(a)) for a in (X, x))
    T = np.arange(len(X), dtype=np.int32).reshape(-1, 4)
    return S.Scene(name="separate_tets", rest_x=X, tets=T, x0=x, v0=np.zeros_like(x), youngs=E, poisson=NU, density=1000.0,
                   dt=1.0 / 60.0, dhat=1e-6, kappa=1e4, iters=1, steps=1)


def magnitudes(sc, prec, dp):
    """Per tet: the sums of magnitudes for g, diag, p^T H p and H p of the displacement dp."""
    u = 2.0**-53 if prec == 0 else 2.0**-24
    out = []
    for t in sc.tets:
        Dm, s, d = ((a[t[1:]] - a[t[0]]).T for a in (sc.rest_x, sc.x0, dp))
        W = np.linalg.inv(Dm)
        M, c, iD = np.abs(W @ W.T), np.abs(cof(s)), np.linalg.det(W)
        hv, J = sc.dt**2 * np.linalg.det(Dm) / 6, np.linalg.det(s) * iD
        s0, s, d = s, np.abs(s), np.abs(d)
        ca = cof_mixed(s, s) / 2                    # the cofactors' products: their errors do not shrink with c
        rho = np.sum(s[0] * ca[0]) * iD / J         # det's: the relative error of J is rho u
        L = abs(np.log(J))
        k3, k3J = hv * iD * (LAM * L + MU) / J, hv * iD * (LAM * (2 + L) + MU) / J      # |Psi_3| and J |dPsi_3/dJ|
        k33 = hv * (iD / J) ** 2 * (MU + LAM * (1 + L))
        if prec == 0:
            g = hv * MU * s @ M + k3 * ca + k3J * rho * c
        else:
            G = np.abs(s0.T @ s0 - Dm.T @ Dm) + 2.0**-20 * s.T @ s
            g = hv * iD / J * (MU * ca @ G @ M + LAM * ((L + 2.0**-20 * rho) * ca))
        cs, cas = c.sum(axis=1), ca.sum(axis=1)     # x_0's weights are sums
        dg = hv * MU * 2 * M.sum() + k33 * (2 * cs * cas + (1 + 4 * rho) * cs**2).max()
        cd, cad, mx = np.sum(c * d), np.sum(ca * d), cof_mixed(s, d)
        h = hv * MU * d @ M + k33 * (ca * cd + c * cad + 4 * rho * c * cd) + (k3 + k3J * rho) * mx
        out.append((3 * g.max(), dg, np.sum(h * d), 3 * h.max()))
    return (16 if prec == 0 else 64) * u * np.array(out)


def cof_mixed(s, d):
    """entries of |d cof(s)[d]|: the cross products with one factor from each, magnitudes added"""
    def ax(a, b):
        return np.stack([a[1] * b[2] + a[2] * b[1], a[2] * b[0] + a[0] * b[2], a[0] * b[1] + a[1] * b[0]])
    return np.stack([ax(d[:, j], s[:, k]) + ax(s[:, j], d[:, k]) for j, k in ((1, 2), (2, 0), (0, 1))], axis=1)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("aspect", [1.0, 30.0, 1000.0])
def test_separate_tets(B, O, aspect, prec):  # noqa: F811
    rng = np.random.default_rng(int(aspect))
    sc = separate_tets(aspect, rng)
    o = O.Oracle.from_scene(sc)
    sim = B.Sim(sc, precision=prec)
    u = 2.0**-53 if prec == 0 else 2.0**-24
    x, p = sc.x0, 1e-3 * rng.normal(size=sc.x0.shape)
    tol = magnitudes(sc, prec, p)
    g, d = B.sim_eval_gradient(sim.h, x, x)
    go, do, na = o.grad_diag(x, x)
    assert na == 0
    hv, hvo = B.sim_eval_hvp(sim.h, x, p), o.hvp(x, p)
    for n, t in enumerate(sc.tets):
        J = J_EDGE[n]
        assert np.abs(g[t] - go[t]).max() <= tol[n, 0], (J, "g")
        assert (np.abs(d[t] - do[t]) <= tol[n, 1] + 8 * u * do[t]).all(), (J, "diag")
        assert np.abs(hv[t] - hvo[t]).max() <= tol[n, 3] + 8 * u * np.abs(hvo[t]).max(), (J, "hvp")
        q = np.zeros_like(p)
        q[t] = p[t]
        ref = o.pHp(x, q)
        assert abs(B.sim_eval_pHp(sim.h, x, q) - ref) <= tol[n, 2] + 8 * u * abs(ref), (J, "pHp")
    sim.close()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("aspect", [1.0, 30.0, 1000.0])
def test_flat_tets_along_smooth_directions(B, O, aspect, prec):  # noqa: F811
    """p^T H p of flat tets along p = A X, whose dF = A does not grow with the aspect ratio: forming dF from
    the edges costs u times the aspect ratio, and no more than four times that may go into the sum of the terms' magnitudes.
    (On M = Dm^-1 Dm^-T, whose entries are the ratio's square, it costs u times that.)"""
    for seed in range(4):
        rng = np.random.default_rng(10 * int(aspect) + seed)
        sc = separate_tets(aspect, rng)
        o = O.Oracle.from_scene(sc)
        sim = B.Sim(sc, precision=prec)
        u = 2.0**-53 if prec == 0 else 2.0**-24
        for n, t in enumerate(sc.tets):
            J = J_EDGE[n]
            if not 0.4 < J < 2.1:
                continue
            Dm = (sc.rest_x[t[1:]] - sc.rest_x[t[0]]).T
            F = (sc.x0[t[1:]] - sc.x0[t[0]]).T @ np.linalg.inv(Dm)
            A = rng.normal(size=(3, 3))
            p = np.zeros_like(sc.x0)
            p[t] = (sc.rest_x[t] - sc.rest_x[t].mean(axis=0)) @ A.T
            hv, L, a2, f = sc.dt**2 * np.linalg.det(Dm) / 6, abs(np.log(J)), np.sum(A * A), np.linalg.norm(F)
            scale = hv * a2 * (MU + (MU + LAM * (1 + L)) / J**2 * f**4 + (LAM * L + MU) / J * 2 * f)
            scale += 1000.0 * np.linalg.det(Dm) / 24 * np.sum(p * p)
            err = abs(B.sim_eval_pHp(sim.h, sc.x0, p) - o.pHp(sc.x0, p))
            assert err <= 4 * aspect * u * scale, (J, err / (aspect * u * scale))
        sim.close()
