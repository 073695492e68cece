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
