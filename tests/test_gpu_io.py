"""State and evaluation arrays in host or device memory: the values go through one kernel each way (on host arrays by way
of a staging buffer), so the numbers are the same, and a part that is not given stays as it is."""
import numpy as np
import pytest
import torch

from paper_2405_08001_gb300 import scenes as S
from test_gpu_parity import B  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("cells", [(1, 1, 1), (7, 5, 9)])   # 8 vertices; 480, no multiple of a block
def test_host_and_device_arrays(B, cells, prec):  # noqa: F811
    sc = S.cube_drop(n=max(cells), cells=cells, drop=0.01)
    rng = np.random.default_rng(5)
    x, v, p = (a + 1e-4 * rng.normal(size=sc.x0.shape) for a in (sc.x0, sc.v0, 0.0 * sc.x0))
    dx, dv, dp = (torch.from_numpy(a).cuda() for a in (x, v, p))
    out = []
    for sx, sv, sp in ((x, v, p), (dx, dv, dp)):
        sim = B.Sim(sc, precision=prec)
        B.sim_set_state(sim.h, sx, None)                       # v as it was
        x0, v0, _ = B.sim_get_state(sim.h)
        assert np.array_equal(x0, x) and np.array_equal(v0, sc.v0)
        B.sim_set_state(sim.h, None, sv)
        xo, vo = (torch.zeros(sc.x0.shape, dtype=torch.float64, device="cuda") for _ in range(2))
        B.sim_get_state(sim.h, xo, vo)
        x1, v1, _ = B.sim_get_state(sim.h)
        assert np.array_equal(x1, x) and np.array_equal(v1, v)
        assert np.array_equal(xo.cpu().numpy(), x) and np.array_equal(vo.cpu().numpy(), v)
        g, d = B.sim_eval_gradient(sim.h, sx, sx)
        out.append((g, d, B.sim_eval_pHp(sim.h, sx, sp), B.sim_eval_hvp(sim.h, sx, sp)))
        sim.close()
    u = 2.0**-53 if prec == 0 else 2.0**-24
    for a, b in zip(*out):     # equal up to the order of the atomic adds: at most 24 tets a vertex, and the sums' cancellation
        assert np.abs(a - b).max() <= 64 * u * max(np.abs(a).max(), np.abs(out[0][1]).max() * 1e-4)
