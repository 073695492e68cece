"""Device memory of a handle."""
import pytest

from paper_2405_08001_gb300 import scenes as S
from test_gpu_parity import B  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scatter", [0, 3])
@pytest.mark.parametrize("prec", [0, 1])
def test_corotated_handles_hold_only_what_their_passes_read(B, prec, scatter):  # noqa: F811
    """FCR and ARAP work on F: their handles hold none of the constants of the passes on edge vectors.  FP64: 64 bytes a tet
    of constants and 16 of the record less than Neo-Hookean (and the constants' copy in colour order).  FP32: 56 bytes of
    rest metric in the place of 80 of constants and 4 of the record."""
    import torch
    sc = S.cube_drop(n=30)
    used = []
    for model in (0, 2, 0, 2):     # the first two load the kernels
        torch.cuda.synchronize()
        f = torch.cuda.mem_get_info()[0]
        sim = B.Sim(sc, precision=prec, model=model, scatter=scatter)
        used.append(f - torch.cuda.mem_get_info()[0])
        sim.close()
    copies = 2 if scatter == 3 else 1
    less = (copies * 64 + 16 if prec == 0 else copies * (80 - 56) + 4) * sc.n_tets
    assert used[2] - used[3] >= less - (4 << 20), used      # the driver's 2 MB pages
