"""The cluster form of the persistent step (small meshes, default block shape): lock-step against the oracle on both
sides of the size rule, with ragged cell counts, down to one cell, in both precisions; and against the whole-grid form
over the options that it takes (beta rule, densities, p-norm, split objects, batches)."""
import numpy as np
import pytest

from paper_2405_08001_gb300 import scenes as S
from test_gpu_parity import B, CHECKED, O, TOL, lockstep  # noqa: F401  (B and O are fixtures)

pytestmark = pytest.mark.gpu


def cells_for(tets):
    """Cell counts (ragged) of a box of at most that many tets, and of nearly as many."""
    n = tets // 6
    k = max(1, round(n ** (1.0 / 3.0)))
    return max(((i, j, n // (i * j)) for i in range(k - 4, k + 5) for j in range(k - 4, i)), key=lambda c: c[0] * c[1] * c[2])


def rounds(q):
    """q tets a thread of one block of 256 threads an SM."""
    import torch
    return int(q * 256 * torch.cuda.get_device_properties(0).multi_processor_count)


# ... and of the next rule: one block of 256 threads an SM up to three rounds of 256 x SMs tets, two above (and in FP64 up to
# four thirds of a round above one)
@pytest.mark.parametrize("prec,cells,blocks", [(1, (1, 1, 1), 1), (1, (9, 11, 13), 1), (1, (11, 11, 12), 1),
                                               (0, (1, 2, 1), 1), (0, (8, 8, 10), 1), (0, (8, 9, 10), 1),
                                               (0, 0.99, 1), (0, 1.1, 2), (0, 1.32, 2), (0, 1.45, 1), (1, 2.98, 1), (1, 3.1, 2)])
def test_both_sides_of_the_size_rule(B, O, prec, cells, blocks):  # noqa: F811
    if isinstance(cells, float):
        q, cells = cells, cells_for(rounds(cells))
        assert abs(6 * np.prod(cells) / rounds(q) - 1.0) < 0.02     # within the side that q names
    sc = S.cube_drop(n=max(cells), cells=cells, drop=0.0)
    sc.x0 = sc.x0 + np.array([0.0, 0.0, 0.6 * sc.dhat])
    sim = B.Sim(sc, precision=prec)
    st = sim.state()[2]
    assert (st["block_threads"], st["blocks_per_sm"]) == (256, blocks), st
    worst = lockstep(B, O, O.Oracle.from_scene(sc), sim, sc, 3, prec)
    for k in CHECKED:
        assert worst[k] < TOL[prec], (k, worst[k])
    sim.close()


@pytest.mark.parametrize("make,kw", [(lambda: S.two_blocks(1), dict(beta=1)), (lambda: S.two_blocks(1), dict(pnorm=1)),
                                     (lambda: S.two_blocks(2), dict(model=1)), (lambda: S.two_blocks(2), dict(model=2)),
                                     (lambda: S.two_blocks(2), dict(use_graph=0)),
                                     (lambda: S.two_blocks(2), dict(scatter=1)),
                                     (lambda: S.objects(0), dict(split_objects=1)),
                                     (lambda: S.batched(3, n_min=2, n_max=4), {})])
def test_same_step_as_the_whole_grid(B, make, kw):  # noqa: F811
    """One FP64 step in the cluster form and in 256 x 1 blocks on the whole grid (the same arithmetic, another order of
    the sums): equal within the growth of rounding over the step's iterations, up to 1e4 over four on these scenes (1e7 over
    eight)."""
    sc = make()
    out = []
    for shape in (0, 3):
        sim = B.Sim(sc, precision=0, block_shape=shape, iters=4, **kw)
        sim.step(1, sc.targets(0))
        out.append(sim.state()[0])
        sim.close()
    assert np.abs(out[0] - out[1]).max() <= 1e-9 * np.abs(out[1] - sc.x0).max()


@pytest.mark.parametrize("persistent", [0, 1])
def test_fp64_first_direction_is_the_rounded_quotient(B, persistent):  # noqa: F811
    """p_1 = -P g with P = 1 / diag, each operation rounded once: bit by bit, in both launch forms."""
    sc = S.two_blocks(0)
    sim = B.Sim(sc, precision=0, persistent=persistent)
    B.sim_begin_step(sim.h)
    B.sim_iterate(sim.h, 1)
    x, g, P, p, *_ = B.sim_get_iterate(sim.h)
    assert np.array_equal(p, -(P * g))
    sim.close()


@pytest.mark.parametrize("prec", [0, 1])
def test_autotuner_times_every_shape_on_a_small_mesh(B, prec):  # noqa: F811
    """block_shape = -1 on a mesh that the default runs as one cluster: the tuned steps run 256 x 2 on the whole grid too."""
    sim = B.Sim(S.two_blocks(0), precision=prec, block_shape=-1)
    seen = set()
    for _ in range(14):
        sim.step(1)
        st = sim.state()[2]
        seen.add((st["block_threads"], st["blocks_per_sm"]))
    assert {(256, 1), (256, 2), (256, 3), (512, 1), (384, 1)} <= seen, seen
    sim.close()
