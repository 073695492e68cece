"""Host-side checks of arithmetic that the device shares (the geometry header is host and device code): compiled by nvcc and
run on the CPU, with and without contraction of products and sums."""
import os
import subprocess

import pytest

from paper_2405_08001_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module", params=["off", "fast"])
def program(request, tmp_path_factory):
    out = str(tmp_path_factory.mktemp("host") / f"arithmetic_{request.param}")
    # "fast" lets the compiler contract; only where the CPU has FMA by default (aarch64) does it
    subprocess.run([build.NVCC, *build.ARCH, "-O2", "-std=c++17", "-I", build.CSRC, "-Xcompiler", f"-ffp-contract={request.param}",
                    os.path.join(HERE, "host", "arithmetic.cu"), "-o", out], check=True, capture_output=True)
    return lambda *a: subprocess.run([out, *map(str, a)], check=True, capture_output=True, text=True).stdout.split()


# sin^2 of the angle around the interior solution's limit of 1e-5, up to where it does not matter, and nearly 0
@pytest.mark.parametrize("sin2", [(1e-12, 1e-9), (1e-7, 8e-6), (8e-6, 1e-5), (1e-5, 1.5e-5), (1.5e-5, 1e-3), (1e-3, 1.0)])
@pytest.mark.parametrize("ratio", [5, 20, 100, 300])
@pytest.mark.parametrize("ee", [0, 1])
def test_candidate_bound_is_below_the_distance(program, ee, ratio, sin2):
    """No candidate's stored bound exceeds its distance: nearly parallel edges and sliver triangles, edges of 5 to 300 dhat."""
    above, worst = program("bounds", ee, ratio, *sin2, 100000)
    assert above == "0", worst


def test_quotients_by_one_reciprocal_are_the_divisions(program):
    """The FP64 pairs' and beta's quotients, formed from one reciprocal and corrected by their residual, are those of the
    division: by Markstein's theorem for every divisor but the one whose mantissa is all ones."""
    assert program("quotients", 2000000) == ["0"]


# x = 1 - d / dhat, from just below dhat to near contact
@pytest.mark.parametrize("x", [(1e-8, 1e-4), (1e-4, 1e-2), (1e-2, 0.3), (0.3, 0.99)])
def test_fp64_barrier_slope_rounds_no_more_than_its_formula(program, x):
    """b' = -2 r L - r^2 / d from r / d, which b'' needs too: as many roundings as the formula's own (200,000 samples give
    either rms to 1 %, the margin is 5)."""
    ours, ref = map(float, program("barrier", *x, 200000))
    assert ours <= 1.05 * ref, (ours, ref)
