"""The outer update as a pass of its own (no post sweep to carry it), in pairs of cells for even nx, against FP64."""
import numpy as np
import pytest

from paper_2605_30082_gb300 import Solver

from _helpers import dev, host, random_rho, rel

pytestmark = pytest.mark.gpu


# one pair, an odd number of pairs per row and a row pitch off a multiple of four, full rows; odd nx: one cell per thread
@pytest.mark.parametrize("dims", [(2, 6, 10), (10, 6, 14), (72, 40, 24), (7, 6, 10)])
def test_unfused_update_reaches_the_fp64_solution(dims):
    nx, ny, nz = dims
    b = dev(np.random.default_rng(95).standard_normal((nz, ny, nx)))
    rho = dev(random_rho(dims, 96))
    p = {}
    for prec in ("mixed", "fp64"):
        s = Solver(dims, h=1.0 / 64, precision=prec, pre=2, post=0 if prec == "mixed" else 2, coarsest=4, rtol=1e-11, max_cycles=400)
        s.set_density(rho)
        p[prec] = host(s.solve(b))
    # both residuals are at most 1e-11 of b; the condition of these small problems is below 1e3
    assert rel(p["mixed"], p["fp64"]) < 1e-7
