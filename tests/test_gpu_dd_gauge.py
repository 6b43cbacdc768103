"""The decomposed FP64 solve against the whole-grid one, both of which take the mean of p off at the exit only.

A right-hand side of small whole numbers that sum to zero leaves b - mean(b) exact whatever the order of the sums, and
the cycles are bitwise the same: the two pressures differ by their means at the exit, a rounding of each.  With 512
coarse cells a shift of p in every cycle, on one side only, moved p by 9e-14 on 128^3 and 1e-12 on 512^3.
"""
import pytest
import torch

import dropfilm as D
from paper_2605_30082_gb300 import Solver
from paper_2605_30082_gb300 import _lib as L

from test_gpu_dd import DD

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ranks,coarsest", [(64, 2, 4), (128, 4, 8), (256, 4, 8)])
def test_decomposed_solve_differs_by_a_rounding(n, ranks, coarsest):
    g = D.scaled_geometry(n)
    fd, ff = D.fractions_ramp(g)
    rho = (998 * fd + 880 * ff + 1.2 * (1 - fd - ff)).cuda()
    dims, m = (n, n, n), n ** 3
    gen = torch.Generator(device="cuda").manual_seed(4)
    half = torch.randint(-50, 51, (m // 2,), generator=gen, device="cuda", dtype=torch.float64)
    b = torch.cat([half, -half])[torch.randperm(m, generator=gen, device="cuda")].view(n, n, n)
    s = Solver(dims, h=1.0 / n, precision="fp64", coarsest=coarsest, rtol=1e-10)
    s.set_density(rho)
    pw = s.solve(b)
    dd = DD(dims, ranks, 0, h=1.0 / n, rtol=1e-10, coarsest=coarsest)
    assert L.mg_dd_set_density(dd.h, rho, dims) == L.MG_OK
    pd, st = torch.zeros_like(b), L.mg_stats()
    assert L.mg_dd_solve(dd.h, b, pd, dims, st) == L.MG_OK, L.mg_dd_last_error(dd.h)
    assert st.cycles == s.last_stats.cycles
    assert float((pd - pw).norm() / pw.norm()) <= 4 * 2.0 ** -53
    dd.close()
    s.close()
