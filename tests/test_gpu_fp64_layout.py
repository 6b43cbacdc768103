"""The FP64 path where b and the reciprocal diagonal lie colour by colour, and its red prolongation."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2605_30082_gb300 import _lib as L
from paper_2605_30082_gb300 import Solver

from _helpers import dev, host, random_rho, rel

pytestmark = pytest.mark.gpu


# a block of the prolongation takes 254 coarse cells: fewer, exactly one and two blocks, one more; rows of one and two
# coarse cells, a single row, a single plane
@pytest.mark.parametrize("dims", [(4, 4, 4), (2, 254, 4), (4, 254, 4), (508, 2, 2), (510, 2, 2), (34, 30, 8), (8, 4, 254), (130, 6, 10)])
def test_red_prolongation_matches_oracle(dims):
    nx, ny, nz = dims
    s = Solver(dims, h=1.0 / 64, precision="fp64", coarsest=2)
    if s.num_levels < 2:
        pytest.skip("a single level has no prolongation")
    rho = random_rho(dims, 71)
    s.set_density(dev(rho))
    rng = np.random.default_rng(72)
    x, b = rng.standard_normal((nz, ny, nx)), rng.standard_normal((nz, ny, nx))
    ec = rng.standard_normal((nz // 2, ny // 2, nx // 2))
    xg = dev(x)
    assert L.mg_prolong_postsmooth(s._h, 0, dev(ec), xg, dev(b), 1) == L.MG_OK
    want = O.rbgs(O.faces_from_density(rho), b, O.prolong_correct(ec, x, O.TRILINEAR), 1.0 / 64, 1, 1)
    assert rel(host(xg), want) < 1e-13  # the tolerance of the other FP64 comparisons of these operations


@pytest.mark.parametrize("dims", [(24, 36, 20), (48, 20, 28), (2, 8, 16), (96, 64, 48)])
@pytest.mark.parametrize("pre,post", [(2, 2), (0, 2), (1, 0)])
def test_one_cycle_matches_oracle(dims, pre, post):
    nx, ny, nz = dims
    h = 1.0 / max(dims)
    rho = random_rho(dims, 73)
    rng = np.random.default_rng(74)
    b = rng.standard_normal((nz, ny, nx))
    s = Solver(dims, h=h, precision="fp64", coarsest=4, pre=pre, post=post, rtol=0.0, max_cycles=1)
    s.set_density(dev(rho))
    M = O.Multigrid(O.faces_from_density(rho), h, coarsest=4, pre=pre, post=post)
    want = M.vcycle(b - b.mean(), np.zeros_like(b))
    want -= want.mean()
    pool = torch.zeros(b.size + 1, dtype=torch.float64, device="cuda")
    for shift in (0, 1):  # a right-hand side on a 16-byte boundary and off it
        bg = pool[shift:shift + b.size].view(nz, ny, nx)
        bg.copy_(dev(b))
        p = host(s.solve(bg, raise_on_nonconvergence=False))
        assert rel(p, want) < 1e-12  # as the other single-cycle comparisons
