"""One V-cycle whose coarse levels run as one cluster launch, against the oracle's V-cycle.

Grids at the edges of the distribution of rows over the cluster: fewer row quads than CTAs, a
ragged last CTA, rows of two cells, long rows, an odd and a two-plane coarsest level, one to three levels in
the cluster, more coarse cells than the cluster solves itself (descent and ascent as two launches), the largest
level it holds.
"""
import numpy as np
import pytest

import oracle as O
from paper_2605_30082_gb300 import Solver

from _helpers import dev, host, random_rho, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,coarsest", [((32, 32, 32), 4), ((64, 64, 64), 8), ((24, 36, 20), 4), ((8, 12, 256), 4),
                                           ((512, 8, 8), 4), ((4, 256, 16), 4), ((72, 80, 88), 8), ((40, 56, 24), 4)])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("pre,post", [(2, 2), (1, 3)])
def test_one_vcycle_matches_oracle(dims, coarsest, prec, pre, post):
    nx, ny, nz = dims
    h = 1.0 / max(dims)
    rho = random_rho(dims, 41)
    b = np.random.default_rng(8).standard_normal((nz, ny, nx))
    b -= b.mean()
    s = Solver(dims, h=h, precision=prec, coarsest=coarsest, pre=pre, post=post, rtol=0.0, max_cycles=1)
    assert s.num_levels >= 3
    s.set_density(dev(rho))
    p = host(s.solve(dev(b), raise_on_nonconvergence=False))
    assert s.last_stats.cycles == 1
    M = O.Multigrid(O.faces_from_density(rho), h, coarsest=coarsest, pre=pre, post=post)
    want = M.vcycle(b, np.zeros_like(b))
    want = want - want.mean()
    # FP64: the tolerance of the other single-cycle comparisons; FP32: 6e-8 per operation, some hundred
    # rounded operations per cell and cycle
    assert rel(p, want) < (1e-12 if prec == "fp64" else 1e-5)
