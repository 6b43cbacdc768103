"""A handle after a solve that left no numbers in its levels: the next solve must not see them.

A warm start from p of the order of 1e200 overflows the FP32 residual, so that every level's x becomes NaN and the
solve ends with MG_ERR_DIVERGED.  A sweep from zero writes such a level without having cleared it.
"""
import pytest
import torch

from paper_2605_30082_gb300 import MgError, Solver
from paper_2605_30082_gb300 import _lib as L

from _helpers import dev, random_rho

pytestmark = pytest.mark.gpu


# nx / 2 a multiple of four or not on the finest level (from a density) and below it; with the coarse levels
# launch by launch and in the cluster
@pytest.mark.parametrize("dims,coarsest,kw", [((72, 80, 88), 11, {}), ((36, 20, 28), 7, dict(prolong="constant")),
                                              ((40, 20, 28), 7, dict(prolong="constant")), ((36, 20, 28), 14, {}),
                                              ((64, 64, 64), 8, {}), ((64, 64, 64), 8, dict(prolong="constant"))])
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_solve_after_a_diverged_one(dims, coarsest, kw, prec):
    s = Solver(dims, precision=prec, coarsest=coarsest, warm_start=True, max_cycles=300, **kw)
    s.set_density(dev(random_rho(dims, 5)))
    g = torch.Generator(device="cuda").manual_seed(1)
    b = torch.randn(s.cell_shape, generator=g, device="cuda", dtype=torch.float64)
    p_ref = s.solve(b)
    with pytest.raises(MgError) as ei:
        s.solve(b, 1e200 * torch.randn(s.cell_shape, generator=g, device="cuda", dtype=torch.float64))
    assert ei.value.code == L.MG_ERR_DIVERGED
    assert torch.equal(s.solve(b), p_ref)
    s.close()
