"""The FP64 solve against the V-cycle assembled from the component entry points.

A right-hand side of small whole numbers that sum to zero and a spacing that is a power of two leave the solve's
b - mean(b) and h^2 b exact, so its cycles must be bitwise the component ones; what differs is the mean taken off at
the exit, one rounding of p and one of the mean.
"""
import pytest
import torch

from paper_2605_30082_gb300 import Solver

from _helpers import dev, random_rho
from test_gpu_dd import whole_vcycle

pytestmark = pytest.mark.gpu


# one to three levels in the cluster of the coarse levels, with 64 to 512 cells below them, with 990 (descent and ascent as
# two launches), no cluster
@pytest.mark.parametrize("dims,coarsest,pre,post", [((64, 64, 64), 4, 2, 2), ((32, 48, 24), 6, 1, 3), ((72, 80, 88), 11, 2, 1),
                                                    ((16, 64, 128), 4, 1, 1), ((16, 16, 16), 8, 2, 2), ((64, 64, 64), 8, 2, 2)])
def test_solve_is_the_component_cycles(dims, coarsest, pre, post):
    s = Solver(dims, h=1.0 / 64, precision="fp64", coarsest=coarsest, pre=pre, post=post, rtol=0.0, max_cycles=8)
    s.set_density(dev(random_rho(dims, 31)))
    g = torch.Generator(device="cuda").manual_seed(4)
    n = dims[0] * dims[1] * dims[2]
    half = torch.randint(-50, 51, (n // 2,), generator=g, device="cuda", dtype=torch.float64)
    b = torch.cat([half, -half])[torch.randperm(n, generator=g, device="cuda")].view(s.cell_shape)
    p = s.solve(b, raise_on_nonconvergence=False)
    x = torch.zeros_like(b)
    for _ in range(8):
        whole_vcycle(s, b, x)
    want = x - x.mean()
    # the means are sums of n numbers in another order: n^(1/2) roundings of their mean size, as a mean below one of p's
    assert float((p - want).abs().max()) <= 4 * 2.0 ** -53 * float(x.abs().max())
    s.close()
