"""The bounded waits of the coarse levels' cluster, made to run out by a one-shot fault armed on the host.

Its first CTA expects bytes that nobody sends, gives up after about a second and stops sending, so that the waits of
all others run out in turn; every CTA stays until the whole cluster is done, sets bit 8 of the error word and leaves NaN.
mg_solve must report MG_ERR_CUDA with that reason, and the next solve must be bitwise the clean one.
"""
import pytest
import torch

from paper_2605_30082_gb300 import MgError, Solver
from paper_2605_30082_gb300 import _lib as L

from _helpers import dev, random_rho

pytestmark = pytest.mark.gpu


# one launch a cycle; descent and ascent as two launches around the product of 990 cells; conjugate gradients;
# a single half sweep of each colour on the way up, after which the CTAs leave
@pytest.mark.parametrize("dims,prec,kw", [((64, 64, 64), "mixed", {}), ((32, 32, 32), "fp64", dict(coarsest=4)),
                                          ((72, 80, 88), "mixed", {}), ((72, 80, 88), "fp64", dict(coarsest=11)),
                                          ((64, 64, 64), "mixed", dict(method="fcg", inner_cycles=2)),
                                          ((64, 48, 32), "mixed", dict(pre=1, post=1))])
def test_cluster_wait_runs_out_and_handle_recovers(dims, prec, kw):
    s = Solver(dims, precision=prec, max_cycles=300, **{"coarsest": 11 if dims[0] == 72 else 8, **kw})
    s.set_density(dev(random_rho(dims, 5)))
    g = torch.Generator(device="cuda").manual_seed(1)
    b = torch.randn(s.cell_shape, generator=g, device="cuda", dtype=torch.float64)
    p_ref = s.solve(b).clone()
    assert L.mg_debug_inject(s._h, L.MG_INJECT_TAIL_WAIT) == L.MG_OK
    with pytest.raises(MgError) as ei:
        s.solve(b)
    assert ei.value.code == L.MG_ERR_CUDA
    assert "gave up waiting" in str(ei.value)
    p = s.solve(b)  # one-shot, and the error word was cleared
    assert s.last_stats.status == L.MG_OK
    assert torch.equal(p, p_ref)
    s.close()
