"""A wait of the coarse levels' cluster that runs out in the decomposed mixed solve is reported as such.

The cluster runs on the whole-grid handle of the switch level; the decomposed solve, which only sees its NaN, must
return MG_ERR_CUDA with the handle's reason instead of a divergence, and solve as before afterwards.
"""
import pytest
import torch

from paper_2605_30082_gb300 import _lib as L

from _helpers import dev, random_rho
from test_gpu_dd import _mixed_opts

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("inner", [1, 3])  # launched, and behind replayed cycles
def test_cluster_wait_in_the_decomposed_solve(inner):
    dims = (64, 64, 64)
    st, dd = L.mg_dd_create(_mixed_opts(dims, 1 / 64, inner, coarsest=4), 2, 1)
    assert st == L.MG_OK
    assert L.mg_dd_set_density(dd, dev(random_rho(dims, 5)), dims) == L.MG_OK
    g = torch.Generator(device="cuda").manual_seed(1)
    b = torch.randn(dims, generator=g, device="cuda", dtype=torch.float64)
    p_ref, p = torch.zeros_like(b), torch.zeros_like(b)
    assert L.mg_dd_solve(dd, b, p_ref, dims) == L.MG_OK
    assert L.mg_dd_debug_inject(dd, L.MG_INJECT_TAIL_WAIT) == L.MG_OK
    assert L.mg_dd_solve(dd, b, p, dims) == L.MG_ERR_CUDA
    assert "gave up waiting" in L.mg_dd_last_error(dd)
    assert L.mg_dd_solve(dd, b, p, dims) == L.MG_OK, L.mg_dd_last_error(dd)
    assert torch.equal(p, p_ref)
    L.mg_dd_destroy(dd)
