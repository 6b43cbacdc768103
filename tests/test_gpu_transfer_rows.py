"""FP32 restriction and prolongation of red-only levels against the oracle, either side of the sizes at which
one thread takes one fine row instead of all four.

A last group of fewer than eight vectors, rows of one vector, one and several coarse rows per warp, a
single coarse plane; then the last size below and the first above each threshold.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2605_30082_gb300 import _lib as L
from paper_2605_30082_gb300 import Solver

from _helpers import dev, host, random_rho, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(16, 6, 10), (8, 12, 20), (24, 36, 4), (80, 4, 12), (48, 20, 28), (128, 4, 8), (80, 64, 192),
                                  (96, 96, 112), (160, 192, 256), (192, 192, 224)])
@pytest.mark.parametrize("coeffs", ["rho", "faces"])
def test_row_transfers_match_oracle(dims, coeffs):
    nx, ny, nz = dims
    s = Solver(dims, h=1.0 / 64, precision="mixed", coarsest=2)
    rho = random_rho(dims, 61)
    if coeffs == "rho":
        s.set_density(dev(rho))
    else:
        s.set_face_coeffs(*(dev(f) for f in O.faces_from_density(rho)))
    rng = np.random.default_rng(62)
    x, b = (rng.standard_normal((nz, ny, nx)).astype(np.float32) for _ in range(2))
    ec = rng.standard_normal((nz // 2, ny // 2, nx // 2)).astype(np.float32)
    faces = tuple(f.astype(np.float32).astype(np.float64) for f in O.faces_from_density(rho))
    # after one sweep ending in black the red cells alone carry a residual, which is what the restriction reads
    xg, bg = dev(x, torch.float32), dev(b, torch.float32)
    bc = torch.empty((nz // 2, ny // 2, nx // 2), dtype=torch.float32, device="cuda")
    assert L.mg_presmooth_restrict(s._h, 0, xg, bg, 1, bc) == L.MG_OK
    # the tolerances of the other comparisons of these two operations
    assert rel(host(bc), O.restrict(O.residual(faces, b, host(xg), 1.0 / 64))) < 2e-5
    xp = dev(x, torch.float32)
    assert L.mg_prolong_postsmooth(s._h, 0, dev(ec, torch.float32), xp, bg, 1) == L.MG_OK
    want = O.rbgs(faces, b, O.prolong_correct(ec, x, O.TRILINEAR), 1.0 / 64, 1, 1)
    assert rel(host(xp), want) < 1e-5
