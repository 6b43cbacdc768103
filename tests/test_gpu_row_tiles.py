"""The row-sharing half sweep of large s-form levels against the oracle, at the edges of its tiles."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2605_30082_gb300 import _lib as L
from paper_2605_30082_gb300 import Solver

from _helpers import dev, host, random_rho, rel

pytestmark = pytest.mark.gpu


# whole rows of 32 and 64 vectors (every thread in use), rows of 24 and 40 vectors with a ragged last row
# tile, rows split into tiles of 16 and 24 vectors, two tiles of 64 vectors; and one
# level just below the threshold, which takes the plain kernel
@pytest.mark.parametrize("dims", [(256, 144, 112), (512, 96, 80), (192, 224, 192), (320, 160, 160), (384, 96, 160),
                                  (576, 128, 96), (1024, 64, 64), (256, 144, 80)])
def test_row_tiles_match_oracle(dims):
    nx, ny, nz = dims
    h = 1.0 / 64
    s = Solver(dims, h=h, precision="mixed", coarsest=4)
    rho = random_rho(dims, 51)
    s.set_density(dev(rho))
    faces = tuple(f.astype(np.float32).astype(np.float64) for f in O.faces_from_density(rho))
    rng = np.random.default_rng(52)
    x = rng.standard_normal((nz, ny, nx)).astype(np.float32)
    b = rng.standard_normal((nz, ny, nx)).astype(np.float32)
    xs = dev(x, torch.float32)
    assert L.mg_smooth(s._h, 0, xs, dev(b, torch.float32), 2, 1) == L.MG_OK
    # the tolerance of the other FP32 smoothing comparisons
    assert rel(host(xs), O.rbgs(faces, b, x, h, 2, 1)) < 2e-6
