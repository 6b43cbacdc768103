"""The row-sharing half sweep, which takes levels of 60 M cells and more, against the oracle at the edges of its tiles."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2605_30082_gb300 import _lib as L
from paper_2605_30082_gb300 import Solver

from _helpers import dev, host, rel

pytestmark = pytest.mark.gpu


# whole rows of 64 and of 32 vectors; rows of 104 vectors in tiles of 16, the last of them half empty
@pytest.mark.parametrize("dims", [(512, 384, 320), (256, 512, 512), (832, 320, 256)])
def test_large_row_tiles_match_oracle(dims):
    nx, ny, nz = dims
    s = Solver(dims, h=1.0 / 64, precision="mixed", coarsest=4)
    rng = np.random.default_rng(91)
    rho = rng.uniform(1.0, 100.0, (nz, ny, nx))
    s.set_density(dev(rho))
    faces = tuple(f.astype(np.float32).astype(np.float64) for f in O.faces_from_density(rho))
    x = rng.standard_normal((nz, ny, nx), dtype=np.float32)
    b = rng.standard_normal((nz, ny, nx), dtype=np.float32)
    xs = dev(x, torch.float32)
    assert L.mg_smooth(s._h, 0, xs, dev(b, torch.float32), 1, 1) == L.MG_OK
    # the tolerance of the other FP32 smoothing comparisons
    assert rel(host(xs), O.rbgs(faces, b, x, 1.0 / 64, 1, 1)) < 2e-6
