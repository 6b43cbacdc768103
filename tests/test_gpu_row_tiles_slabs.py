"""The row-sharing half sweep where test_gpu_row_tiles_large.py does not go: other tile widths, and slabs.

A whole grid of 60 M cells and more has sides that are multiples of 64 (or its coarsest level would exceed the dense
solve), so tiles are whole in y and z there; a slab's last planes can be part of a tile.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2605_30082_gb300 import _lib as L
from paper_2605_30082_gb300 import Solver

from _helpers import dev, host, rel
from test_gpu_dd import _mixed_opts

pytestmark = pytest.mark.gpu


# whole rows of 8 vectors; two full tiles of 64; 88 vectors in tiles of 32, the last a quarter empty
@pytest.mark.parametrize("dims", [(64, 1024, 1024), (1024, 256, 256), (704, 384, 256)])
def test_tile_widths_match_oracle(dims):
    nx, ny, nz = dims
    s = Solver(dims, h=1.0 / 64, precision="mixed", coarsest=4 if nx > 64 else 16)
    rng = np.random.default_rng(93)
    rho = rng.uniform(1.0, 100.0, (nz, ny, nx))
    s.set_density(dev(rho))
    faces = tuple(f.astype(np.float32).astype(np.float64) for f in O.faces_from_density(rho))
    x = rng.standard_normal((nz, ny, nx), dtype=np.float32)
    b = rng.standard_normal((nz, ny, nx), dtype=np.float32)
    xs = dev(x, torch.float32)
    assert L.mg_smooth(s._h, 0, xs, dev(b, torch.float32), 1, 1) == L.MG_OK
    # the tolerance of the other FP32 smoothing comparisons
    assert rel(host(xs), O.rbgs(faces, b, x, 1.0 / 64, 1, 1)) < 2e-6


# slabs of 256 planes, one tile per row; of 40 planes, two tiles and half of one, five tiles per row (a slab whose planes are
# no multiple of 16 takes this sweep in 16 slabs of 960 M cells at least)
@pytest.mark.parametrize("dims,ranks", [((512, 512, 512), 2), ((1280, 1280, 640), 16)])
def test_slabs_are_the_whole_grid(dims, ranks):
    """One V-cycle.  With a right-hand side of small whole numbers that sum to zero all sums before it are exact, so
    every cell sees the same arithmetic; the means taken off at the exit differ by a rounding."""
    nx, ny, nz = dims
    n, h = nx * ny * nz, 1.0 / max(dims)
    gen = torch.Generator(device="cuda").manual_seed(4)
    rho = torch.exp(torch.rand((nz, ny, nx), generator=gen, device="cuda", dtype=torch.float64).mul_(6.7))
    half = torch.randint(-50, 51, (n // 2,), generator=gen, device="cuda", dtype=torch.float64)
    b = torch.empty_like(rho).view(2, -1)
    b[0], b[1] = half, -half.roll(12345)
    b = b.view(nz, ny, nx)
    del half
    s = Solver(dims, h=h, precision="mixed", coarsest=10, max_cycles=1)
    s.set_density(rho)
    pw = s.solve(b, raise_on_nonconvergence=False)
    s.close()
    o = _mixed_opts(dims, h, 1, coarsest=10)
    o.max_cycles = 1
    st, dd = L.mg_dd_create(o, ranks, 1)
    assert st == L.MG_OK, st
    assert L.mg_dd_set_density(dd, rho, dims) == L.MG_OK
    pd = torch.zeros_like(b)
    assert L.mg_dd_solve(dd, b, pd, dims) == L.MG_ERR_NOT_CONVERGED, L.mg_dd_last_error(dd)
    L.mg_dd_destroy(dd)
    assert float(pw.abs().max()) > 0
    assert float((pd - pw).abs().max()) <= 4 * 2.0 ** -53 * float(pw.abs().max())
