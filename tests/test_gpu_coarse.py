"""The dense coarse pseudo-inverse at the edges of its plane and pivot-block sizes."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2605_30082_gb300 import Solver
from paper_2605_30082_gb300 import _lib as L

from _helpers import dev, host, random_rho, rel

pytestmark = pytest.mark.gpu


def _cond(faces, h):
    """Largest over smallest nonzero eigenvalue of the operator."""
    nz, ny, nx = faces[0].shape[0], faces[0].shape[1], faces[0].shape[2] - 1
    n = nx * ny * nz
    ids = np.arange(n).reshape(nz, ny, nx)
    A = np.zeros((n, n))
    for a, b, f in ((ids[:, :, 1:], ids[:, :, :-1], faces[0][:, :, 1:-1]), (ids[:, 1:], ids[:, :-1], faces[1][:, 1:-1]),
                    (ids[1:], ids[:-1], faces[2][1:-1])):
        a, b, f = a.ravel(), b.ravel(), np.asarray(f).ravel() / (h * h)
        np.add.at(A, (a, a), f)
        np.add.at(A, (b, b), f)
        A[a, b] -= f
        A[b, a] -= f
    ev = np.linalg.eigvalsh(A)
    return ev[-1] / ev[1]


# one cell per plane (2 and 1024 planes), planes of 8 cells and one more, of 64, 100 and 96 cells, each
# axis as the longest, a two-dimensional grid, a middle plane with nothing above it
@pytest.mark.parametrize("dims", [(2, 1, 1), (1, 1024, 1), (2, 4, 9), (3, 3, 8), (8, 8, 8), (16, 8, 8), (10, 10, 10),
                                  (8, 10, 12), (10, 8, 12), (5, 20, 10), (32, 32, 1), (9, 10, 11), (1, 1, 3)])
@pytest.mark.parametrize("contrast", [1.0, 832.0])
def test_coarse_inverse_matches_oracle(dims, contrast):
    nx, ny, nz = dims
    h = 1.0 / max(dims)
    faces = O.faces_from_density(random_rho(dims, 31, 1.2, 1.2 * contrast))
    s = Solver(dims, h=h, precision="fp64", coarsest=max(dims))
    s.set_face_coeffs(*(dev(f) for f in faces))
    assert s.num_levels == 1
    r = np.random.default_rng(7).standard_normal((nz, ny, nx))
    e = torch.empty((nz, ny, nx), dtype=torch.float64, device="cuda")
    assert L.mg_coarse_solve(s._h, dev(r), e) == L.MG_OK
    # both sides solve directly: each may be off by a few units of rounding times the condition number
    tol = 1e-14 + 8 * np.finfo(np.float64).eps * _cond(faces, h)
    assert rel(host(e), O.coarse_solve(faces, r, h)) < tol
    assert abs(host(e).mean()) <= tol * np.abs(host(e)).max()
