"""The wide set-up passes against the oracle and against the general ones, which take arrays off a 16-byte boundary."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2605_30082_gb300 import Solver

from _helpers import dev, host, random_rho, rel

pytestmark = pytest.mark.gpu


def off_boundary(a):
    pool = torch.empty(a.numel() + 1, dtype=a.dtype, device=a.device)
    v = pool[1:].view(a.shape)
    v.copy_(a)
    return v


# less than one block of the density pass, a full one, odd numbers of cells, several blocks
@pytest.mark.parametrize("dims", [(4, 4, 4), (16, 8, 8), (31, 11, 3), (3, 7, 9), (64, 36, 20)])
@pytest.mark.parametrize("nfrac", [1, 2, 3, 4])
def test_density_matches_definition(dims, nfrac):
    nx, ny, nz = dims
    rng = np.random.default_rng(81)
    f = [rng.random((nz, ny, nx)) / nfrac for _ in range(nfrac)]
    phase = [1000.0, 850.0, 1.2, 60.0, 7.0][:nfrac + 1]
    want = phase[-1] + sum((p - phase[-1]) * q for p, q in zip(phase, f))
    s = Solver(dims, h=1.0 / 64, precision="fp64", coarsest=64 if nx % 2 else 4)
    a = s.density_from_fractions([dev(q) for q in f], phase)
    assert rel(host(a), want) < 1e-14  # nfrac + 1 roundings of 1.1e-16
    assert torch.equal(a, s.density_from_fractions([off_boundary(dev(q)) for q in f], phase))


@pytest.mark.parametrize("dims", [(24, 12, 20), (72, 40, 24), (36, 6, 10), (9, 7, 5)])
@pytest.mark.parametrize("prec", ["mixed", "mixed_df", "fp64"])
def test_density_set_up_does_not_depend_on_alignment(dims, prec):
    nx, ny, nz = dims
    if prec == "mixed_df" and nx % 2:
        pytest.skip("mixed_df takes even nx")
    rho = dev(random_rho(dims, 82))
    b = dev(np.random.default_rng(83).standard_normal((nz, ny, nx)))
    p = []
    for r in (rho, off_boundary(rho)):
        s = Solver(dims, h=1.0 / 64, precision=prec, coarsest=64 if nx % 2 else 4, rtol=1e-8)
        s.set_density(r)
        p.append(s.solve(b))
    assert torch.equal(p[0], p[1])


def test_double_float_operator_from_density_then_from_faces():
    """The pairs of the faces and of the diagonal are formed only for an operator from faces: also after one from a density."""
    dims = (24, 12, 20)
    b = dev(np.random.default_rng(84).standard_normal(dims[::-1]))
    faces = [dev(f) for f in O.faces_from_density(random_rho(dims, 85))]
    p = []
    for first in (True, False):
        s = Solver(dims, h=1.0 / 64, precision="mixed_df", coarsest=4, rtol=1e-8)
        if first:
            s.set_density(dev(random_rho(dims, 86)))
            s.solve(b)
        s.set_face_coeffs(*faces)
        p.append(s.solve(b))
    assert torch.equal(p[0], p[1])
