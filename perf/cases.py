"""The workloads whose speed this framework is held to.

A case is one pass of work that a flow solver or a training loop hands to the framework through
its public entry points: the projection step of one time step (density from the volume
fractions, operator set-up, right-hand side, pressure solve, velocity correction), the
differentiable step (the same and the adjoint with its gradients), and the autograd Functions.
Grids run from 32^3 to 512^3, cubic and not, with rows that are and are not multiples of the
vector widths, in the three precisions and with both solver methods.

Fields are a liquid drop above a liquid film in gas (densities 998, 880 and 1.2, interfaces
smeared over 1.5 cells), the drop's place and size and the film's depth shifted a little by the
seed, random face velocities and normal loss weights.
"""
import math

import torch

from paper_2605_30082_gb300 import Solver
from paper_2605_30082_gb300.solver import PoissonSolve, PoissonSolveFractions

RHO_PHASE = [998.0, 880.0, 1.2]
SIGMA = 0.03
WIDTH = 1.5  # cells over which an interface is smeared

# kinds of work
#   project   density_from_fractions, set_density, rhs, solve, project: one time step
#   train     project, then adjoint and density_grads: one differentiable step; with csf, the
#             surface-tension term on both sides of the solve
#   fractions PoissonSolveFractions, forward and backward, with the surface-tension term
#   faces     PoissonSolve, forward and backward, on face coefficients


def _case(name, kind, dims, precision="mixed", inner=0, method="vcycle", coarsest=8, csf=False):
    c = {"kind": kind, "nx": dims[0], "ny": dims[1], "nz": dims[2], "precision": precision,
         "inner": inner, "method": method, "coarsest": coarsest, "csf": csf}
    return c if name is None else {"name": name, **c}


def listed():
    return [
        # the smallest configuration: a 32^3 test grid in plain FP64, all launches and latency
        _case("project_32_fp64", "project", (32, 32, 32), "fp64", 1, coarsest=4),
        # a small grid as in parameter studies and unit-sized blocks, default mixed solver
        _case("project_64_mixed", "project", (64, 64, 64)),
        # fitting fractions and surface tension through the solve on the 64^3 gradient-check grid
        _case("fractions_64_csf", "fractions", (64, 64, 64), inner=1, csf=True),
        # face coefficients from another code, sizes 8 x (9, 10, 11): rows of 36 and 18 cells per
        # colour, an odd coarsest level
        _case("faces_72x80x88", "faces", (72, 80, 88), inner=1),
        # one block of the paper's strong-scaling runs (128^3 cells per device)
        _case("project_128_mixed", "project", (128, 128, 128)),
        # a flat box: three different extents, differentiable step
        _case("train_224x160x96", "train", (224, 160, 96)),
        # the double-float outer loop
        _case("project_192_df", "project", (192, 192, 192), "mixed_df"),
        # conjugate gradients around the V-cycle, on a long box
        _case("project_256x128x192_fcg", "project", (256, 128, 192), inner=3, method="fcg"),
        # the 256^3 configurations: plain FP64, mixed, and the differentiable step with surface
        # tension (the 1024^3 configuration's terms at a size that fits several times)
        _case("project_256_fp64", "project", (256, 256, 256), "fp64", 1, coarsest=4),
        _case("project_256_mixed", "project", (256, 256, 256)),
        _case("train_256_csf", "train", (256, 256, 256), csf=True),
        # the headline workload: forward and adjoint at 512^3
        _case("train_512_mixed", "train", (512, 512, 512)),
    ]


def draw(rng):
    """A case of the same kinds on another grid: small odd multiples of a power of two."""
    kind = rng.choice(["project", "project", "project", "train", "train", "fractions", "faces"])
    precision = rng.choice(["mixed", "mixed", "mixed", "fp64", "mixed_df"]) if kind == "project" else "mixed"
    method = rng.choice(["vcycle", "vcycle", "vcycle", "fcg"]) if kind == "project" and precision == "mixed" else "vcycle"
    # cells: up to the largest listed case for the mixed V-cycle, less where a cell costs more
    top = 8e7 if kind in ("project", "train") and precision == "mixed" and method == "vcycle" else 1.7e7
    cells = math.exp(rng.uniform(math.log(32 ** 3), math.log(top)))
    base = [rng.randint(4, 9) for _ in range(3)]
    lev = max(3, round(math.log2((cells / (base[0] * base[1] * base[2])) ** (1 / 3))))
    dims = [v << lev for v in base]
    if dims[0] * dims[1] * dims[2] > 1.3e8:
        dims = [v >> 1 for v in dims]
    # the large ones with the adaptive cycle count and without the surface term, as the largest listed
    large = dims[0] * dims[1] * dims[2] > 3e7
    inner = 1 if precision == "fp64" else 3 if method == "fcg" else 0 if large else rng.choice([0, 0, 1, 2])
    csf = kind == "fractions" or (kind == "train" and not large and rng.random() < 0.3)
    return _case(None, kind, tuple(dims), precision, inner, method, rng.choice([4, 8]), csf)


def _spacing(case):
    return 1.0 / max(case["nx"], case["ny"], case["nz"])


def _inputs(case, seed, device):
    """Fractions, curvature, face velocities and loss weights of one seed."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    f8 = torch.float64
    g = torch.Generator(device="cpu").manual_seed(2 * seed + 1)
    jit = (torch.rand(5, generator=g, dtype=f8) * 2 - 1).tolist()
    m = min(nx, ny, nz)
    c = [nx / 2 + jit[0] * nx / 16, ny / 2 + jit[1] * ny / 16, 5 * nz / 8 + jit[2] * nz / 32]
    radius = m / 4 * (1 + jit[3] / 16)
    zfilm = 3 * nz / 16 * (1 + jit[4] / 16)

    def axis(n):
        return torch.arange(n, device=device, dtype=f8) + 0.5

    x2 = ((axis(nx) - c[0]) ** 2).view(1, 1, nx)
    y2 = ((axis(ny) - c[1]) ** 2).view(1, ny, 1)
    z2 = ((axis(nz) - c[2]) ** 2).view(nz, 1, 1)
    drop = (x2 + y2 + z2).sqrt_().sub_(radius).mul_(-1.0 / WIDTH).add_(0.5).clamp_(0.0, 1.0)
    film = (0.5 - (axis(nz) - zfilm) / WIDTH).clamp_(0.0, 1.0).view(nz, 1, 1)
    film = torch.minimum(film.expand(nz, ny, nx), 1.0 - drop).contiguous()
    gd = torch.Generator(device=device).manual_seed(2 * seed)
    u = []
    for q, sh in enumerate(((nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx))):
        a = torch.rand(sh, generator=gd, device=device, dtype=f8).mul_(2.0).sub_(1.0)
        a.select(2 - q, 0).zero_()
        a.select(2 - q, -1).zero_()
        u.append(a)
    out = {"fracs": [drop, film], "u": tuple(u)}
    if case["kind"] != "project":
        out["w"] = torch.randn((nz, ny, nx), generator=gd, device=device, dtype=f8)
    if case["csf"]:
        kappa = torch.zeros_like(drop)
        kappa.masked_fill_((drop > 0) & (drop < 1), 2.0 / (radius * _spacing(case)))
        out["kappa"] = kappa
    return out


def _density(fracs):
    rho = torch.full_like(fracs[0], RHO_PHASE[-1])
    for f, r in zip(fracs, RHO_PHASE):
        rho += (r - RHO_PHASE[-1]) * f
    return rho


def _faces(rho):
    """1 / harmonic mean on the interior faces, 0 on the walls: (bx, by, bz)."""
    s = 1.0 / rho
    nz, ny, nx = rho.shape
    bx, by, bz = (torch.zeros(sh, dtype=rho.dtype, device=rho.device)
                  for sh in ((nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx)))
    bx[:, :, 1:-1] = 0.5 * (s[:, :, 1:] + s[:, :, :-1])
    by[:, 1:-1] = 0.5 * (s[:, 1:] + s[:, :-1])
    bz[1:-1] = 0.5 * (s[1:] + s[:-1])
    return bx, by, bz


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    st = {"case": case, "in": _inputs(case, seed, dev)}
    st["solver"] = s = Solver((case["nx"], case["ny"], case["nz"]), h=_spacing(case), precision=case["precision"],
                              coarsest=case["coarsest"], inner_cycles=case["inner"], method=case["method"])
    if case["kind"] in ("project", "train"):
        # the arrays that a time loop keeps
        st["rho"], st["b"], st["p"] = s.empty_cells(), s.empty_cells(), s.empty_cells()
        st["u"] = tuple(torch.empty_like(a) for a in st["in"]["u"])
    if case["kind"] == "train":
        st["lam"], st["drho"] = s.empty_cells(), s.empty_cells()
        st["dfrac"] = [s.empty_cells() for _ in st["in"]["fracs"]]
    if case["kind"] in ("fractions", "faces"):
        st["b"] = s.rhs(u=st["in"]["u"])
        if case["kind"] == "faces":
            st["faces"] = _faces(_density(st["in"]["fracs"]))
        else:
            st["csf"] = s.csf_faces(st["in"]["fracs"][0], st["in"]["kappa"])
    return st


def run(state):
    case, s, a = state["case"], state["solver"], state["in"]
    if case["kind"] == "fractions":
        b = state["b"].detach().requires_grad_()
        fr = [f.detach().requires_grad_() for f in a["fracs"]]
        sig = torch.tensor(SIGMA, dtype=torch.float64, requires_grad=True)
        p = PoissonSolveFractions.apply(s, b, RHO_PHASE, sig, state["csf"], *fr)
        gr = torch.autograd.grad(p, [b, *fr, sig], a["w"])
        return {"p": p.detach(), "db": gr[0], "dfrac": list(gr[1:-1]), "dsigma": gr[-1]}
    if case["kind"] == "faces":
        b = state["b"].detach().requires_grad_()
        fc = [f.detach().requires_grad_() for f in state["faces"]]
        p = PoissonSolve.apply(s, b, *fc)
        gr = torch.autograd.grad(p, [b, *fc], a["w"])
        return {"p": p.detach(), "db": gr[0], "dbeta": list(gr[1:])}
    rho = s.density_from_fractions(a["fracs"], RHO_PHASE, out=state["rho"])
    s.set_density(rho)
    csf = s.csf_faces(a["fracs"][0], a["kappa"]) if case["csf"] else None
    sigma = SIGMA if case["csf"] else 0.0
    b = s.rhs(u=a["u"], csf=csf, sigma=sigma, out=state["b"])
    p = s.solve(b, state["p"])
    un = s.project(p, a["u"], csf=csf, sigma=sigma, out=state["u"])
    out = {"p": p, "u": list(un)}
    if case["kind"] == "train":
        lam, g, ds = s.adjoint(a["w"], p, csf=csf, sigma=sigma, lam=state["lam"])
        drho, dfrac = s.density_grads(rho, g, RHO_PHASE, out=(state["drho"], state["dfrac"]))
        out.update(lam=lam, dbeta=list(g), drho=drho, dfrac=dfrac)
        if case["csf"]:
            out["dsigma"] = ds
    return out


def work(case):
    """Inputs read once and outputs written once; the arithmetic of the solves' V-cycles (four
    red-black sweeps, a residual and two transfers per cycle on all levels, about 20 cycles to a
    relative residual of 1e-10) and of the passes around them."""
    n = case["nx"] * case["ny"] * case["nz"]
    cycle = 8 / 7 * (4 * 14 + 20)
    solves = 1 if case["kind"] == "project" else 2
    cell = {
        "project": 16 + 24 + 8 + 24,                            # fractions, u; p, corrected u
        "train": 16 + 24 + 8 + 8 + 24 + 8 + 12 + 8 + 16,        # and w; lam, dbeta, drho, dfrac
        "fractions": 16 + 8 + 24 + 8 + 8 + 8 + 16,              # fractions, b, csf, w; p, db, dfrac
        "faces": 24 + 8 + 8 + 8 + 8 + 12,                       # faces, b, w; p, db, dbeta
    }[case["kind"]]
    return {"bytes": n * (cell + (8 if case["csf"] and case["kind"] == "train" else 0)),
            "flops": n * (solves * 20 * cycle + 40)}


# ---- the same results in 64 bits, plain torch --------------------------------------------------

def _div(u, h):
    return ((u[0][:, :, 1:] - u[0][:, :, :-1]) + (u[1][:, 1:] - u[1][:, :-1]) + (u[2][1:] - u[2][:-1])) / h


def _grad(p, h):
    """(p_R - p_L) / h on the interior faces, 0 on the walls."""
    g = [torch.zeros((p.shape[0], p.shape[1], p.shape[2] + 1), dtype=p.dtype, device=p.device),
         torch.zeros((p.shape[0], p.shape[1] + 1, p.shape[2]), dtype=p.dtype, device=p.device),
         torch.zeros((p.shape[0] + 1, p.shape[1], p.shape[2]), dtype=p.dtype, device=p.device)]
    g[0][:, :, 1:-1] = (p[:, :, 1:] - p[:, :, :-1]) / h
    g[1][:, 1:-1] = (p[:, 1:] - p[:, :-1]) / h
    g[2][1:-1] = (p[1:] - p[:-1]) / h
    return g


def _cg(beta, rhs, h):
    """Zero-mean solution of -div(beta grad p) = rhs - mean: conjugate gradients with the diagonal as
    preconditioner, to a relative residual of 1e-13."""
    dg = ((beta[0][:, :, 1:] + beta[0][:, :, :-1]) + (beta[1][:, 1:] + beta[1][:, :-1])
          + (beta[2][1:] + beta[2][:-1])) / (h * h)
    r = rhs - rhs.mean()
    n0 = float(r.norm())
    x = torch.zeros_like(r)
    z = r / dg
    d = z.clone()
    rz = (r * z).sum()
    for it in range(20000):
        q = -_div([bf * gf for bf, gf in zip(beta, _grad(d, h))], h)
        al = rz / (d * q).sum()
        x += al * d
        r -= al * q
        if it % 50 == 49 and float(r.norm()) <= 1e-13 * n0:
            break
        z = r / dg
        rz, old = (r * z).sum(), rz
        d = z + (rz / old) * d
    return x - x.mean()


def exact(case, seed):
    if case["nx"] * case["ny"] * case["nz"] > 2.2e6:
        return None  # the plain iteration takes too long there
    a = _inputs(case, seed, torch.device("cuda", torch.cuda.current_device()))
    h = _spacing(case)
    rho = _density(a["fracs"])
    beta = _faces(rho)
    csf = None
    if case["csf"]:
        f, k = a["fracs"][0], a["kappa"]
        csf = _grad(f, h)
        csf[0][:, :, 1:-1] *= 0.5 * (k[:, :, 1:] + k[:, :, :-1])
        csf[1][:, 1:-1] *= 0.5 * (k[:, 1:] + k[:, :-1])
        csf[2][1:-1] *= 0.5 * (k[1:] + k[:-1])
    b = _div(a["u"], h)
    if csf is not None:
        b = b + SIGMA * _div([bf * cf for bf, cf in zip(beta, csf)], h)
    p = _cg(beta, b, h)
    gp = _grad(p, h)
    out = {"p": p}
    if case["kind"] in ("project", "train"):
        out["u"] = [uf + bf * (gf + (SIGMA * cf if csf is not None else 0.0))
                    for uf, bf, gf, cf in zip(a["u"], beta, gp, csf or gp)]
        if case["kind"] == "project":
            return out
    lam = _cg(beta, a["w"], h)
    gl = _grad(lam, h)
    dbeta = [-x * y for x, y in zip(gl, gp)]
    if csf is not None:
        dbeta = [v - SIGMA * cf * x for v, cf, x in zip(dbeta, csf, gl)]
    dsigma = -sum(float((bf * cf * x).sum()) for bf, cf, x in zip(beta, csf, gl)) if csf is not None else None
    drho = -((dbeta[0][:, :, 1:] + dbeta[0][:, :, :-1]) + (dbeta[1][:, 1:] + dbeta[1][:, :-1])
             + (dbeta[2][1:] + dbeta[2][:-1])) / (2 * rho * rho)
    dfrac = [drho * (r - RHO_PHASE[-1]) for r in RHO_PHASE[:-1]]
    if case["kind"] == "fractions":
        return {"p": p, "db": lam, "dfrac": dfrac, "dsigma": torch.tensor(dsigma, dtype=torch.float64)}
    if case["kind"] == "faces":
        return {"p": p, "db": lam, "dbeta": dbeta}
    out.update(lam=lam, dbeta=dbeta, drho=drho, dfrac=dfrac)
    if csf is not None:
        out["dsigma"] = dsigma
    return out
