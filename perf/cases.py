"""The work a user of the KFBI solver has it do, as cases that can be timed.

A case names one call of the public `Solver` binding on one geometry and grid:

  surface    the control-point stages alone: jumps of a density, trace of a
             velocity field, boundary pressure (jumps, trace, pressure_trace)
  poisson    one FP64 FFT Poisson solve on a face grid
  apply      one GMRES matvec of the boundary integral equation
  adjoint    one transposed matvec (gradients with respect to boundary data)
  interface  one interface solve with forcing: velocity and pressure fields
  solve      a whole solve: right-hand side, GMRES, final fields
  batch      several right-hand sides of one geometry in one call

The grids are the ones the library takes (16 to 256 and 96), the geometries and
physical constants those of the workloads, tests and benchmark of this
repository.  Whole solves run GMRES to 1e-12, so that the stopping point of the
iteration does not decide the last digits compared.
"""
import math

import numpy as np
import torch

import kfbim_inputs as ki
from paper_2303_04992_gb300 import FP64, MIXED, Solver

PRECISION = {"fp64": FP64, "mixed": MIXED}


def _case(name, op, geom, N, precision="mixed", **more):
    c = {"name": name, "op": op, "geom": geom, "N": N, "precision": precision, "lam": 0.0, "batch": 1,
         "size": 0.5, "shift": 0.0}
    c.update(more)
    return c


def listed():
    return [
        # the smallest calls: post-processing on the surface of a small problem (launch latency)
        _case("surface_sphere32", "surface", "sphere", 32, "fp64"),
        # a small problem's matvec: launches and host reads count
        _case("apply_sphere32", "apply", "sphere", 32),
        # the batch configuration's grids, one matvec each
        _case("apply_star64", "apply", "star", 64),
        _case("apply_star96", "apply", "star", 96),
        # the headline workload's matvec and its transpose
        _case("apply_star128", "apply", "star", 128),
        _case("adjoint_star128", "adjoint", "star", 128),
        # elasticity (Navier) on the rotated ellipsoid, forced interface solve
        _case("navier_ell128", "interface", "ellipsoid", 128, lam=2.0),
        # the largest grid: a small body in a 256^3 box
        _case("apply_sphere256", "apply", "sphere", 256, size=0.3),
        # everything in double precision
        _case("apply_star64_fp64", "apply", "star", 64, "fp64"),
        _case("poisson128_fp64", "poisson", "sphere", 128, "fp64", comp=1),
        # whole calls: the headline solve, and many right-hand sides at once
        _case("solve_star128", "solve", "star", 128),
        _case("batch8_star64", "batch", "star", 64, batch=8),
    ]


def draw(rng):
    op = rng.choice(["surface", "poisson", "apply", "apply", "apply", "adjoint", "interface", "solve", "batch"])
    geom = rng.choice(["sphere", "star", "ellipsoid"])
    grids = {"surface": [32, 64, 96, 128], "poisson": [16, 32, 64, 96, 128, 256],
             "apply": [16, 32, 64, 96, 128, 256], "adjoint": [32, 64, 96, 128],
             "interface": [32, 64, 96, 128, 256], "solve": [32, 64], "batch": [32, 64]}[op]
    N = rng.choice(grids)
    if N == 16 or N == 256 or op == "poisson":
        geom = "sphere"   # a coarse grid does not resolve the star; a small body on the finest
    precision = "mixed"
    if op in ("surface", "poisson"):
        precision = "fp64"
    elif N <= 64 and op in ("apply", "adjoint", "interface") and rng.random() < 0.25:
        precision = "fp64"
    c = _case("drawn", op, geom, N, precision)
    del c["name"]
    c["size"] = round(rng.uniform(0.2, 0.35) if N == 256 else rng.uniform(0.42, 0.55), 4)
    c["shift"] = round(rng.uniform(0.0, 0.05), 4)
    if op == "poisson":
        c["comp"] = rng.randint(1, 3)
    if op in ("apply", "interface", "solve") and geom != "star" and rng.random() < 0.3:
        c["lam"] = round(rng.uniform(0.5, 4.0), 3)
    if op == "batch":
        c["batch"] = rng.randint(2, 12 if N == 32 else 8)
    return c


# ------------------------------------------------------------------ inputs
def _geometry(case):
    s, d = case["size"], case["shift"]
    center = (d, -0.7 * d, 0.4 * d)
    if case["geom"] == "sphere":
        return ki.sphere(s, center)
    if case["geom"] == "star":
        return ki.star(s, 0.1, 3, 4, center)
    return ki.ellipsoid((1.2 * s, 0.9 * s, 0.7 * s), ki.seeded_rotation(3), center)


# A program keeps one solver per geometry and grid and calls it for every new
# right-hand side; the last few geometries' solvers are kept here.
_solvers = {}


def _solver(case):
    key = tuple((k, case[k]) for k in ("geom", "N", "precision", "lam", "size", "shift")) + (
        case["op"] in ("solve", "batch"),)
    if key not in _solvers:
        while len(_solvers) >= 2:
            _solvers.pop(next(iter(_solvers))).close()
        opts = {"gmres_tol": 1e-12} if key[-1] else {}
        _solvers[key] = Solver(_geometry(case), ki.grid(case["N"]), precision=PRECISION[case["precision"]],
                               lam=case["lam"] if case["lam"] > 0.0 else None, **opts)
    return _solvers[key]


def _smooth(rng, x, modes=4):
    """A sum of low-frequency waves at the points x (..., 3), on x's device."""
    out = torch.zeros(x.shape[:-1], dtype=torch.float64, device=x.device)
    for l in range(modes):
        k = rng.standard_normal(3) * (0.5 + l)
        amp, ph = rng.standard_normal() / (1.0 + l) ** 2, rng.uniform(0.0, 2.0 * math.pi)
        kv = torch.tensor(k, dtype=torch.float64, device=x.device)
        out += amp * torch.cos(x @ kv + ph)
    return out


def _grid_xyz(s, comp):
    """Node coordinates (N^3, 3) of face grid comp (1..3) or of the cells (0), x fastest."""
    ax = []
    for a in range(3):
        off = 0.0 if a == comp - 1 else 0.5
        ax.append(s.lo + (torch.arange(s.N, dtype=torch.float64, device="cuda") + off) * s.h)
    Z, Y, X = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
    return torch.stack([X, Y, Z], -1).reshape(-1, 3)


def _new(n):
    return torch.zeros(n, dtype=torch.float64, device="cuda")


def _poisson_rhs(case, seed):
    N = case["N"]
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    return torch.randn(N ** 3, dtype=torch.float64, device="cuda", generator=g)


def prepare(case, seed):
    s = _solver(case)
    op, N3 = case["op"], s.N ** 3
    st = {"op": op, "solver": s}
    rng = np.random.default_rng(int(seed))
    if op == "poisson":
        st.update(comp=case["comp"], r=_poisson_rhs(case, seed), u=_new(N3))
        return st
    xyz, comp, _, prim = s.points()
    x = torch.from_numpy(xyz).cuda()
    comp = torch.from_numpy(comp.astype(np.int64) - 1).cuda()
    prim = torch.from_numpy(prim).cuda()
    if op in ("solve", "batch"):
        # divergence-free boundary data: harmonic curl fields
        rows = np.arange(s.n_points)
        c0, p0 = comp.cpu().numpy(), prim.cpu().numpy()
        g = np.stack([ki.harmonic_curl_field(int(seed) * 64 + b)(xyz)[rows, c0][p0] for b in range(case["batch"])])
        st["g"] = torch.from_numpy(g).cuda()
        if op == "batch":
            st["phi"] = torch.zeros_like(st["g"])
            return st
        st.update(g=st["g"][0].contiguous(), phi=_new(s.n_primary))
    else:
        # a density: smooth, with the rough part that later Krylov vectors have
        vals = torch.stack([_smooth(rng, x) for _ in range(3)], -1)
        phi = vals.gather(1, comp[:, None])[:, 0][prim]
        g = torch.Generator(device="cuda").manual_seed(int(seed))
        st["phi"] = phi + 0.1 * torch.randn(phi.shape, dtype=torch.float64, device="cuda", generator=g)
    if op in ("apply", "adjoint"):
        st["out"] = _new(s.n_primary)
    if op in ("interface", "solve"):
        seeds = [np.random.default_rng([int(seed), c]) for c in range(3)]
        st["fpts"] = torch.cat([_smooth(r, x) for r in seeds])
        seeds = [np.random.default_rng([int(seed), c]) for c in range(3)]
        st["fgrid"] = torch.cat([_smooth(r, _grid_xyz(s, c + 1)) for c, r in enumerate(seeds)])
        st.update(u=_new(3 * N3), p=_new(N3))
    if op == "surface":
        st["u"] = torch.cat([_smooth(rng, _grid_xyz(s, c + 1)) for c in range(3)])
        st["p"] = _smooth(rng, _grid_xyz(s, 0))
        st.update(J=_new(12 * s.n_points), tr=_new(s.n_primary), ptr=_new(s.n_points))
    return st


def run(st):
    s, op = st["solver"], st["op"]
    if op == "surface":
        s.jumps(st["phi"], st["J"])
        s.trace(st["u"], st["J"], st["tr"])
        s.pressure_trace(st["p"], st["J"], st["ptr"])
        return [st["J"], st["tr"], st["ptr"]]
    if op == "poisson":
        return s.poisson(st["comp"], st["r"], st["u"])
    if op == "apply":
        return s.apply(st["phi"], st["out"])
    if op == "adjoint":
        return s.apply_adjoint(st["phi"], st["out"])
    if op == "interface":
        s.interface(st["phi"], st["u"], st["p"], st["fpts"], st["fgrid"])
        return [st["u"], st["p"]]
    if op == "solve":
        s.solve(st["g"], st["phi"], st["fpts"], st["fgrid"], st["u"], st["p"])
        return [st["phi"], st["u"], st["p"]]
    return s.solve_batch(st["g"], st["phi"])


# -------------------------------------------------------------------- work
def work(case):
    """Bytes: the surface tables (about 72 fit entries of 52 bytes and an
    11 x 18 jump map per control point, 18 pi r^2 / h^2 points), read once, and
    the FP64 grid fields that are inputs or outputs.  Flops: the one-axis real
    transforms (2.5 N^3 log2 N each) of the grid solve, 16 per Schur-CG
    iteration and 36 around a CG run, at the iteration counts the tolerances
    ask for."""
    N, op = case["N"], case["op"]
    N3, h = float(N) ** 3, 2.0 / N
    points = 18.0 * math.pi * case["size"] ** 2 / h ** 2
    tables = points * (72 * 52 + 11 * 18 * 8)
    xf = 2.5 * N3 * math.log2(N)
    solve_flops = (25 * 16 + 2 * 36) * xf
    if op == "surface":
        return {"bytes": tables + points * 8 * 40, "flops": points * (2 * 72 * 6 + 2 * 11 * 18 + 40)}
    if op == "poisson":
        return {"bytes": 16.0 * N3, "flops": 6 * xf}
    if op in ("apply", "adjoint"):
        return {"bytes": tables + 16.0 * points, "flops": solve_flops}
    if op == "interface":
        return {"bytes": tables + 8.0 * 7 * N3, "flops": solve_flops}
    matvecs = 40 * case["batch"]
    grid = 8.0 * 7 * N3 if op == "solve" else 0.0
    return {"bytes": matvecs * tables + grid, "flops": matvecs * 0.6 * solve_flops}


# ------------------------------------------------------------------- exact
def exact(case, seed):
    """The Poisson solve by dense sine matrices in 64 bits; the other calls
    have no value without the solver's own tables."""
    if case["op"] != "poisson":
        return None
    N = case["N"]
    h = 2.0 / N
    i = torch.arange(N, dtype=torch.float64, device="cuda")
    # modes across the wall-normal axis: sin(pi a i / N); along the others
    # sin(pi (a + 1)(i + 1/2) / N), the last mode with twice the norm
    S1 = torch.sin(math.pi * i[:, None] * i[None, :] / N)
    e1 = 4.0 * torch.sin(math.pi * i / (2 * N)) ** 2 / h ** 2
    S2 = torch.sin(math.pi * (i[:, None] + 1.0) * (i[None, :] + 0.5) / N)
    e2 = 4.0 * torch.sin(math.pi * (i + 1.0) / (2 * N)) ** 2 / h ** 2
    inv1 = (2.0 / N) * S1.T
    inv2 = (2.0 / N) * S2.T.clone()
    inv2[:, N - 1] *= 0.5
    ax = 3 - case["comp"]   # axis of the [k][j][i] array normal to the faces
    r = _poisson_rhs(case, seed).reshape(N, N, N).clone()
    r.select(ax, 0).zero_()
    fwd = [S1 if a == ax else S2 for a in range(3)]
    bwd = [inv1 if a == ax else inv2 for a in range(3)]
    lam = [e1 if a == ax else e2 for a in range(3)]
    v = torch.einsum("ak,bj,ci,kji->abc", fwd[0], fwd[1], fwd[2], r)
    d = lam[0][:, None, None] + lam[1][None, :, None] + lam[2][None, None, :]
    v = v / d
    v.select(ax, 0).zero_()
    v = torch.einsum("ka,jb,ic,abc->kji", bwd[0], bwd[1], bwd[2], v)
    return v.reshape(-1)
