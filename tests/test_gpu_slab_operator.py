"""The FP32 Schur operator of the slab CG on every grid it covers, seen without the
FP64 refinement that would correct it.

FP32 contexts stopped after four CG iterations: the pressure is then a fixed
polynomial of the operator applied to the right-hand side, and the slab form has to
agree with the one-axis staged form to FP32 rounding.  Every operator application is
six transforms deep, each about log2(N) + 4 <= 12 roundings of 2^-24: 4.3e-6 for one,
1.7e-5 for four in a row; 2e-5 of the largest value is allowed.  A mode wrong by
1e-3 of its weight would show as about 1e-3.

MIXED solves: where the FP32 operator is right, refinement sweeps and CG
iterations are those of the staged form, give or take the borderline sweep."""
import numpy as np
import pytest

import kfbim_inputs as ki

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2303_04992_gb300 import FP32, MIXED, Solver, build  # noqa: E402

build()

XF_AUTO, XF_STAGED = 0, 3
GRIDS = [(32, 1.0, None), (64, 0.3, 2.0), (96, 1.0, None), (96, 0.7, 1.5), (128, 2.5, None), (256, 1.0, None),
         (256, 0.7, 2.0)]


def body(N):
    return ki.sphere(0.47 if N < 256 else 0.2, (0.01, -0.02, 0.015))


@pytest.mark.parametrize("N,mu,lam", GRIDS)
def test_four_iterations_match_staged(N, mu, lam):
    got = {}
    for xf in (XF_AUTO, XF_STAGED):
        s = Solver(body(N), ki.grid(N), mu=mu, lam=lam, precision=FP32, transforms=xf, cg_max=4, inner_tol=1e-12)
        phi = torch.from_numpy(ki.random_density(s.n_primary, seed=N)).cuda()
        u = torch.zeros(3 * N ** 3, dtype=torch.float64, device="cuda")
        p = torch.zeros(N ** 3, dtype=torch.float64, device="cuda")
        s.interface(phi, u, p)
        got[xf] = (u, p)
        s.close()
    for a, b in zip(got[XF_AUTO], got[XF_STAGED]):
        assert float((a - b).abs().max()) < 2e-5 * float(b.abs().max())


@pytest.mark.parametrize("N,mu,lam", GRIDS)
def test_sweeps_and_iterations_match_staged(N, mu, lam):
    stats = {}
    for xf in (XF_AUTO, XF_STAGED):
        s = Solver(body(N), ki.grid(N), mu=mu, lam=lam, precision=MIXED, transforms=xf, gmres_tol=1e-3)
        g = torch.from_numpy(np.cos(np.arange(s.n_primary) * 0.01)).cuda()
        s.solve(g, torch.zeros_like(g))
        stats[xf] = s.last_stats
        s.close()
    a, b = stats[XF_AUTO], stats[XF_STAGED]
    assert a["gmres_iters"] == b["gmres_iters"]
    assert abs(a["refine_sweeps"] - b["refine_sweeps"]) <= 1
    # a borderline sweep is one run of at most about 30 iterations, and each run may stop one iteration apart
    assert abs(a["cg_iters"] - b["cg_iters"]) <= 30 + b["refine_sweeps"]
