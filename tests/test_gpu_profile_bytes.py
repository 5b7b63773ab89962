"""The algorithmic bytes that kfbim_profile_kernels charges the slab CG's kernels with:
the values per launch that kfbim.h names, 9, 6, 6 and 2 N^3 floats; 3 for the last
kernel of a run that the host stopped with an update pending (d is read too)."""
import pytest

import kfbim_inputs as ki

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2303_04992_gb300 import FP32, MIXED, Solver, build  # noqa: E402

build()


def profiled_matvec(**opts):
    s = Solver(ki.sphere(), ki.grid(32), **opts)
    phi = torch.from_numpy(ki.random_density(s.n_primary, seed=3)).cuda()
    s.profile(True)
    s.apply(phi, torch.zeros_like(phi))
    got = s.profile_kernels()
    s.profile(False)
    s.close()
    return {k: got[k][2] / got[k][1] / (4 * 32 ** 3) for k in ("cg_zfwd", "cg_xy", "cg_zinv", "cg_update")}


def test_values_per_launch():
    assert profiled_matvec(precision=MIXED) == {"cg_zfwd": 9, "cg_xy": 6, "cg_zinv": 6, "cg_update": 2}


def test_pending_update_is_counted():
    assert profiled_matvec(precision=FP32, cg_max=4, inner_tol=1e-12)["cg_update"] == 3
