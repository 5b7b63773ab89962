"""The term kernel of the FP32 Schur CG (one CTA per spectral term and plane)
and its z kernels on every grid they cover, with viscosities other than one and
the Navier block: the MIXED matvec on them against the same context kind on the
one-axis staged passes.  Both refine in FP64 to a relative residual of 1e-11
(1e-10 with the conditioning of the grid solve), whatever the FP32 operator's
rounding; an operator wrong in any mode would not let the refinement converge
within its sweeps."""
import numpy as np
import pytest

import kfbim_inputs as ki

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2303_04992_gb300 import MIXED, Solver, build  # noqa: E402

build()

XF_AUTO, XF_STAGED = 0, 3


@pytest.mark.parametrize("N,mu,lam", [(32, 1.0, None), (32, 0.3, 2.0), (64, 2.5, None), (96, 1.0, None),
                                      (96, 0.7, 1.5), (128, 0.4, 3.0)])
def test_matvec_on_the_term_kernel_matches_staged(N, mu, lam):
    got = {}
    for xf in (XF_AUTO, XF_STAGED):
        s = Solver(ki.sphere(0.47, (0.01, -0.02, 0.015)), ki.grid(N), mu=mu, lam=lam, precision=MIXED, transforms=xf)
        phi = torch.from_numpy(ki.random_density(s.n_primary, seed=N)).cuda()
        out = torch.zeros_like(phi)
        s.apply(phi, out)
        got[xf] = out.cpu().numpy()
        s.close()
    assert np.abs(got[XF_AUTO] - got[XF_STAGED]).max() < 1e-10 * np.abs(got[XF_STAGED]).max()
