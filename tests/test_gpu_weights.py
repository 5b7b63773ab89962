"""The spectral weight of a one-axis FP32 pass, digit for digit: a weighted pass
stores its unweighted output times (numerator times the correctly rounded
reciprocal of the summed eigenvalues), every step one rounding to nearest of
binary32, which numpy's float32 arithmetic reproduces on the host.  mu = 1, so
that the Schur weight's numerator is the table's entry itself."""
import numpy as np
import pytest

import kfbim_inputs as ki

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2303_04992_gb300 import MIXED, Solver, build  # noqa: E402

build()

SCHUR, POISSON = 1, 2


@pytest.fixture(scope="module", params=[32, 96, 128, 256])
def solver(request):
    N = request.param
    s = Solver(ki.sphere(0.5 if N < 256 else 0.2), ki.grid(N), precision=MIXED)
    yield s
    s.close()


def weight(N, mode, wc, axis, scale):
    """The pass's float32 weights as [z, y, x]: the eigenvalues of the two axes across the line are added first
    (lower axis first), then that of the axis itself."""
    a = np.arange(N)
    s = [(4 * np.sin(np.pi * (a if b == wc else a + 1) / (2 * N)) ** 2).astype(np.float32) for b in range(3)]
    s = [v.reshape([N if b == 2 - k else 1 for b in range(3)]) for k, v in enumerate(s)]
    lo, hi = [b for b in range(3) if b != axis]
    den = (s[lo] + s[hi]) + s[axis]
    r = (np.float32(1) / den).astype(np.float32)
    if mode == SCHUR:
        return s[wc] * r
    w = np.float32(scale) * r
    return np.where(s[wc] == 0, np.float32(0), w).astype(np.float32)


@pytest.mark.parametrize("kind,mode", [(1, SCHUR), (2, SCHUR), (5, POISSON), (6, POISSON)])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_weight_is_correctly_rounded(solver, kind, mode, axis):
    N = solver.N
    x = torch.randn(N ** 3, dtype=torch.float32, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(kind + 10 * axis))
    plain, got = torch.empty_like(x), torch.empty_like(x)
    solver.transform_f32(kind, axis, x, plain, backend=1)
    solver.transform_f32(kind, axis, x, got, backend=1, wmode=mode, wc=axis)
    w = weight(N, mode, axis, axis, solver.h * solver.h)
    want = (plain.cpu().numpy().reshape(N, N, N) * w).ravel()
    assert np.array_equal(got.cpu().numpy(), want)
