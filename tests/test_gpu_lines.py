"""The one-axis transform pass (all six transforms, every axis) against dense
transform matrices in 64 bits, on the grid sizes with one to sixteen lanes per
FFT, with and without the spectral weight, on fields that are and are not
aligned for vector accesses, and in place.

An FP32 transform of length N is about log2(N) + 4 roundings of 2^-24 deep and
its error is measured against the largest output: 1e-6 covers 16 of them."""
import numpy as np
import pytest

import kfbim_inputs as ki

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2303_04992_gb300 import MIXED, Solver, build  # noqa: E402

build()

TOL = 1e-6


def matrix(kind, N):
    """Transform matrices (output, input): 1 DCT-II, 3 DST-II, 5 DST-I; even numbers their inverses."""
    n, a = np.arange(N)[None, :], np.arange(N)[:, None]
    if kind in (1, 2):
        F = np.cos(np.pi * a * (n + 0.5) / N)
    elif kind in (3, 4):
        F = np.sin(np.pi * (a + 1) * (n + 0.5) / N)
    else:
        F = np.sin(np.pi * a * n / N)
    if kind % 2:
        return F
    if kind == 6:
        return 2.0 / N * F.T
    G = 2.0 / N * F.T
    G[:, 0 if kind == 2 else N - 1] *= 0.5
    return G


def weight(N, mode, wc, h, mu):
    """The spectral weights 1 Schur, 2 Poisson, 3 Schur right-hand side, as an [axis 0 = x] array."""
    a = np.arange(N)
    s = [4 * np.sin(np.pi * (a if b == wc else a + 1) / (2 * N)) ** 2 for b in range(3)]
    den = s[0][:, None, None] + s[1][None, :, None] + s[2][None, None, :]
    num = np.expand_dims(s[wc], tuple(b for b in range(3) if b != wc))
    if mode == 1:
        return num / den / mu
    w = h * h / mu / den if mode == 2 else -h * np.sqrt(num) / mu / den
    return np.where(num == 0, 0.0, w)


@pytest.fixture(scope="module", params=[32, 64, 96, 128, 256])
def solver(request):
    N = request.param
    s = Solver(ki.sphere(0.5 if N < 256 else 0.2), ki.grid(N), mu=0.7, precision=MIXED)
    yield s
    s.close()


@pytest.mark.parametrize("kind", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_transform_matches_dense(solver, kind, axis):
    N = solver.N
    for wmode, wc, off, inplace in ((0, 0, 0, False), (0, 0, 1, True), (2, (axis + 1) % 3, 0, False),
                                    (1 if kind < 5 else 3, axis, 1, False)):
        x = torch.randn(N ** 3 + 1, dtype=torch.float32, device="cuda",
                        generator=torch.Generator(device="cuda").manual_seed(17 * kind + axis))
        xin = x[off:off + N ** 3]
        want = xin.double().reshape(N, N, N).movedim(2 - axis, -1)   # [.., .., n] along the axis
        F = torch.from_numpy(matrix(kind, N)).cuda()
        want = (want @ F.T).movedim(-1, 2 - axis)
        if wmode:
            w = weight(N, wmode, wc, solver.h, solver.mu)
            want = want * torch.from_numpy(np.ascontiguousarray(w.transpose(2, 1, 0))).cuda()
        out = xin if inplace else torch.zeros(N ** 3 + 1, dtype=torch.float32, device="cuda")[off:off + N ** 3]
        solver.transform_f32(kind, axis, xin, out, backend=1, wmode=wmode, wc=wc)
        got = out.double().reshape(N, N, N)
        assert float((got - want).abs().max()) < TOL * float(want.abs().max()), (wmode, off)


@pytest.mark.parametrize("comp", [1, 2, 3])
def test_poisson_matches_dense(solver, comp):
    """The fused pass (DST-I, weight, inverse DST-I in one kernel) between plain FP64 passes: 1e-12, a few
    thousand roundings of the largest value."""
    N, c = solver.N, comp - 1
    r = torch.randn(N, N, N, dtype=torch.float64, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(comp))
    u = torch.zeros(N ** 3, dtype=torch.float64, device="cuda")
    solver.poisson(comp, r.reshape(-1), u)
    F = [torch.from_numpy(matrix(5 if a == c else 3, N)).cuda() for a in range(3)]
    B = [torch.from_numpy(matrix(6 if a == c else 4, N)).cuda() for a in range(3)]
    w = torch.from_numpy(np.ascontiguousarray(weight(N, 2, c, solver.h, 1.0).transpose(2, 1, 0))).cuda()
    v = torch.einsum("ck,bj,ai,kji->cba", F[2], F[1], F[0], r) * w
    want = torch.einsum("kc,jb,ia,cba->kji", B[2], B[1], B[0], v).reshape(-1)
    assert float((u - want).abs().max()) < 1e-12 * float(want.abs().max())
