"""The reference norm |[f | g - mean(g)]|^2 of the MIXED refinement's stopping test
(k_rhs_moments), compiled from the kernel's source, against long-double sums: a large
constant with a small rest in g, a field that is zero away from a few cells, and the
Navier form.

Bounds.  The norm: |f|^2 sums squares of values rounded to FP32, 2^-23 relative; the
moments of g are FP64 sums of at most 2^20 values in blocks, 1e-11 relative after the
shift by g[0], whose rounding (1e5 + 1e-3 sin is a multiple of 2^-36, the shift exact)
adds nothing: 2e-7.  The mean: 1e-12."""
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2303_04992_gb300 import build as pkg_build  # noqa: E402
from paper_2303_04992_gb300.build import ARCH, SRC, _nvcc  # noqa: E402

pkg_build()
HERE = os.path.dirname(os.path.abspath(__file__))


def test_moments_match_long_double(tmp_path):
    exe = str(tmp_path / "moments_check")
    subprocess.run([_nvcc(), ARCH, "-O2", "-std=c++17", "-I", SRC, os.path.join(HERE, "moments_check.cu"), "-o", exe],
                   check=True, capture_output=True, text=True, timeout=300)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout
    got = {k: (float(m), float(r)) for k, m, r in (line.split() for line in out.splitlines())}
    assert len(got) == 6
    for name, (mean, ref) in got.items():
        assert mean < 1e-12, (name, mean)
        assert ref < 2e-7, (name, ref)
