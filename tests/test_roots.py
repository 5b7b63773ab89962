"""The roots of unity of the transform tables (csrc/roots.h, plain C++) on the host.
Bound: the angle, pi / 4 at most, carries pi's and two more roundings (0.785 x 2.6e-16),
its sine and cosine at most 0.71 of that and one rounding of their own (0.55e-16):
2.0e-16."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
INC = os.path.join(os.path.dirname(HERE), "paper_2303_04992_gb300", "csrc")


def test_roots_match_long_double(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("g++ not found")
    exe = str(tmp_path / "roots_check")
    subprocess.run(["g++", "-std=c++17", "-O2", "-Wall", "-Wextra", "-Werror", "-I", INC,
                    os.path.join(HERE, "roots_check.cpp"), "-o", exe], check=True, capture_output=True, text=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=60).stdout
    got = {k: int(v) for k, v in (line.split() for line in out.splitlines())}
    assert got["bad"] == 0, got
    assert got["worst"] <= 2000, got
