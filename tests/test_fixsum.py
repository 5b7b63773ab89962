"""The integer sums of binary64 values behind the FP64 residual of the MIXED
refinement (csrc/fixsum.h, plain C++ for host and device), on the host: the
seven-point stencil sum within its truncations of 2^-57 of the largest value
(six neighbours and six times the centre: 12) beside the final rounding, closer
than the same sum in binary64; infinities, NaN, zeros, subnormals, overflow and
the conversion's carries."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "fixsum_check.cpp")
INC = os.path.join(os.path.dirname(HERE), "paper_2303_04992_gb300", "csrc")


def test_fixsum_matches_long_double(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("g++ not found")
    exe = str(tmp_path / "fixsum_check")
    subprocess.run(["g++", "-std=c++17", "-O2", "-Wall", "-Wextra", "-Werror", "-I", INC, SRC, "-o", exe],
                   check=True, capture_output=True, text=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=300).stdout
    got = {k: int(v) for k, v in (line.split() for line in out.splitlines())}
    assert got["n"] == 1000000
    assert got["worst_millionths"] <= 12_000_000, got
    assert got["worst_millionths"] < got["worst64_millionths"], got
    assert got["edges"] == 0 and got["carry"] == 0, got
