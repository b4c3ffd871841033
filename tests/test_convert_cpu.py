"""The FP64 <-> FP32 pair conversions of the permutations, checked on the host.

Compiles tests/convert_check.cpp against
paper_2203_05665_gb300/csrc/h2_convert.hpp and runs it: every exponent with
significands around the rounding ties, zeros, subnormals, infinities and NaN,
and 8e6 random values.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_pair_conversions(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    exe = tmp_path / "convert_check"
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2203_05665_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "convert_check.cpp"), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
