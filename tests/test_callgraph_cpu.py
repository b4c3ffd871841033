"""The bookkeeping of the graphs kept for repeated products, checked on the host with
driver calls that fail (tests/callgraph_check.cpp)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = "/usr/local/cuda/include"


def test_call_graph_bookkeeping(tmp_path):
    if shutil.which("g++") is None or not os.path.isdir(CUDA_INC):
        pytest.skip("needs g++ and the CUDA headers")
    exe = tmp_path / "callgraph_check"
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CUDA_INC,
                    "-I", os.path.join(ROOT, "paper_2203_05665_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "callgraph_check.cpp"), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
