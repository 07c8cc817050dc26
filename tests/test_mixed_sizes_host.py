"""Whether the kept workspaces of the mixed path hold a call (host C++, no CUDA), compiled with
g++: over sequences of calls the answer is yes exactly when no buffer of either lane would
have to grow -- the slices' buffers of the residual among them -- and the solve asks for the
free memory whenever it is no."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1903_00548_gb300", "csrc")


def test_mixed_sizes_host(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = tmp_path / "mixed_sizes_test"
    subprocess.run([gxx, "-std=c++17", "-O1", "-Wall", "-I", CSRC, os.path.join(ROOT, "tests", "mixed_sizes_host_test.cpp"),
                    "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stderr + r.stdout
    assert "passed" in r.stdout


def test_solve_decides_by_it():
    with open(os.path.join(CSRC, "solve.cu")) as f:
        body = f.read()
    assert body.index("lanes_hold(") < body.index("cudaMemGetInfo")
