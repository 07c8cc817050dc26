"""The order of a process' contact fills (host C++, no CUDA) compiled with g++ and driven by
threads in the place of contexts: the first use of a block size is alone in the process, a
failed one is not counted, known sizes run side by side and do not starve a first use.  And
fill_leads passes through it once per process, not once per context, and for a single
missing entry too."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1903_00548_gb300", "csrc")


def test_first_use_is_alone(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = tmp_path / "first_use_test"
    subprocess.run([gxx, "-std=c++17", "-O1", "-pthread", "-Wall", "-I", CSRC,
                    os.path.join(ROOT, "tests", "first_use_host_test.cpp"), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stderr + r.stdout
    assert "passed" in r.stdout


def test_contact_fills_pass_through_it():
    with open(os.path.join(CSRC, "lead.cu")) as f:
        body = re.sub(r"//[^\n]*", "", f.read()).split("int fill_leads(")[1]
    gate = body.index("FirstUse::Pass")
    assert "static FirstUse" in body[:gate]                       # one for all contexts
    assert "miss.size() > 1" not in body[:body.index("std::thread> th")]
    assert gate < body.index("compute_lead_shared") and gate < body.index("init()")
