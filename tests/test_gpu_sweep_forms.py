"""The block sweeps of both precisions on made-up systems, every form at the block sizes where
it changes: FP64 in one CTA (n <= 24), by cluster factorisation (26 .. 322) and the general kernel
(480); complex64 with one, two and four warps a panel, one and several rows a lane, ragged panels.
One, few and many energies, an odd number of columns, none from one contact.

sweep_forms_test.cpp calls the built library's sweeps.  Node blocks of condition below 3.5 whose
pivots lie off the diagonal.  Tolerance: elimination's backward error is about n u per unit of
growth, growth at most 2 here, forward and back: 3.5 x 2 x 2 n u, 20 n u with margin, of the
largest entry.  An exactly zero column of a node block sets PWQT_ST_SINGULAR_PIVOT at every energy
and leaves the solution finite; a NaN in the first node block leaves no entry finite."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_1903_00548_gb300")


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    from paper_1903_00548_gb300 import build
    build.build()
    out = str(tmp_path_factory.mktemp("forms") / "sweep_forms")
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-O2", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(PKG, "csrc"),
                    os.path.join(ROOT, "tests", "sweep_forms_test.cpp"), "-o", out, "-L", PKG, "-lpwqt", "-Xlinker", "-rpath=" + PKG],
                   check=True)
    return out


@pytest.mark.parametrize("n,nodes,ms,md,count", [(6, 4, 2, 1, 17), (24, 3, 5, 4, 3), (26, 3, 5, 4, 1), (26, 2, 0, 4, 17), (66, 3, 7, 0, 3),
                                                 (82, 3, 5, 4, 17), (130, 2, 9, 9, 2), (264, 2, 5, 4, 1), (320, 2, 5, 4, 3),
                                                 (322, 2, 5, 4, 1), (480, 2, 3, 2, 1)])
def test_sweep_forms(exe, n, nodes, ms, md, count):
    from paper_1903_00548_gb300 import pwqt as pw
    r = subprocess.run([exe, *map(str, (n, nodes, ms, md, count))], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    lines = [l.split() for l in r.stdout.splitlines()]
    assert [l[0] for l in lines] == (["fp64", "c64"] if 24 < n <= 320 else ["fp64"])
    for form, diff, status, zero_status, zero_bad, _, nan_bad, total in lines:
        u = 2.0 ** -53 if form == "fp64" else 2.0 ** -24
        assert float(diff) <= 20 * n * u, (form, diff)
        assert int(status) & pw.ST_SINGULAR_PIVOT == 0
        assert int(zero_status) & pw.ST_SINGULAR_PIVOT and int(zero_bad) == 0, form
        assert int(nan_bad) == int(total), form
