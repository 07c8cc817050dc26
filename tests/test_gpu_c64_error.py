"""The complex64 sweep on the FP32 pipes is no less accurate than the tensor-core form of the
same factorisation: the residual that PWQT_FP32 reports, geometric mean over 8 energies,
against what the tensor-core form left on the same systems (the figures below), where long
running sums would lose most."""
import numpy as np
import pytest

from paper_1903_00548_gb300 import workloads as W

pytestmark = pytest.mark.gpu

E0 = W.RIBBON13_G30_E64
# bands, nodes, energies from .. to, residual of the tensor-core form
CASES = [(64, 40, 1.5, 2.8, 9.32e-6), (75, 20, 1.5, 2.8, 3.71e-6), (100, 12, 0.0, 0.9, 3.05e-6),
         (128, 12, E0 - 0.05, E0 + 0.9, 8.43e-6), (160, 12, E0 - 0.05, E0 + 0.9, 9.31e-6)]


@pytest.mark.parametrize("n_bands,n_nodes,lo,hi,bound", CASES)
def test_complex64_residual(n_bands, n_nodes, lo, hi, bound):
    from paper_1903_00548_gb300 import build, pwqt as pw
    build.build()
    wl = W.ribbon512()
    ctx = pw.Context()
    ctx.assemble_intrinsic(wl.cell, wl.ff, wl.gcut, n_bands)
    U = W.random_smooth(n_nodes, 0.2, 3)
    U = U - np.linspace(U[0], U[-1], n_nodes)
    U[0] = U[-1] = 0.0
    ctx.set_extrinsic(0, U)
    r = ctx.solve(0, W.midpoint_grid(lo, hi, 8), pw.FP32)
    assert np.all(r.status & (pw.ST_MODE_COUNT | pw.ST_SINGULAR_PIVOT) == 0)
    assert np.exp(np.mean(np.log(r.resid))) <= bound
