"""Both precisions at the block sizes where their kernels change form: just above the
one-CTA FP64 form (n = 26), just above the complex64 panel factorisation's one-CTA limit
(n = 82), a ragged panel past two and four warps of panel rows (n = 66, 130), a block whose
panel rows take several registers a lane (n = 264), one past the FP32-pipe sweep (n = 322);
one energy, and enough that a mixed batch runs in two halves.  Flux conservation and
reciprocity at the FP64 path's 1e-9 of the open channels, the mixed path within its 1e-8 of
the FP64 path (absolute, times the open channels: both paths' bounds in test_gpu_parity)."""
import numpy as np
import pytest

from paper_1903_00548_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_bands,n_nodes,count", [(13, 7, 2), (33, 9, 17), (41, 6, 1), (65, 5, 17), (132, 4, 3), (161, 3, 1)])
def test_precisions_agree_at_block_size(n_bands, n_nodes, count):
    from paper_1903_00548_gb300 import build, pwqt as pw
    build.build()
    wl = W.ribbon512()
    lo, hi = (-1.0, -0.8) if n_bands < 32 else (0.0, 0.9)
    ctx = pw.Context()
    assert ctx.assemble_intrinsic(wl.cell, wl.ff, wl.gcut, n_bands) == 2 * n_bands
    ctx.set_extrinsic(0, W.random_smooth(n_nodes, 0.2, 7))
    E = W.midpoint_grid(lo, hi, count)
    r = ctx.solve(0, E, pw.FP64)
    m = ctx.solve(0, E, pw.MIXED)
    bad = pw.ST_MODE_COUNT | pw.ST_SINGULAR_PIVOT | pw.ST_IR_NO_CONVERGE
    assert np.all((r.status | m.status) & bad == 0), (r.status, m.status)
    assert np.max(r.resid) < 1e-11
    open_s = r.n_open[:, 0]
    assert np.all(open_s > 0)
    assert np.all(np.abs(r.T + r.R - open_s) <= 1e-9 * open_s) and np.all(np.abs(r.T - r.T_ds) <= 1e-9 * open_s)
    assert np.array_equal(m.n_open, r.n_open)
    for q in ("T", "R", "T_ds"):
        assert np.all(np.abs(getattr(m, q) - getattr(r, q)) <= 1e-8 * open_s), q
