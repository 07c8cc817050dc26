"""FP64 sweep at the edges of its three forms: blocks that one CTA carries through shared
memory (n <= 24), blocks just above that (tiles, cluster factorisation and column-block
solves with ragged last tiles), one and several energies (the cluster size and the column
blocks follow from both), and the shortest device.  T, R, T_ds and the node densities
against the oracle at the FP64 path's 1e-9 (relative to the open channels; node densities
1e-7, see test_gpu_parity), widened only by the oracle's own error bar; the reported
residual is the FP64 one."""
import numpy as np
import pytest

from oracle import pwqt_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pw():
    from paper_1903_00548_gb300 import build, pwqt
    build.build()
    return pwqt


@pytest.mark.parametrize("n_bands,n_nodes,count", [(8, 2, 1), (12, 5, 3), (13, 2, 1), (13, 5, 4), (17, 4, 2), (24, 3, 1)])
def test_fp64_sweep_forms_match_oracle(pw, n_bands, n_nodes, count):
    from tests.oracle_fixtures import small_ribbon_system
    s = small_ribbon_system(n_bands=n_bands, n_nodes=n_nodes, gcut=30.0)
    ctx = pw.Context()
    ctx.set_enhancement(s.basis.cell, s.basis.eps, [(g["mx"], g["mz"], g["C"]) for g in s.basis.groups])
    ctx.set_extrinsic(0, s.U)
    Es = np.linspace(0.35, 1.9, count) if count > 1 else np.array([0.6])
    r = ctx.solve(0, Es, pw.FP64)
    assert np.max(r.resid) < 1e-12
    cache = {}
    for e, E in enumerate(Es):
        ref = O.solve_energy(s.blk, s.Vd, s.Vu, s.U, float(E), cache=cache)
        alts = [O.solve_energy(s.blk, s.Vd, s.Vu, s.U, float(E), cache=cache, reciprocal=k) for k in (True, "cayley")]
        bar = max(O.error_bar(ref, *alts), O.perturbation_spread(s.blk, s.U, float(E)))
        t = max(1e-9 * max(1.0, ref.n_open_s), 4 * bar)
        assert tuple(r.n_open[e]) == (ref.n_open_s, ref.n_open_d)
        assert abs(r.T[e] - ref.T) <= t and abs(r.R[e] - ref.R) <= t and abs(r.T_ds[e] - ref.T_ds) <= t, (e, r.T[e], ref.T)
        if np.max(ref.node_n) > 0:
            assert np.max(np.abs(r.node_n[e] - ref.node_n)) <= 1e-7 * np.max(ref.node_n), e
    # several energies and one at a time take different cluster sizes and column blocks
    one = [ctx.solve(0, [E], pw.FP64) for E in Es]
    assert np.allclose([o.T[0] for o in one], r.T, rtol=1e-10, atol=1e-12)
