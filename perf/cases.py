"""What this framework is timed on: the calls of include/pwqt.h as a user's program makes
them, over the range of block sizes, device lengths and energy counts that it is used for.

A program holds one context per structure, with the contact self-energies of its energy
grid in the context's cache, and solves it for one potential after another (bias points,
self-consistent iterations, requests).  So `prepare` takes the context of the case's
structure, gives it a potential made from the seed and fills the cache; `run` is one call
on that system.  The structures are the ones of paper_1903_00548_gb300.workloads: the
chain, the 0.5 nm ribbon of the small systems, and the 13 nm ribbon at the block sizes of
the serving catalog and between them.
"""
import math
import weakref

import numpy as np

from paper_1903_00548_gb300 import pwqt as pw
from paper_1903_00548_gb300 import workloads as W

PRECISION = {"fp64": pw.FP64, "mixed": pw.MIXED}
MU, KT = 0.05, 0.025852          # contact potential difference and temperature (eV) of the integrals


# ----------------------------------------------------------------------------- the cases
def listed():
    return [
        # one resonance scan of the 20-node chain: the smallest blocks, all launches and latency
        dict(name="chain6_fp64_64E", kind="solve", structure="chain", bands=3, nodes=20, energies=64, precision="fp64"),
        # the chain's ballistic current by adaptive quadrature: rounds of small batched solves
        dict(name="chain6_current", kind="integrate", structure="chain", bands=3, nodes=20, tol=1e-11),
        # a new structure from its atoms to T(E): basis, blocks, contacts and solve
        dict(name="cold_ribbon24_4E", kind="cold", structure="narrow", bands=12, nodes=24, energies=4, precision="fp64"),
        # a block size that no tile divides, few energies
        dict(name="ribbon70_fp64_5E", kind="solve", structure="wide", bands=35, nodes=31, energies=5, precision="fp64"),
        # node spectral density from the recursive Green's function
        dict(name="ribbon64_green_4E", kind="green", structure="wide", bands=32, nodes=24, energies=4),
        # a small request of the serving catalog
        dict(name="ribbon64_mixed_8E", kind="solve", structure="wide", bands=32, nodes=100, energies=8, precision="mixed"),
        # an FP64 reference run of a medium block
        dict(name="ribbon128_fp64_16E", kind="solve", structure="wide", bands=64, nodes=50, energies=16, precision="fp64"),
        # n(r): density matrix accumulated over an energy grid, then put on the real-space grid
        dict(name="ribbon128_density_16E", kind="density", structure="wide", bands=64, nodes=50, energies=16,
             precision="mixed", nx=64, nz=16),
        # a large request of the serving catalog's medium block
        dict(name="ribbon128_mixed_32E", kind="solve", structure="wide", bands=64, nodes=200, energies=32, precision="mixed"),
        # FP64 verification of a few energies at a large block
        dict(name="ribbon256_fp64_4E", kind="solve", structure="wide", bands=128, nodes=12, energies=4, precision="fp64"),
        # energies x bias points of one device in one call
        dict(name="ribbon256_bias4_8E", kind="multi", structure="wide", bands=128, nodes=100, energies=8, bias=4,
             precision="mixed"),
        # the block-512 workload: half of a step's energies on a 100-node device
        dict(name="ribbon512_mixed_16E", kind="solve", structure="wide", bands=256, nodes=100, energies=16, precision="mixed"),
    ]


def _spread(rng, lo, hi):
    """A whole number between lo and hi, uniform over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["chain", "integrate", "cold", "fp64", "green", "mixed", "mixed", "mixed", "multi", "density"])
    if kind == "chain":
        return dict(kind="solve", structure="chain", bands=rng.randint(2, 3), nodes=_spread(rng, 3, 60),
                    energies=_spread(rng, 1, 100), precision="fp64")
    if kind == "integrate":
        return dict(kind="integrate", structure="chain", bands=rng.randint(2, 3), nodes=rng.randint(8, 40),
                    tol=10.0 ** -rng.randint(9, 11))
    if kind == "cold":
        return dict(kind="cold", structure="narrow", bands=rng.randint(8, 12), nodes=rng.randint(3, 40),
                    energies=rng.randint(1, 8), precision="fp64")
    if kind in ("fp64", "green"):
        bands = _spread(rng, 16, 128 if kind == "fp64" else 64)
        most = int((1.1e8 if kind == "fp64" else 2.5e7) / (2 * bands) ** 3)      # node count of about a second
        case = dict(kind="solve" if kind == "fp64" else "green", structure="wide", bands=bands,
                    nodes=_spread(rng, 3, max(4, min(200, most))), energies=_spread(rng, 1, 16))
        return dict(case, precision="fp64") if kind == "fp64" else case
    if kind == "multi":
        bands = _spread(rng, 32, 128)
        return dict(kind="multi", structure="wide", bands=bands, nodes=rng.randint(20, 100), energies=rng.randint(2, 6),
                    bias=rng.randint(2, 4), precision="mixed")
    if kind == "density":
        bands = _spread(rng, 24, 72)
        return dict(kind="density", structure="wide", bands=bands, nodes=rng.randint(10, 50), energies=rng.randint(2, 16),
                    precision="mixed", nx=rng.randint(20, 64), nz=rng.randint(6, 16))
    bands = 256 if rng.random() < 0.15 else _spread(rng, 16, 160)      # the block-512 workload, or a smaller block
    return dict(kind="solve", structure="wide", bands=bands, nodes=_spread(rng, 10, 200 if bands < 128 else 100),
                energies=_spread(rng, 1, 32 if bands < 128 else 12), precision="mixed")


# ----------------------------------------------------------------------------- inputs
def _structure(case):
    """(cell, form factor, plane-wave cutoff)"""
    if case["structure"] == "chain":
        return W.chain_cell(0.4), W.FormFactor(), W.chain8().gcut
    if case["structure"] == "narrow":
        return W.armchair_ribbon_cell(W.ribbon_lines_for_width(0.5)), W.FormFactor(), 28.0
    return W.armchair_ribbon_cell(W.ribbon_lines_for_width(13.0)), W.FormFactor(), 30.0


def _energies(case):
    """Injection energies inside the bands that the basis holds, where its complex64 factors refine
    (some bases have energies higher up where they do not)."""
    b = case["bands"]
    if case["structure"] == "chain":
        lo, hi = 0.0, 2.0
    elif case["structure"] == "narrow":
        lo, hi = 0.2, 2.4
    elif b < 32:
        lo, hi = -1.0, 0.0
    elif 64 <= b < 96:
        lo, hi = 1.5, 2.8
    elif b < 128 or b > 160:
        lo, hi = 0.0, 0.9
    else:
        lo, hi = W.RIBBON13_G30_E64 - 0.05, W.RIBBON13_G30_E64 + 0.9
    return W.midpoint_grid(lo, hi, case["energies"])


def _potentials(case, seed):
    """Node potentials made from the seed: one, or one per bias point."""
    rng = np.random.default_rng(seed)
    U = W.random_smooth(case["nodes"], float(rng.uniform(0.15, 0.3)), int(rng.integers(1 << 30)))
    return [U + W.linear_drop(case["nodes"], 0.05 * q) for q in range(case.get("bias", 1))]


def _weights(case):
    E = _energies(case)
    return np.full(len(E), E[1] - E[0] if len(E) > 1 else 0.01), float(np.mean(E))


_context = {}      # the context of the structure in use: one, and the states' own references


class State:
    """A program's handle: the context of its structure and the systems it put there."""

    def __init__(self, case, seed):
        key = (case["structure"], case["bands"], case["kind"] == "cold")
        held = _context.get(key)
        if held is None:
            _context.clear()
            held = (pw.Context(), list(range(63, -1, -1)))
            if case["kind"] != "cold":
                held[0].assemble_intrinsic(*_structure(case), case["bands"])
            _context[key] = held
        self.ctx, free = held
        self.case, self.U = case, _potentials(case, seed)
        self.systems = [free.pop() for _ in self.U]
        weakref.finalize(self, free.extend, list(self.systems)).atexit = False
        self.E = _energies(case) if "energies" in case else None
        if case["kind"] != "cold":
            for s, U in zip(self.systems, self.U):
                self.ctx.set_extrinsic(s, U)
                if self.E is not None:
                    self.ctx.prepare_leads(s, self.E[:1])      # the solver's first use of a block size, alone
                    self.ctx.prepare_leads(s, self.E)


def prepare(case, seed):
    return State(case, seed)


# ----------------------------------------------------------------------------- one pass
def _table(T, R, T_ds):
    """The transport coefficients of the energies, in channels: one row each, T, R and T_ds."""
    return np.stack([T, R, T_ds], axis=1)


def _result(r):
    # the solver's own notes on its way there (residual reached, correction steps) are no result
    return dict(transport=_table(r.T, r.R, r.T_ds), n_open=r.n_open, node_n=r.node_n, status=r.status)


def run(state):
    case, ctx, s = state.case, state.ctx, state.systems[0]
    kind = case["kind"]
    if kind == "solve":
        return _result(ctx.solve(s, state.E, PRECISION[case["precision"]]))
    if kind == "multi":
        return [_result(r) for r in ctx.solve_multi(state.systems, state.E, PRECISION[case["precision"]])]
    if kind == "cold":
        ctx.assemble_intrinsic(*_structure(case), case["bands"])
        ctx.set_extrinsic(s, state.U[0])
        return _result(ctx.solve(s, state.E, PRECISION[case["precision"]]))
    if kind == "green":
        dos, _, status = ctx.green_diagonal(s, state.E)
        return dict(node_dos=dos, status=status)
    if kind == "density":
        w, mu = _weights(case)
        ctx.density_reset(s)
        status = ctx.accumulate_density(s, state.E, w, mu, mu - MU, KT, PRECISION[case["precision"]])
        return dict(n_r=ctx.density_grid(s, case["nx"], case["nz"]), status=status)
    # the current, with the quadrature that gave it (the error estimate is the rule's own note)
    I, _, evals, x, w = ctx.integrate(s, pw.INTEGRAND_CURRENT, 0.02, 1.2, 0.8, 0.8 - MU, KT, case["tol"])
    return dict(current=I, evals=evals, x=x, w=w)


def work(case):
    """Block LU of the N nodes (complex LU, solve for X_i, Schur product: 56/3 n^3 real flops a
    node); the node blocks read once, the node densities and transmissions written."""
    n, N = 2 * case["bands"], case["nodes"]
    nE = case.get("energies", 300) * case.get("bias", 1)
    per_node = {"green": 51.0}.get(case["kind"], 56.0 / 3.0) * n ** 3
    flops = per_node * N * nE
    nbytes = 16.0 * n * n * (2 * N * case.get("bias", 1) + 2 + 2 * nE) + 8.0 * nE * (2 * N + 3)
    if case["kind"] == "density":
        flops += 12.0 * n * n * (0.6 * n) * N * nE + 24.0 * n * n * case["nx"] * case["nz"] * N
        nbytes += 8.0 * (N - 1) * case["nx"] * case["nz"]
    return {"bytes": nbytes, "flops": flops}


# ----------------------------------------------------------------------------- the same in plain numpy
HB2M = 0.0380998212      # hbar^2 / 2 m_e (eV nm^2)
G0 = 2.0 * 1.602176634e-19 ** 2 / 6.62607015e-34


def _bloch_waves(case):
    """Plane waves and the lowest Bloch waves at k = 0 and k = pi/Lz: [(k, Gx, Gz, C, eps)]."""
    cell, ff, gcut = _structure(case)
    bz, bx = 2 * math.pi / cell.Lz, 2 * math.pi / cell.Lx
    out = []
    for k in (0.0, math.pi / cell.Lz):
        mx = int(math.ceil(gcut / bx)) + 1 if cell.dim == 2 else 0
        mz = int(math.ceil((gcut + k) / bz)) + 1
        a, b = (g.ravel() for g in np.meshgrid(np.arange(-mx, mx + 1), np.arange(-mz, mz + 1), indexing="ij"))
        keep = (a * bx) ** 2 + (b * bz + k) ** 2 <= gcut ** 2 * (1 + 1e-14)
        a, b = a[keep], b[keep]
        Gx, Gz = a * bx, b * bz
        qx, qz = Gx[:, None] - Gx[None], Gz[:, None] - Gz[None]
        S = sum(np.exp(-1j * (qx * x + qz * z)) for x, z in cell.atoms)
        H = cell.omega0 / (cell.Lz * cell.Lx) * ff.v0 * np.exp(-(qx ** 2 + qz ** 2) / (2 * ff.sigma ** 2)) * S
        np.fill_diagonal(H, HB2M * (Gx ** 2 + (Gz + k) ** 2))
        eps, C = np.linalg.eigh(H)
        out.append((k, a, b, C[:, :case["bands"]], eps[:case["bands"]]))
    return cell, out


def _blocks(case):
    """Node blocks H0, H1, M0, M1 and the six potential weights from closed-form element integrals."""
    cell, groups = _bloch_waves(case)
    L, nb = cell.Lz, case["bands"]
    n = 2 * nb
    S, R = np.zeros((4, n, n), complex), np.zeros((n, n), complex)
    for ga, (ka, ax, az, Ca, _) in enumerate(groups):
        for gb, (kb, bx, bz, Cb, _) in enumerate(groups):
            same = ax[:, None] == bx[None]
            nu = 2 * (bz[None] - az[:, None]) + (gb - ga)
            q = nu * math.pi / L
            e = np.where(nu % 2 == 0, 1.0, -1.0)
            iq = 1j * np.where(nu == 0, 1.0, q)
            J = [np.where(nu == 0, L, (e - 1) / iq)]
            for p in (1, 2, 3):
                J.append(np.where(nu == 0, L ** (p + 1) / (p + 1), (L ** p * e - p * J[-1]) / iq))
            at = np.s_[ga * nb:(ga + 1) * nb, gb * nb:(gb + 1) * nb]
            for p in range(4):
                S[(p,) + at] = Ca.conj().T @ (same * J[p]) @ Cb
            Q = 2 * math.pi / L * (az[:, None] + bz[None]) + ka + kb
            R[at] = Ca.conj().T @ (same * J[0] * Q) @ Cb
    S, R = S * cell.Lx, R * cell.Lx
    s0, s1, s2, s3 = S[0], S[1] / L, S[2] / L ** 2, S[3] / L ** 3
    ph = np.repeat([1.0, -1.0], nb)
    rr, lr = ph[:, None] * ph[None], ph[None] * np.ones((n, 1))
    eps = np.concatenate([g[4] for g in groups])
    ee = 0.5 * (eps[:, None] + eps[None])
    Mll, Mlr, Mrr = s0 - 2 * s1 + s2, s1 - s2, s2
    Kd, Kx = HB2M / L ** 2 * S[0], HB2M * (-S[0] / L ** 2 - 0.5j / L * R)
    M0, M1 = rr * Mrr + Mll, lr * Mlr
    H0, H1 = ee * Mll + Kd + rr * (ee * Mrr + Kd), lr * (ee * Mlr + Kx)
    Wt = [s0 - 3 * s1 + 3 * s2 - s3, lr * (s1 - 2 * s2 + s3), rr * (s2 - s3), s1 - 2 * s2 + s3, lr * (s2 - s3), rr * s3]
    return cell, groups, (H0, H1, M0, M1, Wt)


def _device(blk, U):
    H0, H1, _, _, Wt = blk
    N = len(U)
    D = [H0 + U[max(i - 1, 0)] * Wt[2] + U[i] * (Wt[5] + Wt[0]) + U[min(i + 1, N - 1)] * Wt[3] for i in range(N)]
    O = [H1 + U[i] * Wt[1] + U[i + 1] * Wt[4] for i in range(N - 1)]
    return D, O


def _contact(L, blk, E):
    """Self-energies, injection vectors and projections of both contacts at lead energy E."""
    H0, H1, M0, M1, _ = blk
    n = len(H0)
    K0, Kp = H0 - E * M0, H1 - E * M1
    Km, Z = Kp.conj().T, np.zeros((n, n))
    A, B = np.block([[K0, Km], [Kp, Z]]), np.block([[-Kp, Z], [Z, Kp]])
    mu, V = np.linalg.eig(np.linalg.solve(A + B, A - B))
    lam = (1 + mu) / (1 - mu)
    C = V[n:] / np.linalg.norm(V[n:], axis=0)
    trav, vel = np.abs(np.abs(lam) - 1) < 1e-4, np.zeros(2 * n)
    for j in np.flatnonzero(trav):
        k, x, done = np.angle(lam[j]), C[:, j], False
        for _ in range(8):
            p = np.exp(1j * k)
            Hk, Mk = H0 + H1 * p + H1.conj().T / p, M0 + M1 * p + M1.conj().T / p
            x = np.linalg.solve(Hk - E * Mk, Mk @ x)
            x /= np.linalg.norm(x)
            m = (x.conj() @ Mk @ x).real
            w = (x.conj() @ Hk @ x).real / m
            K = H1 - w * M1
            slope = -2 * (x.conj() @ (p * K) @ x).imag / m
            if abs(w - E) < 1e-12 * max(1.0, abs(E)):
                done = True
                break
            k -= (w - E) / slope
        trav[j] = done
        if done:
            lam[j], vel[j], C[:, j] = p, L * slope, x * math.sqrt(L / (2 * math.pi) / m)
    d = np.where(trav, vel > 0, np.abs(lam) < 1)
    sides = {}
    for side, out, K, lm in (("d", d, Kp, lam), ("s", ~d, Km, 1 / lam)):
        inj = trav & ~out
        Bm = C[:, out]
        Binv = np.linalg.inv(Bm)
        Sg = K @ (Bm * lm[out]) @ Binv
        sides[side] = dict(sigma=Sg, rhs=K @ (C[:, inj] * lm[inj]) - Sg @ C[:, inj], cin=C[:, inj], v_in=np.abs(vel[inj]),
                           P=Binv[trav[out]], v_out=np.abs(vel[out & trav]))
    return sides


def _solve(L, blk, dev, U, E, contacts):
    """Node coefficients of the injected modes at E: (c [N, n, m], source contact, drain contact)."""
    M0, M1 = blk[2], blk[3]
    D, O = dev
    N, n = len(D), len(M0)
    for e in (E - U[0], E - U[-1]):
        if e not in contacts:
            contacts[e] = _contact(L, blk, e)
    s, d = contacts[E - U[0]]["s"], contacts[E - U[-1]]["d"]
    ms, md = s["rhs"].shape[1], d["rhs"].shape[1]
    up = [E * M1 - O[i] for i in range(N - 1)]
    X, y = [], []
    for i in range(N):
        A = E * M0 - D[i] - (s["sigma"] if i == 0 else 0) - (d["sigma"] if i == N - 1 else 0)
        b = np.zeros((n, ms + md), complex)
        if i == 0:
            b[:, :ms] = s["rhs"]
        if i == N - 1:
            b[:, ms:] = d["rhs"]
        if i:
            lo = up[i - 1].conj().T
            A, b = A - lo @ X[-1], b - lo @ y[-1]
        r = np.linalg.solve(A, np.concatenate([up[i], b], axis=1) if i < N - 1 else b)
        X.append(r[:, :n] if i < N - 1 else None)
        y.append(r[:, n:] if i < N - 1 else r)
    for i in range(N - 2, -1, -1):
        y[i] = y[i] - X[i] @ y[i + 1]
    return np.array(y), s, d


def _observe(c, s, d):
    ms = s["rhs"].shape[1]
    v = np.concatenate([s["v_in"], d["v_in"]])
    T = np.sum(np.abs(d["P"] @ c[-1][:, :ms]) ** 2 * d["v_out"][:, None] / v[:ms])
    back = np.abs(s["P"] @ (c[0] - np.pad(s["cin"], ((0, 0), (0, c.shape[2] - ms))))) ** 2 * s["v_out"][:, None] / v
    dens = np.sum(np.abs(c) ** 2, axis=1) * 2 / v
    return T, back[:, :ms].sum(), back[:, ms:].sum(), np.stack([dens[:, :ms].sum(1), dens[:, ms:].sum(1)], axis=1)


def _exact_results(L, blk, U, Es, contacts):
    dev = _device(blk, U)
    got = [_observe(*_solve(L, blk, dev, U, float(E), contacts)) for E in Es]
    T, R, T_ds, node_n = (np.array([g[q] for g in got]) for q in range(4))
    return dict(transport=_table(T, R, T_ds), n_open=None, node_n=node_n, status=None)


def _exact_green(L, blk, U, Es):
    M0, M1 = blk[2], blk[3]
    D, O = _device(blk, U)
    N, dos = len(U), []
    for E in Es:
        s, d = _contact(L, blk, E - U[0])["s"], _contact(L, blk, E - U[-1])["d"]
        A = [E * M0 - D[i] - (s["sigma"] if i == 0 else 0) - (d["sigma"] if i == N - 1 else 0) for i in range(N)]
        up = [E * M1 - O[i] for i in range(N - 1)]
        g, G = [], None
        for i in range(N):
            g.append(np.linalg.inv(A[i] - (up[i - 1].conj().T @ g[-1] @ up[i - 1] if i else 0)))
        row = np.zeros(N)
        for i in range(N - 1, -1, -1):
            G = g[i] if G is None else g[i] + g[i] @ up[i] @ G @ up[i].conj().T @ g[i]
            row[i] = -2 / math.pi * np.trace(G).imag
        dos.append(row)
    return dict(node_dos=np.array(dos), status=None)


def _exact_density(cell, groups, blk, U, case):
    nx, nz, L = case["nx"], case["nz"], cell.Lz
    bz, bx = 2 * math.pi / L, 2 * math.pi / cell.Lx
    x, z = np.arange(nx) * cell.Lx / nx, (np.arange(nz) + 0.5) * L / nz
    phi = np.concatenate([np.exp(1j * (a * bx * x[:, None, None] + (b * bz + k) * z[None, :, None])) @ C
                          for k, a, b, C, _ in groups], axis=2)
    ph = np.repeat([1.0, -1.0], case["bands"])
    left, right = phi * (1 - z / L)[None, :, None], phi * ph * (z / L)[None, :, None]
    w, mu = _weights(case)
    dev, contacts, N = _device(blk, U), {}, len(U)
    out = np.zeros((N - 1, nx, nz))
    for E, we in zip(_energies(case), w):
        c, s, d = _solve(L, blk, dev, U, float(E), contacts)
        f = [0.5 * (1 - math.tanh(0.5 * (E - m) / KT)) for m in (mu, mu - MU)]
        wt = we * np.concatenate([2 / s["v_in"] * f[0], 2 / d["v_in"] * f[1]])
        for e in range(N - 1):
            out[e] += np.abs(left @ c[e] + right @ c[e + 1]) ** 2 @ wt
    return dict(n_r=out, status=None)


def _exact_current(L, blk, U, tol):
    dev, contacts, seen = _device(blk, U), {}, {}
    lo, hi, ms, md = 0.02, 1.2, 0.8, 0.8 - MU

    def f(E):
        if E not in seen:
            T, _, T_ds, _ = _observe(*_solve(L, blk, dev, U, E, contacts))
            fd = [0.5 * (1 - math.tanh(0.5 * (E - m) / KT)) for m in (ms, md)]
            seen[E] = G0 * (T * fd[0] - T_ds * fd[1])
        return seen[E]

    total, wt = 0.0, {}
    todo = [(lo + (hi - lo) * k / 8, lo + (hi - lo) * (k + 1) / 8) for k in range(8)]
    while todo:
        a, b = todo.pop()
        h, m = b - a, a + (b - a) / 2
        xs = [a, a + (m - a) / 2, m, m + (b - m) / 2, b]
        fa, fl, fm, fr, fb = (f(x) for x in xs)
        S1, S2 = h / 6 * (fa + 4 * fm + fb), h / 12 * (fa + 4 * fl + 2 * fm + 4 * fr + fb)
        if abs(S2 - S1) <= 15 * tol * h / (hi - lo):
            total += S2 + (S2 - S1) / 15
            for x, c in zip(xs, (7, 32, 12, 32, 7)):
                wt[x] = wt.get(x, 0.0) + c * h / 90
        else:
            todo += [(a, m), (m, b)]
    return dict(current=np.array([total]), evals=None, x=np.array(sorted(wt)), w=np.array([wt[x] for x in sorted(wt)]))


def exact(case, seed):
    n, N, kind = 2 * case["bands"], case["nodes"], case["kind"]
    jobs = case.get("energies", 1) * case.get("bias", 1)
    if jobs * (n ** 3 * (4e-9 * 50 + 1e-10 * N * (12 if kind == "density" else 6)) + N * 2e-4) > 15:      # seconds, roughly
        return None
    Us = _potentials(case, seed)
    cell, groups, blk = _blocks(case)
    L, contacts = cell.Lz, {}
    if kind == "integrate":
        return _exact_current(L, blk, Us[0], case["tol"])
    if kind == "green":
        return _exact_green(L, blk, Us[0], _energies(case))
    if kind == "density":
        return _exact_density(cell, groups, blk, Us[0], case)
    got = [_exact_results(L, blk, U, _energies(case), contacts) for U in Us]
    return got if kind == "multi" else got[0]
