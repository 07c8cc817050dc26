// The block sweeps on made-up systems, called as the library calls them: argv = n, nodes, source
// columns, drain columns, energies.  For every form that the block size has (fp64: launch_sweep_fp64,
// c64: c64_sweep) three systems: a regular one (largest difference of the solution from dense
// elimination, over the largest entry), one whose first node block has an exactly zero column, and
// one with a NaN in it.  One line per form: name, difference, then for the zero column and the NaN
// the status bits and how many entries of the solution are not finite, and their number.
#include <algorithm>
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <vector>

#include "pwqt_internal.cuh"
#include "sweep_c64.cuh"
#include "sweep_common.cuh"

using namespace pwqt;
using C = std::complex<double>;
using V = std::vector<C>;

static void ok(cudaError_t e) { if (e != cudaSuccess) { std::printf("cuda: %s\n", cudaGetErrorString(e)); std::exit(1); } }
static void* up(const void* p, size_t bytes) {
    void* d = nullptr;
    ok(cudaMalloc(&d, bytes));
    if (p) ok(cudaMemcpy(d, p, bytes, cudaMemcpyHostToDevice));
    else ok(cudaMemset(d, 0, bytes));
    return d;
}

struct Made {
    int n, N, ms, md;
    V M0, M1, HV0, HV1, sig, rs, rd;
    std::vector<double> E;
};

// dense elimination with partial pivoting of [E M - H - Sigma] c = B, node by node in the result
static V dense(const Made& s, double E) {
    const int n = s.n, N = s.N, m = s.ms + s.md, d = n * N, w = d + m;
    V A((size_t)d * w);
    auto at = [&](int r, int c) -> C& { return A[(size_t)r * w + c]; };
    for (int i = 0; i < N; ++i)
        for (int r = 0; r < n; ++r)
            for (int c = 0; c < n; ++c) {
                const size_t q = (size_t)r * n + c;
                C v = E * s.M0[q] - s.HV0[(size_t)i * n * n + q];
                if (i == 0 || i == N - 1) v -= s.sig[q];
                at(i * n + r, i * n + c) = v;
                if (i + 1 < N) {
                    const C u = E * s.M1[q] - s.HV1[(size_t)i * n * n + q];
                    at(i * n + r, (i + 1) * n + c) = u;
                    at((i + 1) * n + c, i * n + r) = std::conj(u);
                }
            }
    for (int r = 0; r < n; ++r) {
        for (int g = 0; g < s.ms; ++g) at(r, d + g) = s.rs[(size_t)r * s.ms + g];
        for (int g = 0; g < s.md; ++g) at(d - n + r, d + s.ms + g) = s.rd[(size_t)r * s.md + g];
    }
    for (int j = 0; j < d; ++j) {
        int p = j;
        for (int r = j + 1; r < d; ++r)
            if (std::abs(at(r, j)) > std::abs(at(p, j))) p = r;
        for (int c = j; c < w && p != j; ++c) std::swap(at(j, c), at(p, c));
        const int hi = std::min(d, j + 2 * n);
        for (int r = j + 1; r < hi; ++r) {
            const C l = at(r, j) / at(j, j);
            if (l == C(0)) continue;
            for (int c = j + 1; c < w; ++c) {
                if (c == std::min(d, j + 3 * n)) c = d;      // zero past the band
                at(r, c) -= l * at(j, c);
            }
        }
    }
    V x((size_t)d * m);
    for (int j = d - 1; j >= 0; --j)
        for (int g = 0; g < m; ++g) {
            C v = at(j, d + g);
            for (int c = j + 1; c < std::min(d, j + 3 * n); ++c) v -= at(j, c) * x[(size_t)c * m + g];
            x[(size_t)j * m + g] = v / at(j, j);
        }
    return x;
}

struct Got { std::vector<V> x; std::vector<int> status; };

static Got solve(const Made& s, bool c64) {
    const int n = s.n, N = s.N, m = s.ms + s.md, nb = (int)s.E.size();
    const size_t nn = (size_t)n * n;
    SweepSys sys{n, N, (double2*)up(s.M0.data(), 16 * nn), (double2*)up(s.M1.data(), 16 * nn), (double2*)up(s.HV0.data(), 16 * nn * N),
                 (double2*)up(s.HV1.data(), 16 * nn * (N - 1))};
    auto* sig = (double2*)up(s.sig.data(), 16 * nn);
    auto* rs = (double2*)up(s.rs.data(), 16 * std::max<size_t>(s.rs.size(), 1));
    auto* rd = (double2*)up(s.rd.data(), 16 * std::max<size_t>(s.rd.size(), 1));
    auto* status = (int*)up(nullptr, sizeof(int) * nb);
    std::vector<SweepJob> jobs(nb);
    double2 *XY = nullptr, *S = nullptr;
    if (!c64) { XY = (double2*)up(nullptr, 16 * (size_t)nb * N * n * (n + m)); S = (double2*)up(nullptr, 16 * nn * nb); }
    for (int b = 0; b < nb; ++b) {
        SweepJob J{};
        J.E = s.E[b]; J.ms = s.ms; J.md = s.md;
        J.sig_s = J.sig_d = sig; J.rhs_s = rs; J.rhs_d = rd;
        if (!c64) { J.XY = XY + (size_t)b * N * n * (n + m); J.S = S + nn * b; }
        J.status = status + b;
        jobs[b] = J;
    }
    auto* jobs_d = (SweepJob*)up(jobs.data(), sizeof(SweepJob) * nb);
    Got g;
    g.x.assign(nb, V((size_t)N * n * m));
    g.status.resize(nb);
    if (!c64) {
        launch_sweep_fp64(sys, jobs_d, jobs.data(), nb, 0);
        ok(cudaGetLastError());
        V xy((size_t)nb * N * n * (n + m));
        ok(cudaMemcpy(xy.data(), XY, 16 * xy.size(), cudaMemcpyDeviceToHost));
        for (int b = 0; b < nb; ++b)
            for (size_t r = 0; r < (size_t)N * n; ++r)
                for (int q = 0; q < m; ++q) g.x[b][r * m + q] = xy[((size_t)b * N * n + r) * (n + m) + n + q];
    } else {
        const int w = n + m + (m & 1);
        C64Sweep cs{};
        cs.sys = sys; cs.jobs = jobs_d; cs.m = m; cs.w = w;
        cs.sF = cs.sL = (long long)N * nn; cs.sP = (long long)N * n; cs.sXY = (long long)N * n * w; cs.sC = (long long)N * n * m;
        cs.F = (float2*)up(nullptr, 8 * (size_t)cs.sF * nb);
        cs.Lb = (float2*)up(nullptr, 8 * (size_t)cs.sL * nb);
        cs.XY = (float2*)up(nullptr, 8 * (size_t)cs.sXY * nb);
        cs.perm = (int*)up(nullptr, sizeof(int) * (size_t)cs.sP * nb);
        cs.C64 = (double2*)up(nullptr, 16 * (size_t)cs.sC * nb);
        int sms = 0, smem = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, 0);
        cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, 0);
        c64_sweep(cs, jobs.data(), nb, sms, smem, 0);
        ok(cudaGetLastError());
        for (int b = 0; b < nb; ++b) ok(cudaMemcpy(g.x[b].data(), cs.C64 + (size_t)b * cs.sC, 16 * (size_t)cs.sC, cudaMemcpyDeviceToHost));
        cudaFree(cs.F); cudaFree(cs.Lb); cudaFree(cs.XY); cudaFree(cs.perm); cudaFree(cs.C64);
    }
    ok(cudaMemcpy(g.status.data(), status, sizeof(int) * nb, cudaMemcpyDeviceToHost));
    for (const void* p : {(const void*)sys.M0, (const void*)sys.M1, (const void*)sys.HV0, (const void*)sys.HV1, (const void*)sig, (const void*)rs,
                          (const void*)rd, (const void*)status, (const void*)XY, (const void*)S, (const void*)jobs_d})
        cudaFree(const_cast<void*>(p));
    return g;
}

static size_t not_finite(const Got& g) {
    size_t k = 0;
    for (const V& x : g.x)
        for (const C& v : x) k += !(std::isfinite(v.real()) && std::isfinite(v.imag()));
    return k;
}

int main(int argc, char** argv) {
    if (argc != 6) return 2;
    Made s;
    s.n = std::atoi(argv[1]); s.N = std::atoi(argv[2]); s.ms = std::atoi(argv[3]); s.md = std::atoi(argv[4]);
    const int n = s.n, nb = std::atoi(argv[5]), zc = n / 3;       // the zero column
    std::mt19937_64 rng(1234 + n);
    std::normal_distribution<double> g;
    auto fill = [&](V& v, size_t k, double f) { v.resize(k); for (C& x : v) x = f * C(g(rng), g(rng)); };
    const size_t nn = (size_t)n * n;
    // diagonal blocks 6 sqrt(n) P + noise of norm below 3.3 sqrt(n), P a permutation of each node's
    // own: condition below 3.5, and every pivot but a few is off the diagonal
    fill(s.M0, nn, 0.2); fill(s.M1, nn, 0.05); fill(s.HV0, nn * s.N, 0.5); fill(s.HV1, nn * (s.N - 1), 0.15); fill(s.sig, nn, 0.2);
    std::vector<int> p(n);
    for (int i = 0; i < s.N; ++i) {
        for (int r = 0; r < n; ++r) p[r] = r;
        std::shuffle(p.begin(), p.end(), rng);
        for (int r = 0; r < n; ++r) s.HV0[(size_t)i * nn + (size_t)r * n + p[r]] += 6 * std::sqrt((double)n) * std::polar(1.0, 0.7 * r);
    }
    fill(s.rs, (size_t)n * s.ms, 1); fill(s.rd, (size_t)n * s.md, 1);
    for (int b = 0; b < nb; ++b) s.E.push_back(0.3 + 0.1 * b);
    int smem = 0;
    ok(cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, 0));
    for (int form = 0; form < 2; ++form) {
        if (form && !c64_sweep_fits(n, smem)) continue;
        const Got a = solve(s, form);
        double diff = 0;
        for (int b = 0; b < nb; b += std::max(nb - 1, 1)) {       // the first and the last energy
            const V x = dense(s, s.E[b]);
            double big = 0, d = 0;
            for (size_t q = 0; q < x.size(); ++q) { big = std::max(big, std::abs(x[q])); d = std::max(d, std::abs(x[q] - a.x[b][q])); }
            diff = std::max(diff, d / big);
        }
        Made z = s;
        for (int r = 0; r < n; ++r) z.M0[(size_t)r * n + zc] = z.sig[(size_t)r * n + zc] = z.HV0[(size_t)r * n + zc] = 0;
        const Got zg = solve(z, form);
        Made q = s;
        q.HV0[(size_t)(n / 2) * n + n / 4] = C(std::nan(""), 0);
        const Got ng = solve(q, form);
        int reg = 0, zall = -1, nany = 0;
        for (int b = 0; b < nb; ++b) { reg |= a.status[b]; zall &= zg.status[b]; nany |= ng.status[b]; }
        std::printf("%s %.3e %d %d %zu %d %zu %zu\n", form ? "c64" : "fp64", diff, reg, zall, not_finite(zg), nany, not_finite(ng),
                    (size_t)nb * s.N * n * (s.ms + s.md));
    }
    return 0;
}
