// Complex64 block sweep of [E M - H - Sigma] c = B (Eq. qtbm_system) for a batch of
// energies, for block sizes up to 320: the factorisation stage of the mixed-precision path
// on the FP32 pipes.
//
// Per node three launches, where the tensor-core form (sweep_mixed.cu) takes 5 n / 32:
//   k_c64_node   S_i = D_i - L_i X_{i-1} and y_i = b_i - L_i y_{i-1}, tiles
//   k_lu_panel   LU of S_i, one CTA or a small cluster per energy (lu_panel.cuh)
//   k_c64_solve  [X_i | y_i] = S_i^{-1} [U_i | y_i], each CTA a block of columns
// and one launch each for all couplings L_i before the sweep and the node back substitution
// after it.  At these sizes the tensor-core GEMM is latency: its 128 x 128 tile takes 36 us
// to stage, split and drain for a product that the FP32 pipes finish in 2, and the products
// here round to nearest where the tensor cores' accumulation truncates.  D_i, U_i and L_i
// are formed in FP64 (E M - HV) and rounded once.
//
// Sums of products are made 16 terms at a time and the partial sums added: a running sum over
// all n terms left residuals of 1.3e-5 and 1.8e-5 at n = 128 and 320 (geometric mean of 8
// energies, complex64 alone), above the tensor-core form's 9.3e-6, where this leaves 6.4e-6 and
// 7.0e-6; the time is the same (n = 128, 200 nodes, 32 energies 134 -> 129 ms, n = 256 235 ->
// 226, the tile kernel held to two CTAs an SM).
#include <algorithm>

#include "lu_panel.cuh"
#include "pwqt_internal.cuh"
#include "sweep_c64.cuh"

namespace pwqt {
namespace {

__device__ __forceinline__ float2 r32(double2 v) { return make_float2((float)v.x, (float)v.y); }
__device__ __forceinline__ const double2* hv0(const C64Sweep& S, const SweepJob& J, int i) {
    return (J.HV0 ? J.HV0 : S.sys.HV0) + (size_t)i * S.sys.n * S.sys.n;
}
__device__ __forceinline__ const double2* hv1(const C64Sweep& S, const SweepJob& J, int i) {
    return (J.HV1 ? J.HV1 : S.sys.HV1) + (size_t)i * S.sys.n * S.sys.n;
}
__device__ __forceinline__ void fma2(float2& a, float2 b, float2 c) {
    a.x = fmaf(b.x, c.x, fmaf(-b.y, c.y, a.x));
    a.y = fmaf(b.x, c.y, fmaf(b.y, c.x, a.y));
}

// ---------------------------------------------------------------- couplings
// L_i = (E M1 - HV1_{i-1})^H of nodes 1 .. N-1, 32 x 32 tiles transposed through shared memory
__global__ void __launch_bounds__(256) k_c64_couplings(C64Sweep S) {
    __shared__ float2 tile[32][33];
    const SweepJob& J = S.jobs[blockIdx.z];
    const int n = S.sys.n, i = blockIdx.x + 1, nt = (n + 31) / 32;
    const int a0 = (int)blockIdx.y / nt * 32, b0 = (int)blockIdx.y % nt * 32;    // rows and columns of U_{i-1}
    const double2* H = hv1(S, J, i - 1);
    const double E = J.E;
    const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
    for (int y = ty; y < 32; y += 8)
        if (a0 + y < n && b0 + tx < n) {
            const size_t q = (size_t)(a0 + y) * n + b0 + tx;
            tile[y][tx] = r32(cconj(csub(cscale(S.sys.M1[q], E), H[q])));
        }
    __syncthreads();
    float2* L = S.Lb + blockIdx.z * S.sL + (size_t)i * n * n;
    for (int y = ty; y < 32; y += 8)
        if (b0 + y < n && a0 + tx < n) L[(size_t)(b0 + y) * n + a0 + tx] = tile[tx][y];
}

// ---------------------------------------------------------------- node block and Schur product
// T x T tiles, T = 16 R, 256 threads with R x R outputs: S into F_i (column tiles first),
// then the y columns (the source's; at the last node the drain's too)
template <int R>
__global__ void __launch_bounds__(256, 2) k_c64_node(C64Sweep S, int i) {
    constexpr int T = 16 * R;
    __shared__ float2 As[T][17], Bs[16][T + 1];
    const int e = blockIdx.z;
    const SweepJob& J = S.jobs[e];
    const int n = S.sys.n, N = S.sys.N, w = S.w, ms = J.ms;
    const int st = (n + T - 1) / T, r0 = blockIdx.y * T;
    const bool y = (int)blockIdx.x >= st;
    const int c0 = (y ? (int)blockIdx.x - st : (int)blockIdx.x) * T;
    const int cols = y ? (i == N - 1 ? ms + J.md : ms) : n;
    if (c0 >= cols) return;
    const int t = threadIdx.x, tx = t % 16, ty = t / 16;
    float2* XYi = S.XY + e * S.sXY + (size_t)i * n * w;
    float2 acc[R][R] = {};
    if (i > 0) {
        const float2* L = S.Lb + e * S.sL + (size_t)i * n * n;
        const float2* P = XYi - (size_t)n * w + (y ? n : 0);
        const int pc = y ? ms : n;
        float2 fa[R], fb[R];
        auto fetch = [&](int k0) {
#pragma unroll
            for (int q = 0; q < R; ++q) {
                const int x = t + q * 256, r = r0 + x / 16, ka = k0 + x % 16, kb = k0 + x / T, c = c0 + x % T;
                fa[q] = r < n && ka < n ? L[(size_t)r * n + ka] : make_float2(0.f, 0.f);
                fb[q] = kb < n && c < pc ? P[(size_t)kb * w + c] : make_float2(0.f, 0.f);
            }
        };
        fetch(0);
        for (int k0 = 0; k0 < n; k0 += 16) {
            __syncthreads();
#pragma unroll
            for (int q = 0; q < R; ++q) {
                const int x = t + q * 256;
                As[x / 16][x % 16] = fa[q];
                Bs[x / T][x % T] = fb[q];
            }
            __syncthreads();
            if (k0 + 16 < n) fetch(k0 + 16);
            float2 part[R][R] = {};
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                float2 b[R];
#pragma unroll
                for (int v = 0; v < R; ++v) b[v] = Bs[k][tx + 16 * v];
#pragma unroll
                for (int x = 0; x < R; ++x) {
                    const float2 a = As[ty + 16 * x][k];
#pragma unroll
                    for (int v = 0; v < R; ++v) fma2(part[x][v], a, b[v]);
                }
            }
#pragma unroll
            for (int x = 0; x < R; ++x)
#pragma unroll
                for (int v = 0; v < R; ++v) {
                    acc[x][v].x += part[x][v].x;
                    acc[x][v].y += part[x][v].y;
                }
        }
    }
    const double2* H = hv0(S, J, i);
    float2* F = S.F + e * S.sF + (size_t)i * n * n;
#pragma unroll
    for (int x = 0; x < R; ++x)
#pragma unroll
        for (int v = 0; v < R; ++v) {
            const int r = r0 + ty + 16 * x, c = c0 + tx + 16 * v;
            if (r >= n || c >= cols) continue;
            float2 o;
            if (!y) {
                const size_t q = (size_t)r * n + c;
                double2 d = csub(cscale(S.sys.M0[q], J.E), H[q]);
                if (i == 0 && J.sig_s) d = csub(d, J.sig_s[q]);
                if (i == N - 1 && J.sig_d) d = csub(d, J.sig_d[q]);
                o = r32(d);
            } else {
                o = make_float2(0.f, 0.f);
                if (i == 0 && c < ms) o = r32(J.rhs_s[(size_t)r * ms + c]);
                if (i == N - 1 && c >= ms) o = r32(J.rhs_d[(size_t)r * J.md + (c - ms)]);
            }
            o.x -= acc[x][v].x;
            o.y -= acc[x][v].y;
            if (!y) F[(size_t)r * n + c] = o;
            else XYi[(size_t)r * w + n + c] = o;
        }
}

// ---------------------------------------------------------------- solve for [X_i | y_i]
// Columns [c0, c0 + CB) of P [U_i | y] through L and U, in shared memory; the factors in
// panels of 16 columns, the next ones copied in while the current one is applied.  Diagonal
// 16 x 16 systems: half a warp per column, a lane per row.  The update gives a thread four
// rows of one column (two k of four factor rows per 16-byte load).
constexpr int SP = 16;
constexpr int SPL = SP + 2;        // rows on 16-byte boundaries
// shared memory with ns panels in flight
size_t solve_smem(int n, int cb, int ns) { return sizeof(float2) * (ns * (size_t)n * SPL + (size_t)n * cb + n); }

// rows of 16 factors (zero past column n, n even) to a panel buffer, 16 bytes at a time
__device__ __forceinline__ void copy_panel(float2* dst, const float2* src, size_t ld, int rows, int kb, int n) {
    for (int q = threadIdx.x; q < rows * (SP / 2); q += 256) {
        const int r = q / (SP / 2), k = q % (SP / 2) * 2;
        float2* d = dst + r * SPL + k;
        if (kb + k < n)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"((uint32_t)__cvta_generic_to_shared(d)), "l"(src + r * ld + kb + k) : "memory");
        else *reinterpret_cast<float4*>(d) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}
__device__ __forceinline__ void commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// all but the newest K groups have landed
template <int K> __device__ __forceinline__ void wait_groups() { asm volatile("cp.async.wait_group %0;" :: "n"(K) : "memory"); }

// rows r .. r+3 (those below `re`) of column c: X -= panel rows (P + (r - ra) SPL) x solved block xb
__device__ __forceinline__ void solve_rows(float2* X, int CB, const float2* P, const float2* xb, int r, int re) {
    float2 v[4], s[4];
    const float4* f[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        const int rr = min(x, re - 1 - r);
        v[x] = X[rr * CB];
        s[x] = make_float2(0.f, 0.f);
        f[x] = reinterpret_cast<const float4*>(P + rr * SPL);
    }
#pragma unroll
    for (int k = 0; k < SP / 2; ++k) {
        const float2 b0 = xb[2 * k * CB], b1 = xb[(2 * k + 1) * CB];
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const float4 l = f[x][k];
            fma2(s[x], make_float2(l.x, l.y), b0);
            fma2(s[x], make_float2(l.z, l.w), b1);
        }
    }
#pragma unroll
    for (int x = 0; x < 4; ++x)
        if (r + x < re) X[x * CB] = make_float2(v[x].x - s[x].x, v[x].y - s[x].y);
}

// 16 x 16 diagonal systems of up to two columns, a lane (hl) per row: D is the lane's row of
// the block (columns past wd zero), iv the reciprocal of its diagonal; unit lower or (back)
// upper.  The two chains run side by side: a step is latency (two shuffles, two FMAs).
__device__ __forceinline__ void diagonal(float2 (&x)[2], const float2* D, float2 iv, int hl, int wd, bool back) {
    float2 d[SP];
#pragma unroll
    for (int j = 0; j < SP; j += 2) {
        const float4 f = *reinterpret_cast<const float4*>(D + j);
        d[j] = make_float2(f.x, f.y);
        d[j + 1] = make_float2(f.z, f.w);
    }
    if (!back) {
#pragma unroll
        for (int j = 0; j < SP - 1; ++j)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const float2 xj = make_float2(__shfl_sync(0xffffffffu, x[c].x, j, 16), __shfl_sync(0xffffffffu, x[c].y, j, 16));
                const float2 y = lu::fnma(x[c], d[j], xj);
                x[c] = hl > j ? y : x[c];
            }
    } else {
#pragma unroll
        for (int j = SP - 1; j >= 0; --j)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const float2 z = lu::mul(x[c], iv);
                x[c] = hl == j ? z : x[c];
                const float2 xj = make_float2(__shfl_sync(0xffffffffu, x[c].x, j, 16), __shfl_sync(0xffffffffu, x[c].y, j, 16));
                const float2 y = lu::fnma(x[c], d[j], xj);
                x[c] = hl < j && j < wd ? y : x[c];
            }
    }
}

// rows [rb, re) of the columns minus panel x solved block (rows kb .. kb + wd)
__device__ __forceinline__ void panel_update(float2* X, int CB, int cb, const float2* P, int ra, int kb, int wd, int rb, int re) {
    const int t = threadIdx.x;
    if (wd == SP) {
        for (int q = t; q < (re - rb + 3) / 4 * cb; q += 256) {
            const int r = rb + q / cb * 4, c = q % cb;
            solve_rows(X + r * CB + c, CB, P + (r - ra) * SPL, X + kb * CB + c, r, re);
        }
    } else {                        // the ragged last block
        for (int q = t; q < (re - rb) * cb; q += 256) {
            const int r = rb + q / cb, c = q % cb;
            float2 v = X[r * CB + c];
            for (int k = 0; k < wd; ++k) v = lu::fnma(v, P[(r - ra) * SPL + k], X[(kb + k) * CB + c]);
            X[r * CB + c] = v;
        }
    }
}

template <int NS>
__global__ void __launch_bounds__(256) k_c64_solve(C64Sweep S, int i, int CB) {
    extern __shared__ __align__(16) float2 fsm[];
    const int e = blockIdx.y;
    const SweepJob& J = S.jobs[e];
    const int n = S.sys.n, N = S.sys.N, w = S.w, np = (n + SP - 1) / SP * SP;
    const bool last = i == N - 1;
    const int first = last ? n : 0, end = n + (last ? J.ms + J.md : J.ms);     // X_{N-1} is not used
    const int c0 = first + blockIdx.x * CB, cb = min(CB, end - c0);
    if (cb <= 0) return;
    float2* F0 = fsm;                           // NS panels of n x 16
    float2* X = fsm + NS * (size_t)n * SPL;     // n x CB (block rows past n are read from the last row)
    float2* invd = X + (size_t)n * CB;
    const int t = threadIdx.x, hl = t & 15, half = t >> 4;
    float2* XYi = S.XY + e * S.sXY + (size_t)i * n * w;
    const int* perm = S.perm + e * S.sP + (size_t)i * n;
    const float2* F = S.F + e * S.sF + (size_t)i * n * n;
    const double2* H = last ? nullptr : hv1(S, J, i);
    const int nk = np / SP;
    auto geom = [&](int s, int& kb, int& ra, int& rows) {
        const bool back = s >= nk;
        kb = (back ? 2 * nk - 1 - s : s) * SP;
        ra = back ? 0 : kb;
        rows = (back ? min(kb + SP, n) : n) - ra;
    };
    auto copy = [&](int s) {
        if (s < 2 * nk) {
            int kb, ra, rows;
            geom(s, kb, ra, rows);
            copy_panel(F0 + (size_t)(s % NS) * n * SPL, F + (size_t)ra * n, n, rows, kb, n);
        }
        commit();
    };
#pragma unroll
    for (int s = 0; s < NS - 1; ++s) copy(s);
    for (int q = t; q < n * cb; q += 256) {
        const int r = q / cb, c = c0 + q % cb, p = perm[r];
        const size_t u = (size_t)p * n + c;
        X[r * CB + q % cb] = c < n ? r32(csub(cscale(S.sys.M1[u], J.E), H[u])) : XYi[(size_t)p * w + c];
    }
    for (int r = t; r < n; r += 256) {
        const float2 d = F[(size_t)r * n + r];
        invd[r] = lu::inverse(d.x == 0.f && d.y == 0.f ? make_float2(1.f, 0.f) : d);
    }
    for (int s = 0; s < 2 * nk; ++s) {
        int kb, ra, rows;
        geom(s, kb, ra, rows);
        const bool back = s >= nk;
        const int wd = min(SP, n - kb);
        wait_groups<NS - 2>();
        __syncthreads();            // panel s landed, panel s - 1 applied
        copy(s + NS - 1);
        const float2* P = F0 + (size_t)(s % NS) * n * SPL;
        const float2* D = P + (kb - ra) * SPL;
        for (int cp = half; cp < (cb + 15) / 16 * 16; cp += 32) {
            const int c = min(cp, cb - 1), c2 = min(cp + 16, cb - 1), row = min(kb + hl, n - 1);
            float2 x[2] = {X[row * CB + c], X[row * CB + c2]};
            diagonal(x, D + min(hl, wd - 1) * SPL, invd[row], hl, wd, back);
            if (hl < wd && cp < cb) X[row * CB + c] = x[0];
            if (hl < wd && cp + 16 < cb) X[row * CB + c2] = x[1];
        }
        __syncthreads();
        panel_update(X, CB, cb, P, ra, kb, wd, back ? 0 : kb + wd, back ? kb : n);
    }
    __syncthreads();
    for (int q = t; q < n * cb; q += 256) XYi[(size_t)(q / cb) * w + c0 + q % cb] = X[(q / cb) * CB + q % cb];
}

// ---------------------------------------------------------------- node back substitution
// c_i = y_i - X_i c_{i+1}, i = N-2 .. 0, for columns [g0, g0 + CB) of one energy through all
// nodes, written as FP64 (columns past the energy's own: zero).  X_i passes through shared
// memory in panels of 16 columns, NS in flight; a thread keeps up to BI groups of four rows
// of one column in registers.
constexpr int BI = 4;
size_t back_smem(int n, int cb, int ns) { return sizeof(float2) * (ns * (size_t)n * SPL + 2 * (size_t)(n + SP) * cb); }

template <int NS>
__global__ void __launch_bounds__(256) k_c64_back(C64Sweep S, int CB) {
    extern __shared__ __align__(16) float2 fsm[];
    const int e = blockIdx.y;
    const SweepJob& J = S.jobs[e];
    const int n = S.sys.n, N = S.sys.N, w = S.w, m = S.m, mj = J.ms + J.md;
    const int g0 = blockIdx.x * CB, cb = min(CB, m - g0);
    if (cb <= 0) return;
    float2* F0 = fsm;
    float2* cur = fsm + NS * (size_t)n * SPL;          // rows n .. n + 15: zero
    float2* nxt = cur + (size_t)(n + SP) * CB;
    const int t = threadIdx.x, nk = (n + SP - 1) / SP, groups = (n + 3) / 4;
    const float2* XY = S.XY + e * S.sXY;
    double2* Cd = S.C64 + e * S.sC;
    auto copy = [&](int s) {                           // panel s counts over all nodes, N-2 first
        if (s < (N - 1) * nk) copy_panel(F0 + (size_t)(s % NS) * n * SPL, XY + (size_t)(N - 2 - s / nk) * n * w, w, n, s % nk * SP, n);
        commit();
    };
#pragma unroll
    for (int s = 0; s < NS - 1; ++s) copy(s);
    for (int q = t; q < 2 * (n + SP) * CB; q += 256) cur[q] = make_float2(0.f, 0.f);
    __syncthreads();
    for (int q = t; q < n * cb; q += 256) {
        const int r = q / cb, g = g0 + q % cb;
        const float2 v = g < mj ? XY[((size_t)(N - 1) * n + r) * w + n + g] : make_float2(0.f, 0.f);
        cur[r * CB + q % cb] = v;
        Cd[((size_t)(N - 1) * n + r) * m + g] = make_double2(v.x, v.y);
    }
    for (int i = N - 2; i >= 0; --i) {
        float2 v[BI][4];
#pragma unroll
        for (int b = 0; b < BI; ++b) {
            const int q = t + b * 256, r = q / cb * 4, g = g0 + q % cb;
#pragma unroll
            for (int x = 0; x < 4; ++x)                // drain columns of y_i are zero
                v[b][x] = r + x < n && g < J.ms ? XY[((size_t)i * n + r + x) * w + n + g] : make_float2(0.f, 0.f);
        }
        for (int k = 0; k < nk; ++k) {
            const int s = (N - 2 - i) * nk + k;
            wait_groups<NS - 2>();
            __syncthreads();
            copy(s + NS - 1);
            const float2* P = F0 + (size_t)(s % NS) * n * SPL;
#pragma unroll
            for (int b = 0; b < BI; ++b) {
                const int q = t + b * 256;
                if (q >= groups * cb) break;
                const int r = q / cb * 4;
                const float2* xb = cur + k * SP * CB + q % cb;
                const float4* f[4];
                float2 s[4] = {};
#pragma unroll
                for (int x = 0; x < 4; ++x) f[x] = reinterpret_cast<const float4*>(P + min(r + x, n - 1) * SPL);
#pragma unroll
                for (int z = 0; z < SP / 2; ++z) {
                    const float2 b0 = xb[2 * z * CB], b1 = xb[(2 * z + 1) * CB];
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        const float4 l = f[x][z];
                        fma2(s[x], make_float2(l.x, l.y), b0);
                        fma2(s[x], make_float2(l.z, l.w), b1);
                    }
                }
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    v[b][x].x -= s[x].x;
                    v[b][x].y -= s[x].y;
                }
            }
        }
#pragma unroll
        for (int b = 0; b < BI; ++b) {
            const int q = t + b * 256, r = q / cb * 4, g = g0 + q % cb;
            if (q >= groups * cb) break;
#pragma unroll
            for (int x = 0; x < 4; ++x)
                if (r + x < n) {
                    nxt[(r + x) * CB + q % cb] = v[b][x];
                    Cd[((size_t)i * n + r + x) * m + g] = make_double2(v[b][x].x, v[b][x].y);
                }
        }
        float2* o = cur;
        cur = nxt;
        nxt = o;
    }
}

// columns per CTA so that `cols` columns of nb energies fill the SMs once (or, where `most`
// forbids it, a whole number of times)
int column_block(int cols, int nb, int sms, int most, int least) {
    for (int waves = 1;; ++waves) {
        int cb = (int)(((long long)cols * nb + (long long)sms * waves - 1) / ((long long)sms * waves));
        cb = std::max(cb, least);
        while (cb <= most && (long long)((cols + cb - 1) / cb) * nb > (long long)sms * waves) ++cb;
        if (cb <= most || waves > cols * nb) return std::min(cb, most);
    }
}
// panels in flight: 4 where four CTAs of that size share an SM, else 2 (the two halves of a
// batch run side by side: at n = 128 four panels leave room for two CTAs, which cost 2 % of
// the whole call)
template <class Smem> int stages(int n, int cb, int smem_max, Smem smem) { return 4 * smem(n, cb, 4) <= (size_t)smem_max ? 4 : 2; }
template <class F> void allow_smem(F* f, int smem_max) { cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max); }
}  // namespace

bool c64_sweep_fits(int n, int smem_max) {
    return n > 24 && lup::pick_cluster(n, smem_max) > 0 && solve_smem(n, 8, 2) <= (size_t)smem_max && back_smem(n, 8, 2) <= (size_t)smem_max;
}

int c64_sweep(const C64Sweep& S, const SweepJob* host, int nb, int sms, int smem_max, cudaStream_t st) {
    const int n = S.sys.n, N = S.sys.N;
    int ms = 0, launches = 0;
    for (int b = 0; b < nb; ++b) ms = std::max(ms, host[b].ms);
    const int C = lup::pick_cluster(n, smem_max);
    allow_smem(k_c64_solve<2>, smem_max);
    allow_smem(k_c64_solve<4>, smem_max);
    allow_smem(k_c64_back<2>, smem_max);
    allow_smem(k_c64_back<4>, smem_max);
    // 64 x 64 tiles once they give every other SM a CTA (two halves of a batch share the chip)
    const int t32 = (n + 31) / 32, t64 = (n + 63) / 64;
    const bool big = (long long)t64 * t64 * nb * 2 >= sms;
    k_c64_couplings<<<dim3(N - 1, t32 * t32, nb), 256, 0, st>>>(S);
    ++launches;
    const int most_s = (int)std::min<size_t>(64, ((size_t)smem_max - solve_smem(n, 0, 2)) / (sizeof(float2) * n));
    for (int i = 0; i < N; ++i) {
        const bool last = i == N - 1;
        const int yc = last ? S.m : ms;
        if (big) k_c64_node<4><<<dim3(t64 + (yc + 63) / 64, t64, nb), 256, 0, st>>>(S, i);
        else k_c64_node<2><<<dim3(t32 + (yc + 31) / 32, t32, nb), 256, 0, st>>>(S, i);
        const lup::Batch B{S.F + (size_t)i * n * n, S.sF, S.perm + (size_t)i * n, S.sP, S.jobs};
        lup::launch(B, n, nb, C, smem_max, st);
        launches += 2;
        const int cols = (last ? 0 : n) + yc;
        if (cols > 0) {
            const int cb = column_block(cols, nb, sms, most_s, 4);
            const int ns = stages(n, cb, smem_max, solve_smem);
            const dim3 grid((cols + cb - 1) / cb, nb);
            if (ns == 4) k_c64_solve<4><<<grid, 256, solve_smem(n, cb, 4), st>>>(S, i, cb);
            else k_c64_solve<2><<<grid, 256, solve_smem(n, cb, 2), st>>>(S, i, cb);
            ++launches;
        }
    }
    const int groups = (n + 3) / 4;
    const int most_b = (int)std::min<size_t>(256 * BI / groups, ((size_t)smem_max - back_smem(n, 0, 2)) / (2 * sizeof(float2) * (n + SP)));
    const int cb = column_block(S.m, nb, sms, most_b, 4);
    const int ns = stages(n, cb, smem_max, back_smem);
    const dim3 grid((S.m + cb - 1) / cb, nb);
    if (ns == 4) k_c64_back<4><<<grid, 256, back_smem(n, cb, 4), st>>>(S, cb);
    else k_c64_back<2><<<grid, 256, back_smem(n, cb, 2), st>>>(S, cb);
    return launches + 1;
}

}  // namespace pwqt
