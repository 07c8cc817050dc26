// Complex128 block sweep of the QTBM system [E M - H - Sigma] c = B (Eq. qtbm_system,
// Sec. 3.2 of arXiv:1903.00548) for a batch of energies, and the recursive
// Green's-function form of the same elimination.
//
// Block forward elimination over the nodes i = 0..N-1 (D_i = E M0 - HV0_i,
// U_i = E M1 - HV1_i, L_{i+1} = U_i^H for real E, Sigma_s / Sigma_d on the end
// blocks):
//     S_i = D_i - L_i X_{i-1},   [X_i | y_i] = S_i^{-1} [U_i | b_i - L_i y_{i-1}]
// with partial pivoting (pivot = max |re| + |im|), then back substitution
// c_{N-1} = y_{N-1}, c_i = y_i - X_i c_{i+1}.  FP64 throughout.
//
// The FP64 pipe is the bound: 1.0 TFLOP/s measured over the chip, 1.7 FMA per clock and
// SM, so a 32 x 32 x 128 complex product occupies one SM for 150 us.  The sweep is
// therefore spread over every SM however few energies there are, in three forms:
//  * n <= SMALL_N: one CTA per energy does the whole sweep from shared memory
//    (k_sweep_small; the chain of dependent steps bounds it).
//  * larger n: per node the Schur product as tiles over (rows, columns, energies)
//    (k_node), the LU of S_i by a thread-block cluster per energy (k_lu), and the solve
//    for [X_i | y_i] over column blocks (k_solve); the node back substitution is one
//    launch, each CTA carrying its columns through all nodes (k_back).
//  * n whose rows no cluster holds in shared memory (above ~450): one CTA per energy
//    (k_sweep_fp64), streaming its blocks through L2.
// The source-injected columns of b live at node 0 and the drain-injected ones at node
// N-1, so the drain columns of y_i are zero before the last node and are not computed.
#include <algorithm>

#include "lu_cluster.cuh"
#include "pwqt_internal.cuh"
#include "sweep_common.cuh"
#include "sweep_mixed.cuh"

namespace pwqt {

constexpr int TS = 32, TK = 16, NT = 256;

// C[r][c] -= sum_k A(r,k) * B[k][c], r < M, c < Nc, k < K.  A is read through a functor,
// B and C are row-major with strides ldb / ldc.  256 threads, 32x32 output tiles, 2x2 per thread.
template <class AF, class CF>
__device__ void cta_gemm_sub(double2* smem, int M, int Nc, int K, AF A, const double2* __restrict__ B, int ldb, CF Cptr) {
    double2 (*As)[TK + 1] = reinterpret_cast<double2 (*)[TK + 1]>(smem);
    double2 (*Bs)[TS + 1] = reinterpret_cast<double2 (*)[TS + 1]>(smem + TS * (TK + 1));
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;   // 16 x 16 threads, each 2x2 outputs
    for (int r0 = 0; r0 < M; r0 += TS)
        for (int c0 = 0; c0 < Nc; c0 += TS) {
            double2 acc[2][2] = {{{0, 0}, {0, 0}}, {{0, 0}, {0, 0}}};
            for (int k0 = 0; k0 < K; k0 += TK) {
                for (int t = threadIdx.x; t < TS * TK; t += NT) {
                    int rr = t / TK, kk = t % TK;
                    As[rr][kk] = (r0 + rr < M && k0 + kk < K) ? A(r0 + rr, k0 + kk) : make_double2(0, 0);
                    int kb = t / TS, cb = t % TS;
                    Bs[kb][cb] = (k0 + kb < K && c0 + cb < Nc) ? B[(size_t)(k0 + kb) * ldb + c0 + cb] : make_double2(0, 0);
                }
                __syncthreads();
#pragma unroll 4
                for (int kk = 0; kk < TK; ++kk) {
                    double2 a0 = As[ty * 2][kk], a1 = As[ty * 2 + 1][kk];
                    double2 b0 = Bs[kk][tx * 2], b1 = Bs[kk][tx * 2 + 1];
                    cfma(acc[0][0], a0, b0); cfma(acc[0][1], a0, b1);
                    cfma(acc[1][0], a1, b0); cfma(acc[1][1], a1, b1);
                }
                __syncthreads();
            }
            for (int i = 0; i < 2; ++i)
                for (int j = 0; j < 2; ++j) {
                    int r = r0 + ty * 2 + i, cc = c0 + tx * 2 + j;
                    if (r < M && cc < Nc) {
                        double2* p = Cptr(r, cc);
                        *p = csub(*p, acc[i][j]);
                    }
                }
        }
}

// block-wide argmax of |re|+|im| over rows j..n-1 of column j of S (row stride lds)
__device__ int cta_pivot(const double2* S, int lds, int n, int j) {
    __shared__ double bv[NT / 32];
    __shared__ int bi[NT / 32];
    double best = -1.0;
    int idx = j;
    for (int r = j + threadIdx.x; r < n; r += NT) {
        double v = cabs1(S[(size_t)r * lds + j]);
        if (v > best) { best = v; idx = r; }
    }
    for (int o = 16; o > 0; o >>= 1) {
        double ov = __shfl_down_sync(0xffffffff, best, o);
        int oi = __shfl_down_sync(0xffffffff, idx, o);
        if (ov > best || (ov == best && oi < idx)) { best = ov; idx = oi; }
    }
    if ((threadIdx.x & 31) == 0) { bv[threadIdx.x >> 5] = best; bi[threadIdx.x >> 5] = idx; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < NT / 32; ++w)
            if (bv[w] > bv[0] || (bv[w] == bv[0] && bi[w] < bi[0])) { bv[0] = bv[w]; bi[0] = bi[w]; }
    }
    __syncthreads();
    int p = bi[0];
    __syncthreads();
    return p;
}

// -(2/pi) Im Tr of the n x n block at G (row stride ldg), block-wide; thread 0 gets it
__device__ double cta_dos(const double2* G, int ldg, int n) {
    __shared__ double part[NT / 32];
    double acc = 0.0;
    for (int r = threadIdx.x; r < n; r += NT) acc += G[(size_t)r * ldg + r].y;
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffff, acc, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < NT / 32; ++w) t += part[w];
    __syncthreads();
    return -(2.0 / 3.141592653589793) * t;
}

// Backward pass of the Green's-function recursion over the forward panels
// R_i = [X_i | g_i] (row stride 2n).  Per node, with the n x n scratch S:
//   S = -X_i G_{i+1};  X-part of R_i = -L_{i+1} g_i;  g-part of R_i -= (-S)(X-part)
// so that the g-part becomes g_i + (X_i G_{i+1})(L_{i+1} g_i) = G_i.
__device__ void green_backward(const SweepSys& sys, const SweepJob& J, double2* smem, int st) {
    const int n = sys.n, N = sys.N, w = 2 * n;
    const double E = J.E;
    double2* S = J.S;
    double d = cta_dos(J.XY + (size_t)(N - 1) * n * w + n, w, n);
    if (threadIdx.x == 0) J.dos[N - 1] = d;
    for (int i = N - 2; i >= 0; --i) {
        double2* R = J.XY + (size_t)i * n * w;
        const double2* Gn = J.XY + (size_t)(i + 1) * n * w + n;
        for (int t = threadIdx.x; t < n * n; t += NT) S[t] = make_double2(0, 0);
        __syncthreads();
        {
            auto A = [&](int r, int k) { return R[(size_t)r * w + k]; };
            auto C = [&](int r, int cc) -> double2* { return S + (size_t)r * n + cc; };
            cta_gemm_sub(smem, n, n, n, A, Gn, w, C);                 // S = -X_i G_{i+1}
        }
        __syncthreads();
        for (int t = threadIdx.x; t < n * n; t += NT) R[(size_t)(t / n) * w + t % n] = make_double2(0, 0);
        __syncthreads();
        {
            const double2* HV1 = (J.HV1 ? J.HV1 : sys.HV1) + (size_t)i * n * n;
            const double2* M1 = sys.M1;
            auto A = [&](int r, int k) {                               // L_{i+1}[r][k] = conj(U_i[k][r])
                size_t t = (size_t)k * n + r;
                return cconj(csub(cscale(M1[t], E), HV1[t]));
            };
            auto C = [&](int r, int cc) -> double2* { return R + (size_t)r * w + cc; };
            cta_gemm_sub(smem, n, n, n, A, R + n, w, C);             // X-part = -L_{i+1} g_i
        }
        __syncthreads();
        {
            auto A = [&](int r, int k) { const double2 v = S[(size_t)r * n + k]; return make_double2(-v.x, -v.y); };
            auto C = [&](int r, int cc) -> double2* { return R + (size_t)r * w + n + cc; };
            cta_gemm_sub(smem, n, n, n, A, R, w, C);                 // g-part -= (X_i G_{i+1})(-L_{i+1} g_i)
        }
        __syncthreads();
        d = cta_dos(R + n, w, n);
        if (threadIdx.x == 0) J.dos[i] = d;
    }
    if (threadIdx.x == 0) atomicOr(J.status, st);
}

// GREEN = false: the QTBM solve of the file header.  GREEN = true: the recursive Green's-function
// form of the same elimination (the NEGF side of Sec. 3.2).  The forward pass is the
// sweep with [U_i | I] as every node's right-hand side and no coupling between the
// right-hand sides of neighbouring nodes, so that R_i = [X_i | g_i] with the
// left-connected g_i = S_i^{-1}; the backward pass then forms the diagonal blocks
//     G_{N-1} = g_{N-1},   G_i = g_i + (X_i G_{i+1}) (L_{i+1} g_i)
// in place of g_i, with L_{i+1} = U_i^H, and records -(2/pi) Im Tr G_i.
template <bool GREEN>
__global__ void __launch_bounds__(NT) k_sweep_fp64(SweepSys sys, const SweepJob* __restrict__ jobs) {
    const SweepJob J = jobs[blockIdx.x];
    const int n = sys.n, N = sys.N, m = J.ms + J.md, w = n + m;
    const double E = J.E;
    double2* S = J.S;
    // shared: GEMM tiles, reused as the multiplier column of the elimination (n <= 1024)
    __shared__ double2 smem[TS * (TK + 1) + TK * (TS + 1) > 1024 ? TS * (TK + 1) + TK * (TS + 1) : 1024];
    double2* lcol = smem;
    int st = 0;
    for (int i = 0; i < N; ++i) {
        double2* R = J.XY + (size_t)i * n * w;
        const double2* HV0 = (J.HV0 ? J.HV0 : sys.HV0) + (size_t)i * n * n;
        const double2* HV1 = (J.HV1 ? J.HV1 : sys.HV1) + (size_t)i * n * n;
        for (int t = threadIdx.x; t < n * n; t += NT) {
            double2 v = csub(cscale(sys.M0[t], E), HV0[t]);
            if (i == 0 && J.sig_s) v = csub(v, J.sig_s[t]);
            if (i == N - 1 && J.sig_d) v = csub(v, J.sig_d[t]);
            S[t] = v;
        }
        for (int t = threadIdx.x; t < n * w; t += NT) {
            int r = t / w, cc = t % w;
            double2 v = make_double2(0, 0);
            if (cc < n) {
                if (i < N - 1) v = csub(cscale(sys.M1[(size_t)r * n + cc], E), HV1[(size_t)r * n + cc]);
            } else if (GREEN) {
                if (cc - n == r) v = make_double2(1.0, 0.0);
            } else {
                int col = cc - n;
                if (i == 0 && col < J.ms) v = J.rhs_s[(size_t)r * J.ms + col];
                if (i == N - 1 && col >= J.ms) v = J.rhs_d[(size_t)r * J.md + (col - J.ms)];
            }
            R[t] = v;
        }
        __syncthreads();
        if (i > 0) {
            const double2* P = J.XY + (size_t)(i - 1) * n * w;   // [X_{i-1} | y_{i-1}]
            const double2* HVp = (J.HV1 ? J.HV1 : sys.HV1) + (size_t)(i - 1) * n * n;
            const double2* M1 = sys.M1;
            // L_i[r][k] = conj(U_{i-1}[k][r]), U_{i-1} = E M1 - HV1_{i-1}
            auto A = [&](int r, int k) {
                size_t t = (size_t)k * n + r;
                return cconj(csub(cscale(M1[t], E), HVp[t]));
            };
            auto C = [&](int r, int cc) -> double2* { return cc < n ? S + (size_t)r * n + cc : R + (size_t)r * w + cc; };
            // [S | *, y] -= L_i [X_{i-1} | y_{i-1}]  (cols n..w-1 of R); S alone for GREEN
            cta_gemm_sub(smem, n, GREEN ? n : w, n, A, P, w, C);
            __syncthreads();
        }
        // Gaussian elimination with partial pivoting on S, applied to the rows of R
        for (int j = 0; j < n; ++j) {
            int p = cta_pivot(S, n, n, j);
            if (p != j) {
                for (int cc = threadIdx.x; cc < n; cc += NT) {
                    double2 a = S[(size_t)j * n + cc]; S[(size_t)j * n + cc] = S[(size_t)p * n + cc]; S[(size_t)p * n + cc] = a;
                }
                for (int cc = threadIdx.x; cc < w; cc += NT) {
                    double2 a = R[(size_t)j * w + cc]; R[(size_t)j * w + cc] = R[(size_t)p * w + cc]; R[(size_t)p * w + cc] = a;
                }
            }
            __syncthreads();
            double2 piv = S[(size_t)j * n + j];
            if (piv.x == 0.0 && piv.y == 0.0) { st |= PWQT_ST_SINGULAR_PIVOT; piv = make_double2(1.0, 0.0); }
            for (int r = j + 1 + threadIdx.x; r < n; r += NT) lcol[r] = cdiv(S[(size_t)r * n + j], piv);
            __syncthreads();
            const int rows = n - j - 1, cs = n - j - 1, cols = cs + w;
            for (long t = threadIdx.x; t < (long)rows * cols; t += NT) {
                int r = j + 1 + (int)(t / cols), cc = (int)(t % cols);
                double2 l = lcol[r];
                if (cc < cs) {
                    int col = j + 1 + cc;
                    cfma(S[(size_t)r * n + col], make_double2(-l.x, -l.y), S[(size_t)j * n + col]);
                } else {
                    int col = cc - cs;
                    cfma(R[(size_t)r * w + col], make_double2(-l.x, -l.y), R[(size_t)j * w + col]);
                }
            }
            __syncthreads();
        }
        // back substitution with the upper triangle
        for (int j = n - 1; j >= 0; --j) {
            double2 d = S[(size_t)j * n + j];
            if (d.x == 0.0 && d.y == 0.0) d = make_double2(1.0, 0.0);
            for (int cc = threadIdx.x; cc < w; cc += NT) R[(size_t)j * w + cc] = cdiv(R[(size_t)j * w + cc], d);
            __syncthreads();
            for (long t = threadIdx.x; t < (long)j * w; t += NT) {
                int r = (int)(t / w), cc = (int)(t % w);
                double2 s = S[(size_t)r * n + j];
                cfma(R[(size_t)r * w + cc], make_double2(-s.x, -s.y), R[(size_t)j * w + cc]);
            }
            __syncthreads();
        }
    }
    if constexpr (GREEN) {
        green_backward(sys, J, smem, st);
    } else {
        // back substitution over nodes: c_i = y_i - X_i c_{i+1} (c overwrites y)
        for (int i = N - 2; i >= 0; --i) {
            double2* R = J.XY + (size_t)i * n * w;
            const double2* Cn = J.XY + (size_t)(i + 1) * n * w + n;
            auto A = [&](int r, int k) { return R[(size_t)r * w + k]; };
            auto C = [&](int r, int cc) -> double2* { return R + (size_t)r * w + n + cc; };
            cta_gemm_sub(smem, n, m, n, A, Cn, w, C);
            __syncthreads();
        }
        if (threadIdx.x == 0) atomicOr(J.status, st);
    }
}

// ---------------------------------------------------------------- tile product
// acc = sum_k A(r0 + ., k) B(k, c0 + .) over a T x T tile, T = 16 R: 256 threads, R x R
// outputs each.  A and B are read through functors that return zero outside the operands;
// the next 16 k are fetched while the current ones are multiplied.  A warp holds 2 R rows and
// skips those past M and the column halves past Nc: an FP64 instruction costs a warp 64
// cycles however few of its lanes count.
template <int R> struct TileMem { double2 a[16 * R][17], b[16][16 * R + 1]; };

template <int R, class AF, class BF>
__device__ __forceinline__ void tile_product(TileMem<R>& sm, int r0, int c0, int M, int Nc, int K, AF A, BF B, double2 (&out)[R][R]) {
    constexpr int T = 16 * R;
    const int t = threadIdx.x, tx = t % 16, ty = t / 16;
#pragma unroll
    for (int x = 0; x < R; ++x)
#pragma unroll
        for (int y = 0; y < R; ++y) out[x][y] = make_double2(0, 0);
    double2 fa[R], fb[R];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const int e = t + q * 256;
            fa[q] = k0 + e % 16 < K ? A(r0 + e / 16, k0 + e % 16) : make_double2(0, 0);
            fb[q] = k0 + e / T < K ? B(k0 + e / T, c0 + e % T) : make_double2(0, 0);
        }
    };
    fetch(0);
    for (int k0 = 0; k0 < K; k0 += 16) {
        __syncthreads();
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const int e = t + q * 256;
            sm.a[e / 16][e % 16] = fa[q];
            sm.b[e / T][e % T] = fb[q];
        }
        __syncthreads();
        if (k0 + 16 < K) fetch(k0 + 16);
        const int ke = min(16, K - k0);
#pragma unroll 4
        for (int k = 0; k < ke; ++k)
#pragma unroll
            for (int x = 0; x < R; ++x) {
                if (r0 + 16 * x + (ty & ~1) >= M) continue;
                const double2 a = sm.a[ty + 16 * x][k];
#pragma unroll
                for (int y = 0; y < R; ++y) {
                    if (c0 + 16 * y >= Nc) continue;
                    cfma(out[x][y], a, sm.b[k][tx + 16 * y]);
                }
            }
    }
}

__device__ __forceinline__ const double2* hv0_of(const SweepSys& s, const SweepJob& J, int i) {
    return (J.HV0 ? J.HV0 : s.HV0) + (size_t)i * s.n * s.n;
}
__device__ __forceinline__ const double2* hv1_of(const SweepSys& s, const SweepJob& J, int i) {
    return (J.HV1 ? J.HV1 : s.HV1) + (size_t)i * s.n * s.n;
}
// the row permutation of the node in work sits in the X part of the last node's panel,
// which the recursion does not use (n ints in its first row)
__device__ __forceinline__ int* perm_of(const SweepSys& s, const SweepJob& J) {
    return reinterpret_cast<int*>(J.XY + (size_t)(s.N - 1) * s.n * (s.n + J.ms + J.md));
}
// columns of y that are not zero at node i (GREEN: the identity at every node)
__device__ __forceinline__ int y_cols(const SweepJob& J, bool last, bool green) { return green || !last ? J.ms : J.ms + J.md; }

// ---------------------------------------------------------------- node block and Schur product
// S = D_i - L_i X_{i-1} and the y columns of R_i = b_i - L_i y_{i-1}; column tiles of S
// first, then those of y (not for GREEN, whose right-hand sides do not couple).
template <int R, bool GREEN>
__global__ void __launch_bounds__(256) k_node(SweepSys sys, const SweepJob* __restrict__ jobs, int i) {
    constexpr int T = 16 * R;
    __shared__ TileMem<R> sm;
    const SweepJob& J = jobs[blockIdx.z];
    const int n = sys.n, N = sys.N, w = n + J.ms + J.md, ms = J.ms;
    const int st = (n + T - 1) / T, r0 = blockIdx.y * T;
    const bool y = (int)blockIdx.x >= st;
    const int c0 = (y ? (int)blockIdx.x - st : (int)blockIdx.x) * T;
    const int cols = y ? y_cols(J, i == N - 1, false) : n;
    if (c0 >= cols) return;
    const double E = J.E;
    const double2* M0 = sys.M0;
    double2 acc[R][R] = {};
    if (i > 0) {
        const double2* P = J.XY + (size_t)(i - 1) * n * w + (y ? n : 0);
        const double2* HVm = hv1_of(sys, J, i - 1);
        const double2* M1 = sys.M1;
        const int pc = y ? ms : n;      // y_{i-1}: the source columns
        auto A = [&](int r, int k) {
            if (r >= n) return make_double2(0, 0);
            const size_t q = (size_t)k * n + r;      // L_i[r][k] = conj(U_{i-1}[k][r])
            return cconj(csub(cscale(M1[q], E), HVm[q]));
        };
        auto B = [&](int k, int c) { return c < pc ? P[(size_t)k * w + c] : make_double2(0, 0); };
        tile_product<R>(sm, r0, c0, n, cols, n, A, B, acc);
    }
    const double2* HV0 = hv0_of(sys, J, i);
#pragma unroll
    for (int x = 0; x < R; ++x)
#pragma unroll
        for (int v = 0; v < R; ++v) {
            const int r = r0 + (int)threadIdx.x / 16 + 16 * x, c = c0 + (int)threadIdx.x % 16 + 16 * v;
            if (r >= n || c >= cols) continue;
            if (!y) {
                const size_t q = (size_t)r * n + c;
                double2 d = csub(cscale(M0[q], E), HV0[q]);
                if (i == 0 && J.sig_s) d = csub(d, J.sig_s[q]);
                if (i == N - 1 && J.sig_d) d = csub(d, J.sig_d[q]);
                J.S[q] = csub(d, acc[x][v]);
            } else {
                double2 b = make_double2(0, 0);
                if (i == 0 && c < ms) b = J.rhs_s[(size_t)r * ms + c];
                if (i == N - 1 && c >= ms) b = J.rhs_d[(size_t)r * J.md + (c - ms)];
                J.XY[((size_t)i * n + r) * w + n + c] = csub(b, acc[x][v]);
            }
        }
}

struct Where64 {
    const SweepJob* jobs;
    SweepSys sys;
    __device__ lu::Place operator()(int e) const {
        const SweepJob& J = jobs[e];
        return {J.S, J.S, sys.n, perm_of(sys, J), J.status};
    }
};

// ---------------------------------------------------------------- solve for [X_i | y_i]
// Columns [c0, c0 + CB) of P [U_i | y] through L and U (unit lower; the factors in S): the
// columns stay in shared memory, the factors pass through it in panels of 8 columns, the
// next one copied in (cp.async) while the current one is applied.  The 8 x 8 diagonal
// systems take half a warp per column, real and imaginary part of a row in neighbouring
// lanes: a step of their chain is two FP64 instructions, and of the lanes' work only half is
// idle (blocks of 16 spent a quarter of the kernel there).  Bound by the FP64 pipe, n^2 CB
// complex multiply-adds a CTA, and by the 2 n dependent steps when CB is small.
constexpr int SP = 8;              // panel columns
constexpr int SPL = SP + 1;
size_t solve_smem(int n, int cb) { return sizeof(double2) * ((size_t)n * cb + 2 * (size_t)n * SPL + n); }

template <bool GREEN>
__global__ void __launch_bounds__(256) k_solve(SweepSys sys, const SweepJob* __restrict__ jobs, int i, int CB) {
    extern __shared__ __align__(16) double2 sv[];
    const SweepJob& J = jobs[blockIdx.y];
    const int n = sys.n, N = sys.N, w = n + J.ms + J.md;
    const bool last = i == N - 1;
    const int first = last ? n : 0, end = n + y_cols(J, last, GREEN);   // X_{N-1} is not used
    const int c0 = first + blockIdx.x * CB, cb = min(CB, end - c0);
    if (cb <= 0) return;
    double2* X = sv;                        // n x CB
    double2* F = sv + (size_t)n * CB;       // two panels: rows x 8
    double2* invd = F + 2 * (size_t)n * SPL;
    const int t = threadIdx.x, hl = (t & 15) >> 1, part = t & 1, half = t >> 4;
    double2* R = J.XY + (size_t)i * n * w;
    const int* perm = perm_of(sys, J);
    const double2* HV1 = last ? nullptr : hv1_of(sys, J, i);
    const double2* S = J.S;
    const int nk = (n + SP - 1) / SP;
    // panel step s = 0 .. 2 nk - 1: forward panels from the left, then backward from the right
    auto geom = [&](int s, int& kb, int& ra, int& rows) {
        const bool back = s >= nk;
        kb = (back ? 2 * nk - 1 - s : s) * SP;
        ra = back ? 0 : kb;
        rows = (back ? min(kb + SP, n) : n) - ra;
    };
    auto copy = [&](int s) {
        int kb, ra, rows;
        geom(s, kb, ra, rows);
        double2* dst = F + (size_t)(s & 1) * n * SPL;
        for (int q = t; q < rows * SP; q += 256) {
            const int r = q / SP, k = q % SP;
            if (kb + k < n)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" :: "r"((uint32_t)__cvta_generic_to_shared(dst + r * SPL + k)),
                             "l"(S + (size_t)(ra + r) * n + kb + k) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    copy(0);
    for (int q = t; q < n * cb; q += 256) {
        const int r = q / cb, c = c0 + q % cb, p = perm[r];
        double2 v;
        if (c < n) {
            const size_t u = (size_t)p * n + c;
            v = csub(cscale(sys.M1[u], J.E), HV1[u]);
        } else if (GREEN) {
            v = make_double2(c - n == p ? 1.0 : 0.0, 0.0);
        } else {
            v = R[(size_t)p * w + c];
        }
        X[r * CB + q % cb] = v;
    }
    for (int r = t; r < n; r += 256) {
        const double2 d = S[(size_t)r * n + r];
        invd[r] = d.x == 0.0 && d.y == 0.0 ? make_double2(1, 0) : lu::inverse(d);
    }
    for (int s = 0; s < 2 * nk; ++s) {
        int kb, ra, rows;
        geom(s, kb, ra, rows);
        const bool back = s >= nk;
        const int wd = min(SP, n - kb);
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();            // panel s landed, panel s - 1 applied
        if (s + 1 < 2 * nk) copy(s + 1);
        double2* P = F + (size_t)(s & 1) * n * SPL;
        double2* D = P + (kb - ra) * SPL;             // diagonal block
        if (back) {                 // its rows over their diagonal: a unit upper triangle
            if (t < SP * SP && t / SP < wd && t % SP < wd) D[t / SP * SPL + t % SP] = cmul(D[t / SP * SPL + t % SP], invd[kb + t / SP]);
            __syncthreads();
        }
        for (int cp = half; cp < (cb + 15) / 16 * 16; cp += 16) {
            const int c = min(cp, cb - 1), row = min(kb + hl, n - 1);
            const bool in = hl < wd && cp < cb;
            double* xp = reinterpret_cast<double*>(X + row * CB + c) + part;
            double x = *xp;
            if (back) {
                const double o = __shfl_xor_sync(0xffffffffu, x, 1);
                const double2 v = invd[row];
                x = part ? fma(x, v.x, o * v.y) : fma(x, v.x, -(o * v.y));
            }
            for (int q = 0; q < wd - 1; ++q) {
                const int j = back ? wd - 1 - q : q;
                const double xr = __shfl_sync(0xffffffffu, x, 2 * j, 16), xi = __shfl_sync(0xffffffffu, x, 2 * j + 1, 16);
                if (in && (back ? hl < j : hl > j)) {
                    const double2 d = D[hl * SPL + j];
                    x = part ? fma(-d.x, xi, fma(-d.y, xr, x)) : fma(-d.x, xr, fma(d.y, xi, x));
                }
            }
            if (in) *xp = x;
        }
        __syncthreads();
        // the rows still to come minus panel x solved block
        const int rb = back ? 0 : kb + wd, re = back ? kb : n;
        for (int q = t; q < (re - rb) * cb; q += 256) {
            const int r = rb + q / cb, c = q % cb;
            const double2* f = P + (r - ra) * SPL;
            const double2* x = X + kb * CB + c;
            double2 v = X[r * CB + c];
#pragma unroll
            for (int k = 0; k < SP; ++k)
                if (k < wd) v = lu::fnma(v, f[k], x[k * CB]);
            X[r * CB + c] = v;
        }
    }
    __syncthreads();
    for (int q = t; q < n * cb; q += 256) R[(size_t)(q / cb) * w + c0 + q % cb] = X[(q / cb) * CB + q % cb];
}

// ---------------------------------------------------------------- node back substitution
// c_i = y_i - X_i c_{i+1} for columns [g0, g0 + CB) of one energy, i = N-2 .. 0 (c
// overwrites y): the columns are independent, so a CTA carries its own through all nodes.
// KS (a power of two) threads split an entry's sum where the entries alone leave threads idle.
size_t back_smem(int n, int cb) { return sizeof(double2) * 2 * (size_t)n * cb; }

__global__ void __launch_bounds__(256) k_back(SweepSys sys, const SweepJob* __restrict__ jobs, int CB, int KS) {
    extern __shared__ __align__(16) double2 sv[];
    const SweepJob& J = jobs[blockIdx.y];
    const int n = sys.n, N = sys.N, m = J.ms + J.md, w = n + m;
    const int g0 = blockIdx.x * CB, cb = min(CB, m - g0);
    if (cb <= 0) return;
    double2 *cur = sv, *nxt = sv + (size_t)n * CB;
    const int t = threadIdx.x;
    const double2* last = J.XY + (size_t)(N - 1) * n * w + n + g0;
    for (int q = t; q < n * cb; q += 256) cur[q] = last[(size_t)(q / cb) * w + q % cb];
    for (int i = N - 2; i >= 0; --i) {
        double2* R = J.XY + (size_t)i * n * w;
        __syncthreads();
        // KS neighbouring threads share an entry, each with every KS-th k
        for (int q0 = 0; q0 < n * cb * KS; q0 += 256) {
            const int q = min(q0 + t, n * cb * KS - 1) / KS, r = q / cb, g = q % cb;
            const double2* x = R + (size_t)r * w;
            double2 s = make_double2(0, 0);
#pragma unroll 4
            for (int k = t % KS; k < n; k += KS) cfma(s, x[k], cur[k * cb + g]);
            for (int o = KS >> 1; o > 0; o >>= 1) {
                s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
                s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
            }
            if (t % KS == 0 && q0 + t < n * cb * KS) {
                double2& y = R[(size_t)r * w + n + g0 + g];
                const double2 y0 = g0 + g < J.ms ? y : make_double2(0, 0);      // drain columns of y_i are zero
                const double2 v = csub(y0, s);
                y = v;
                nxt[q] = v;
            }
        }
        double2* s = cur;
        cur = nxt;
        nxt = s;
    }
}

// ---------------------------------------------------------------- Green's-function products
// stage 0: S = X_i G_{i+1};  stage 1: X part of R_i = L_{i+1} g_i;  stage 2: g part of
// R_i += S (X part), i.e. G_i = g_i + (X_i G_{i+1})(L_{i+1} g_i).
template <int R>
__global__ void __launch_bounds__(256) k_green_product(SweepSys sys, const SweepJob* __restrict__ jobs, int i, int stage) {
    constexpr int T = 16 * R;
    __shared__ TileMem<R> sm;
    const SweepJob& J = jobs[blockIdx.z];
    const int n = sys.n, w = 2 * n, r0 = blockIdx.y * T, c0 = blockIdx.x * T;
    double2* P = J.XY + (size_t)i * n * w;
    const double2* Gn = J.XY + (size_t)(i + 1) * n * w + n;
    const double2 zero = make_double2(0, 0);
    double2 acc[R][R];
    if (stage == 0) {
        tile_product<R>(sm, r0, c0, n, n, n, [&](int r, int k) { return r < n ? P[(size_t)r * w + k] : zero; },
                        [&](int k, int c) { return c < n ? Gn[(size_t)k * w + c] : zero; }, acc);
    } else if (stage == 1) {
        const double2* HV1 = hv1_of(sys, J, i);
        const double2* M1 = sys.M1;
        const double E = J.E;
        tile_product<R>(sm, r0, c0, n, n, n,
                        [&](int r, int k) {
                            if (r >= n) return zero;
                            const size_t q = (size_t)k * n + r;
                            return cconj(csub(cscale(M1[q], E), HV1[q]));
                        },
                        [&](int k, int c) { return c < n ? P[(size_t)k * w + n + c] : zero; }, acc);
    } else {
        tile_product<R>(sm, r0, c0, n, n, n, [&](int r, int k) { return r < n ? J.S[(size_t)r * n + k] : zero; },
                        [&](int k, int c) { return c < n ? P[(size_t)k * w + c] : zero; }, acc);
    }
#pragma unroll
    for (int x = 0; x < R; ++x)
#pragma unroll
        for (int v = 0; v < R; ++v) {
            const int r = r0 + (int)threadIdx.x / 16 + 16 * x, c = c0 + (int)threadIdx.x % 16 + 16 * v;
            if (r >= n || c >= n) continue;
            if (stage == 0) J.S[(size_t)r * n + c] = acc[x][v];
            else if (stage == 1) P[(size_t)r * w + c] = acc[x][v];
            else P[(size_t)r * w + n + c] = cadd(P[(size_t)r * w + n + c], acc[x][v]);
        }
}

// -(2/pi) Im Tr G_ii of every node
__global__ void __launch_bounds__(256) k_green_dos(int n, const SweepJob* __restrict__ jobs) {
    const SweepJob& J = jobs[blockIdx.y];
    const double d = cta_dos(J.XY + (size_t)blockIdx.x * n * 2 * n + n, 2 * n, n);
    if (threadIdx.x == 0) J.dos[blockIdx.x] = d;
}

// ---------------------------------------------------------------- FP64 residual
// r_i = b_i - (L_i c_{i-1} + D_i c_i + U_i c_{i+1}) (FP64), per column sums of |r|^2 and
// |b|^2.  Tiles of (rows, columns) per node and energy; the block elements are formed while
// they are staged, once per tile row and 16 R columns.
template <int R>
__global__ void __launch_bounds__(256) k_residual_fp64(SweepSys sys, const ResJob* __restrict__ jobs) {
    constexpr int T = 16 * R;
    __shared__ TileMem<R> sm;
    __shared__ double sr[T], sb[T];
    const ResJob& J = jobs[blockIdx.z];
    const int n = sys.n, N = sys.N, m = J.ms + J.md, i = blockIdx.x;
    const int rt = (n + T - 1) / T, r0 = ((int)blockIdx.y % rt) * T, c0 = ((int)blockIdx.y / rt) * T;
    if (c0 >= m) return;
    const double E = J.E;
    const size_t nn = (size_t)n * n;
    const double2* HV0 = (J.HV0 ? J.HV0 : sys.HV0) + i * nn;
    const double2* HV1 = (J.HV1 ? J.HV1 : sys.HV1) + i * nn;
    const double2 *M0 = sys.M0, *M1 = sys.M1;
    const double2 zero = make_double2(0, 0);
    double2 sum[R][R] = {}, acc[R][R];
    auto add = [&] {
#pragma unroll
        for (int x = 0; x < R; ++x)
#pragma unroll
            for (int v = 0; v < R; ++v) sum[x][v] = cadd(sum[x][v], acc[x][v]);
    };
    auto rhs = [&](const double2* c) { return [=](int k, int g) { return g < m ? c[(size_t)k * J.row_stride + g] : zero; }; };
    const double2* ci = J.C + (size_t)i * J.node_stride;
    tile_product<R>(sm, r0, c0, n, m, n, [&](int r, int k) {
        if (r >= n) return zero;
        const size_t q = (size_t)r * n + k;
        double2 d = csub(cscale(M0[q], E), HV0[q]);
        if (i == 0) d = csub(d, J.sig_s[q]);
        if (i == N - 1) d = csub(d, J.sig_d[q]);
        return d;
    }, rhs(ci), acc);
    add();
    if (i + 1 < N) {
        tile_product<R>(sm, r0, c0, n, m, n, [&](int r, int k) {
            if (r >= n) return zero;
            const size_t q = (size_t)r * n + k;
            return csub(cscale(M1[q], E), HV1[q]);
        }, rhs(ci + J.node_stride), acc);
        add();
    }
    if (i > 0) {
        const double2* HVm = HV1 - nn;
        tile_product<R>(sm, r0, c0, n, m, n, [&](int r, int k) {
            if (r >= n) return zero;
            const size_t q = (size_t)k * n + r;
            return cconj(csub(cscale(M1[q], E), HVm[q]));
        }, rhs(ci - J.node_stride), acc);
        add();
    }
    const bool ends = i == 0 || i == N - 1;
    if (threadIdx.x < T) sr[threadIdx.x] = sb[threadIdx.x] = 0.0;
    __syncthreads();
#pragma unroll
    for (int v = 0; v < R; ++v) {
        const int cl = (int)threadIdx.x % 16 + 16 * v, g = c0 + cl;
        double nr = 0, nb = 0;
#pragma unroll
        for (int x = 0; x < R; ++x) {
            const int r = r0 + (int)threadIdx.x / 16 + 16 * x;
            if (r >= n || g >= m) continue;
            double2 b = zero;
            if (i == 0 && g < J.ms) b = J.rhs_s[(size_t)r * J.ms + g];
            if (i == N - 1 && g >= J.ms) b = J.rhs_d[(size_t)r * J.md + (g - J.ms)];
            const double2 res = csub(b, sum[x][v]);
            if (J.Rout) J.Rout[(size_t)i * J.r_node_stride + (size_t)r * J.r_row_stride + g] = res;
            nr += cnorm2(res);
            nb += cnorm2(b);
        }
        nr += __shfl_xor_sync(0xffffffffu, nr, 16);
        nb += __shfl_xor_sync(0xffffffffu, nb, 16);
        if ((threadIdx.x & 16) == 0) {
            atomicAdd(&sr[cl], nr);
            if (ends) atomicAdd(&sb[cl], nb);
        }
    }
    __syncthreads();
    if (threadIdx.x < T && c0 + (int)threadIdx.x < m) {
        atomicAdd(&J.rn2[c0 + threadIdx.x], sr[threadIdx.x]);
        if (ends) atomicAdd(&J.bn2[c0 + threadIdx.x], sb[threadIdx.x]);
    }
}

// ---------------------------------------------------------------- whole sweep in one CTA
// One CTA per energy, the augmented node block [S | U_i | y] (n rows) in shared memory, as
// is the previous node's [X | y].  Rows are not moved (see lu_cluster.cuh); warp 0 updates
// the next pivot column and searches it while the other warps update the rest.  Bounded by
// the chain of n pivots per node (about 1000 cycles each, the reciprocal 430 of them).
constexpr int SMALL_N = 24;

size_t small_smem(int n, int m) {
    const size_t w = (size_t)n + m;
    return sizeof(double2) * ((size_t)n * (n + w + 1) + (size_t)n * w + (size_t)n * n + (n + w) + n + 2 * (size_t)n * m) + sizeof(int) * 2 * n + 64;
}

__global__ void __launch_bounds__(128) k_sweep_small(SweepSys sys, const SweepJob* __restrict__ jobs) {
    extern __shared__ __align__(16) double2 sv[];
    const SweepJob J = jobs[blockIdx.x];
    const int n = sys.n, N = sys.N, ms = J.ms, m = J.ms + J.md, w = n + m, la = n + w + 1;
    const int t = threadIdx.x, NTS = blockDim.x, warp = t >> 5, lane = t & 31;
    double2* A = sv;                      // n x la: [S | U | y]
    double2* P = A + (size_t)n * la;      // n x w: [X | y] of the previous node
    double2* Lm = P + (size_t)n * w;      // n x n: L_i
    double2* urow = Lm + (size_t)n * n;   // n + w
    double2* invs = urow + n + w;         // n
    double2* cc = invs + n;               // 2 x n x m: c_{i+1}, c_i
    int* step = reinterpret_cast<int*>(cc + 2 * (size_t)n * m);
    int* prow = step + n;                 // pivot row of step j
    __shared__ int sel, szero;
    __shared__ double2 sinv;
    const double E = J.E;
    int bad = 0;
    // warp 0: best row of column c not used yet (n <= 32: a lane per row)
    auto search = [&](int c) {
        const bool in = lane < n && step[lane] < 0;
        const double2 p = in ? A[(size_t)lane * la + c] : make_double2(1, 0);
        const bool z = p.x == 0.0 && p.y == 0.0;
        const double2 inv = z ? make_double2(1, 0) : lu::inverse(p);       // every row's, beside the search
        if (lu::warp_best(in ? lu::mag_key(fabs(p.x) + fabs(p.y)) : 0ull) == lane) {
            sel = lane;
            szero = z;
            sinv = inv;
        }
    };
    for (int i = 0; i < N; ++i) {
        const double2* HV0 = hv0_of(sys, J, i);
        const double2* HV1 = i < N - 1 ? hv1_of(sys, J, i) : nullptr;
        if (i > 0) {
            const double2* HVm = hv1_of(sys, J, i - 1);
            for (int q = t; q < n * n; q += NTS) {
                const int k = q / n, r = q % n;
                Lm[r * n + k] = cconj(csub(cscale(sys.M1[q], E), HVm[q]));
            }
        }
        for (int r = t; r < n; r += NTS) step[r] = -1;
        __syncthreads();
        const int yc = y_cols(J, i == N - 1, false);
        const int x0 = i < N - 1 ? n : 2 * n, xe = 2 * n + yc;       // right-hand sides in use
        for (int q = t; q < n * (n + w); q += NTS) {
            const int r = q / (n + w), c = q % (n + w), g = c - 2 * n;
            double2 v = make_double2(0, 0);
            if (c < n) {
                const size_t u = (size_t)r * n + c;
                v = csub(cscale(sys.M0[u], E), HV0[u]);
                if (i == 0 && J.sig_s) v = csub(v, J.sig_s[u]);
                if (i == N - 1 && J.sig_d) v = csub(v, J.sig_d[u]);
            } else if (c < 2 * n) {
                const size_t u = (size_t)r * n + (c - n);
                if (i < N - 1) v = csub(cscale(sys.M1[u], E), HV1[u]);
            } else {
                if (i == 0 && g < ms) v = J.rhs_s[(size_t)r * ms + g];
                if (i == N - 1 && g >= ms) v = J.rhs_d[(size_t)r * J.md + (g - ms)];
            }
            if (i > 0 && (c < n || (g >= 0 && g < ms))) {
                const double2* l = Lm + r * n;
                const double2* p = P + (c < n ? c : n + g);
                double2 s = make_double2(0, 0);
                for (int k = 0; k < n; ++k) cfma(s, l[k], p[(size_t)k * w]);
                v = csub(v, s);
            }
            A[(size_t)r * la + c] = v;
        }
        __syncthreads();
        if (warp == 0) search(0);
        for (int j = 0; j < n; ++j) {
            __syncthreads();
            const int p = sel;
            const double2 inv = sinv;
            bad |= szero;
            // columns in use right of j: the rest of S, then x0 .. xe
            const int cs = n - 1 - j, nc = cs + (xe - x0);
            for (int q = t; q < nc; q += NTS) {
                const int c = q < cs ? j + 1 + q : x0 + q - cs;
                urow[c] = cmul(A[(size_t)p * la + c], inv);
            }
            if (t == 0) {
                step[p] = j;
                prow[j] = p;
                invs[j] = inv;
            }
            __syncthreads();
            if (warp == 0 && j + 1 < n) {
                if (lane < n && step[lane] < 0) {
                    double2* a = A + (size_t)lane * la;
                    a[j + 1] = lu::fnma(a[j + 1], a[j], urow[j + 1]);
                }
                __syncwarp();
                search(j + 1);
            }
            const int skip = j + 1 < n ? 1 : 0, items = (nc - skip) * n;
            // warp 0 is in the search: the other warps take the items
            if (warp > 0)
                for (int q = t - 32; q < items; q += NTS - 32) {
                    const int r = q / (nc - skip), x = skip + q % (nc - skip);
                    if (step[r] >= 0) continue;
                    const int c = x < cs ? j + 1 + x : x0 + x - cs;
                    double2* a = A + (size_t)r * la;
                    a[c] = lu::fnma(a[c], a[j], urow[c]);
                }
        }
        __syncthreads();
        // back substitution, a thread per column; [X_i | y_i] to P and to the panel
        double2* R = J.XY + (size_t)i * n * w;
        for (int c = t; c < w; c += NTS) {
            const int ac = n + c;
            const bool used = ac >= x0 && ac < xe;
            for (int j = n - 1; j >= 0; --j) {
                double2 x = make_double2(0, 0);
                if (used) {
                    x = cmul(A[(size_t)prow[j] * la + ac], invs[j]);
#pragma unroll 4
                    for (int q = 0; q < j; ++q) {
                        double2* a = A + (size_t)prow[q] * la;
                        a[ac] = lu::fnma(a[ac], a[j], x);
                    }
                }
                P[(size_t)j * w + c] = x;
                R[(size_t)j * w + c] = x;
            }
        }
        __syncthreads();
    }
    double2 *cur = cc, *nxt = cc + (size_t)n * m;
    for (int q = t; q < n * m; q += NTS) cur[q] = P[(size_t)(q / m) * w + n + q % m];
    for (int i = N - 2; i >= 0; --i) {
        double2* R = J.XY + (size_t)i * n * w;
        __syncthreads();
        for (int q = t; q < n * m; q += NTS) {
            const int r = q / m, g = q % m;
            const double2* x = R + (size_t)r * w;
            double2 s = make_double2(0, 0);
#pragma unroll 4
            for (int k = 0; k < n; ++k) cfma(s, x[k], cur[k * m + g]);
            double2& y = R[(size_t)r * w + n + g];
            const double2 v = csub(y, s);
            y = v;
            nxt[q] = v;
        }
        double2* s = cur;
        cur = nxt;
        nxt = s;
    }
    if (t == 0 && bad) atomicOr(J.status, PWQT_ST_SINGULAR_PIVOT);
}

// ---------------------------------------------------------------- host side
namespace {

// columns per CTA so that `cols` columns of nb energies fill the SMs once, at most 32
int column_block(int cols, int nb, int sms, size_t per_col, size_t fixed, int smem_max, int least) {
    const int fit = (int)std::min<size_t>(32, ((size_t)smem_max - fixed) / per_col);
    for (int waves = 1;; ++waves) {
        int cb = (int)(((long long)cols * nb + (long long)sms * waves - 1) / ((long long)sms * waves));
        cb = std::max(cb, least);
        while (cb <= fit && (long long)((cols + cb - 1) / cb) * nb > (long long)sms * waves) ++cb;   // ragged blocks
        if (cb <= fit) return cb;
        if (waves > cols * nb) return fit;
    }
}

template <bool GREEN>
int sweep_tiled(const SweepSys& sys, const SweepJob* jobs, const SweepJob* host, int nb, int C, int sms, int smem_max, cudaStream_t st) {
    const int n = sys.n, N = sys.N;
    int ms = 0, m = 0, launches = 0;
    for (int b = 0; b < nb; ++b) { ms = std::max(ms, host[b].ms); m = std::max(m, host[b].ms + host[b].md); }
    const Where64 where{jobs, sys};
    // 32 x 32 tiles once they give every SM two CTAs, else 16 x 16: an SM takes 38 000 cycles
    // for 16 x 16 x 64, so the spread over SMs matters more than the operand traffic
    const int t32 = (n + 31) / 32, t16 = (n + 15) / 16;
    const bool big = (long long)t32 * t32 * nb >= 2 * sms;
    auto attr = [&](const void* f) { cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max); };
    attr((const void*)k_solve<GREEN>);
    attr((const void*)k_back);
    for (int i = 0; i < N; ++i) {
        const bool last = i == N - 1;
        const int yc = GREEN ? 0 : (last ? m : ms);
        if (big) k_node<2, GREEN><<<dim3(t32 + (yc + 31) / 32, t32, nb), 256, 0, st>>>(sys, jobs, i);
        else k_node<1, GREEN><<<dim3(t16 + (yc + 15) / 16, t16, nb), 256, 0, st>>>(sys, jobs, i);
        lu::launch(where, n, nb, C, st);
        launches += 2;
        const int cols = (last ? 0 : n) + (GREEN ? n : yc);
        if (cols > 0) {
            const int cb = column_block(cols, nb, sms, sizeof(double2) * n, solve_smem(n, 0), smem_max, 2);
            k_solve<GREEN><<<dim3((cols + cb - 1) / cb, nb), 256, solve_smem(n, cb), st>>>(sys, jobs, i, cb);
            ++launches;
        }
    }
    if (GREEN) {
        for (int i = N - 2; i >= 0; --i)
            for (int stage = 0; stage < 3; ++stage) {
                if (big) k_green_product<2><<<dim3(t32, t32, nb), 256, 0, st>>>(sys, jobs, i, stage);
                else k_green_product<1><<<dim3(t16, t16, nb), 256, 0, st>>>(sys, jobs, i, stage);
                ++launches;
            }
        k_green_dos<<<dim3(N, nb), 256, 0, st>>>(n, jobs);
        ++launches;
    } else if (m > 0) {
        const int cb = column_block(m, nb, sms, 2 * sizeof(double2) * n, 0, smem_max, 1);
        int ks = 1;
        while (ks < 16 && 2 * ks * n * cb <= 256) ks *= 2;
        k_back<<<dim3((m + cb - 1) / cb, nb), 256, back_smem(n, cb), st>>>(sys, jobs, cb, ks);
        ++launches;
    }
    return launches;
}

template <bool GREEN>
int sweep_any(const SweepSys& sys, const SweepJob* jobs, const SweepJob* host, int nb, cudaStream_t st) {
    int dev = 0, sms = 0, smem_max = 0, m = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    for (int b = 0; b < nb; ++b) m = std::max(m, host[b].ms + host[b].md);
    if (!GREEN && sys.n <= SMALL_N && small_smem(sys.n, m) <= (size_t)smem_max - 1024) {
        cudaFuncSetAttribute(k_sweep_small, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max - 1024);
        k_sweep_small<<<nb, 128, small_smem(sys.n, m), st>>>(sys, jobs);
        return 1;
    }
    const int C = lu::pick_cluster<Where64>(sys.n, nb, sms, smem_max);
    // the solve's shared memory for 4 columns is below the factorisation's limit at any n that has a cluster
    if (C > 0 && nb <= 65535 && solve_smem(sys.n, 4) <= (size_t)smem_max) return sweep_tiled<GREEN>(sys, jobs, host, nb, C, sms, smem_max, st);
    k_sweep_fp64<GREEN><<<nb, NT, 0, st>>>(sys, jobs);
    return 1;
}
}  // namespace

int launch_sweep_fp64(const SweepSys& sys, const SweepJob* jobs, const SweepJob* host, int nb, cudaStream_t st) {
    return sweep_any<false>(sys, jobs, host, nb, st);
}

void launch_residual_fp64(const SweepSys& sys, const ResJob* jobs, int m, int nb, cudaStream_t st) {
    if (m > 0) {
        const int t32 = (sys.n + 31) / 32, t16 = (sys.n + 15) / 16, c32 = (m + 31) / 32, c16 = (m + 15) / 16;
        // 32 x 32 tiles unless 16 x 16 ones cover the rows and columns with a tenth less
        if (10ll * t16 * c16 >= 36ll * t32 * c32) k_residual_fp64<2><<<dim3(sys.N, t32 * c32, nb), 256, 0, st>>>(sys, jobs);
        else k_residual_fp64<1><<<dim3(sys.N, t16 * c16, nb), 256, 0, st>>>(sys, jobs);
    }
    launch_residual_finish(jobs, nb, st);
}

int launch_green_fp64(const SweepSys& sys, const SweepJob* jobs, const SweepJob* host, int nb, cudaStream_t st) {
    return sweep_any<true>(sys, jobs, host, nb, st);
}

}  // namespace pwqt
