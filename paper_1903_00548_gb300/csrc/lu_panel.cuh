// LU factorisation of one n x n complex64 block per energy in panels of 8 columns, by one
// CTA or a small cluster of CTAs.
//
// The columns are dealt out in blocks of 8 (block b to CTA b % C) and stay in shared
// memory, row r of a block in 64 consecutive bytes; a factored panel takes its block's place
// column by column (a lane per row stores without bank conflicts, which rows of 64 bytes
// would cost 400 cycles a column).  The owner of the next panel brings it up to date, then
// up to 4 warps factor it in registers (RPL rows a lane, 8 columns each) while the other
// warps update the remaining blocks with the panel before.  Rows are not moved: a
// row that has served as pivot is left alone and its part of U goes to the output as soon
// as it is known; at the end row r of L is written where its pivot step says.  Factors of
// P A with partial pivoting (max |re| + |im|), unit lower triangle, (P x)_j = x[perm[j]].
//
// Bound: the chain of n pivots, about 500 cycles a column, with the panel held in the
// registers of up to 4 warps (a row or a few per lane): search by REDUX, candidates with
// their rows and reciprocals through shared memory, one named barrier, the rank-1 update of
// what is left of 8 columns.  Measured at n = 128, 16 energies: 92 us; 190 us with a pivot
// exchanged over the cluster per column (lu_cluster.cuh, which the FP64 sweep keeps: a
// warp's FP64 update of its panel rows would take thousands of cycles a column), 217 us with
// one warp holding the panel.
#pragma once
#include "lu_cluster.cuh"
#include "sweep_common.cuh"

namespace pwqt {
namespace lup {

constexpr int PB = 8;            // panel columns
constexpr int NT = 256;

// a panel warp's best row for one column
struct __align__(16) Cand {
    float2 u[PB];            // the row, current column first
    float2 inv;              // reciprocal of u[0]
    int row, zero;           // zero: u[0] is exactly zero
};
// what the panel warps share: candidates and their magnitudes, two columns in turn
struct __align__(16) PanelMem { Cand c[2][4]; unsigned key[2][4]; float2 trash[128]; };

inline int blocks_of(int n) { return (n + PB - 1) / PB; }
inline size_t smem_bytes(int n, int C) {
    const int bl = (blocks_of(n) + C - 1) / C;
    return (size_t)(bl + 1) * n * PB * sizeof(float2) + sizeof(PanelMem) + sizeof(int) * (n + 2 * PB);
}

// u[k] of column `cl` of block V: the panel's 8 pivot rows through its unit lower triangle
__device__ __forceinline__ void pivot_rows(const float2* V, const float2* lp, int n, const int* pv, int cl, float2 (&u)[PB]) {
    int p[PB];
#pragma unroll
    for (int k = 0; k < PB; ++k) p[k] = pv[k];
#pragma unroll
    for (int k = 0; k < PB; ++k) u[k] = V[p[k] * PB + cl];
#pragma unroll
    for (int q = 0; q + 1 < PB; ++q)
#pragma unroll
        for (int k = q + 1; k < PB; ++k) u[k] = lu::fnma(u[k], lp[q * n + p[k]], u[q]);
}

// rows [r0, r1) of B neighbouring local blocks at V: V[r][.] -= l[r][.] u, rows used as pivots
// left alone.  A warp: 16 rows x 8 B columns a step; with two blocks the multipliers are read
// once for both (one block alone is bound by shared-memory reads, 11 to 32 FMAs).
template <int B>
__device__ __forceinline__ void update_rows(float2* V, const float2* lp, int n, const int* step, const float2 (&u)[B][PB], int r0, int r1, int lane) {
    const int cl = lane & 7;
    for (int r = r0 + (lane >> 3); r < r1; r += 16) {
        float2 v[4][B];
        int x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            x[q] = min(r + 4 * q, n - 1);
#pragma unroll
            for (int b = 0; b < B; ++b) v[q][b] = V[((size_t)b * n + x[q]) * PB + cl];
        }
#pragma unroll
        for (int k = 0; k < PB; ++k)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 l = lp[k * n + x[q]];
#pragma unroll
                for (int b = 0; b < B; ++b) v[q][b] = lu::fnma(v[q][b], l, u[b][k]);
            }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (r + 4 * q < r1 && step[x[q]] < 0)
#pragma unroll
                for (int b = 0; b < B; ++b) V[((size_t)b * n + x[q]) * PB + cl] = v[q][b];
    }
}

// local blocks x, .. x + B - 1 (global block x C + rank) by panel p: rows [r0, r1), and the
// panel's rows of U to F when r0 is 0
template <int B>
__device__ __forceinline__ void update_blocks(float2* V, const float2* lp, float2* F, int n, const int* pv, const int* step, int p, int x,
                                              int C, int rank, int r0, int r1, int lane) {
    float2 u[B][PB];
    float2* Q = V + (size_t)x * n * PB;
#pragma unroll
    for (int b = 0; b < B; ++b) pivot_rows(Q + (size_t)b * n * PB, lp, n, pv, lane & 7, u[b]);
    update_rows<B>(Q, lp, n, step, u, r0, r1, lane);
    if (r0 == 0 && lane < PB)
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const int col = ((x + b) * C + rank) * PB + lane;
            if (col < n)
#pragma unroll
                for (int k = 0; k < PB; ++k) F[(size_t)(p * PB + k) * n + col] = u[b][k];
        }
}

// W warps (threads 0 .. 32 W - 1, RPL rows a lane): the panel V (n rows, wd columns) with
// the rows marked in step already used, left as V[k n + r]; its pivots to pv (a NaN counts
// as the largest).  Returns whether a pivot was exactly zero.
template <int W, int RPL>
__device__ __forceinline__ int factor_panel(float2* V, const int* step, int n, int wd, int* pv, PanelMem& pm) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    float2 a[RPL][PB];
    unsigned done = 0;       // rows of this lane that are used
    int bad = 0;
#pragma unroll
    for (int q = 0; q < RPL; ++q) {
        const int r = t + 32 * W * q;
        const bool on = r < n && step[min(r, n - 1)] < 0;
        if (!on) done |= 1u << q;
#pragma unroll
        for (int c = 0; c < PB; c += 2) {
            const float4 v = *reinterpret_cast<const float4*>(V + min(r, n - 1) * PB + c);
            a[q][c] = make_float2(v.x, v.y);
            a[q][c + 1] = make_float2(v.z, v.w);
        }
    }
    auto sync = [] { asm volatile("bar.sync 1, %0;" :: "n"(32 * W) : "memory"); };
    sync();                  // all rows are in registers
    // the current column is always a[.][0]: the update moves the others one to the left, so
    // that one short loop body serves all columns
#pragma unroll 1
    for (int k = 0; k < wd; ++k) {
        unsigned bk = 0;
        int bq = 0;
#pragma unroll
        for (int q = 0; q < RPL; ++q) {
            unsigned key = __float_as_uint(fabsf(a[q][0].x) + fabsf(a[q][0].y)) + 1u;
            key = (done >> q) & 1u ? 0u : key;
            if (key > bk) { bk = key; bq = q; }
        }
        float2 b[PB];        // this lane's candidate
#pragma unroll
        for (int c = 0; c < PB; ++c) {
            b[c] = a[0][c];
#pragma unroll
            for (int q = 1; q < RPL; ++q) b[c] = bq == q ? a[q][c] : b[c];
        }
        const bool zero = b[0].x == 0.f && b[0].y == 0.f;
        const float2 inv = lu::inverse(zero ? make_float2(1.f, 0.f) : b[0]);
        const int win = lu::warp_best(bk), par = k & 1;
        if (lane == win) {
            Cand& s = pm.c[par][warp];
#pragma unroll
            for (int c = 0; c < PB; c += 2) *reinterpret_cast<float4*>(&s.u[c]) = make_float4(b[c].x, b[c].y, b[c + 1].x, b[c + 1].y);
            s.inv = inv;
            s.row = t + 32 * W * bq;
            s.zero = zero;
            pm.key[par][warp] = bk;
        }
        sync();
        int w = 0;
        if (W > 1) {
            const uint4 kk = *reinterpret_cast<const uint4*>(pm.key[par]);
            unsigned best = kk.x;
            if (kk.y > best) { best = kk.y; w = 1; }
            if (W > 2 && kk.z > best) { best = kk.z; w = 2; }
            if (W > 3 && kk.w > best) w = 3;
        }
        const Cand& s = pm.c[par][w];
        float2 u[PB];
#pragma unroll
        for (int c = 0; c < PB; c += 2) {
            const float4 v = *reinterpret_cast<const float4*>(&s.u[c]);
            u[c] = make_float2(v.x, v.y);
            u[c + 1] = make_float2(v.z, v.w);
        }
        const float2 iv = s.inv;
        const int row = s.row;
        bad |= s.zero;
        if (t == 0) pv[k] = row;
#pragma unroll
        for (int q = 0; q < RPL; ++q) {
            const int r = t + 32 * W * q;
            if (r == row) done |= 1u << q;
            // no branch: rows that are done get a zero multiplier, those past n go to trash
            const bool on = !((done >> q) & 1u);
            float2 l = lu::mul(a[q][0], iv);
            *(r < n ? V + k * n + r : pm.trash + t) = on ? l : a[q][0];
            l = on ? l : make_float2(0.f, 0.f);
#pragma unroll
            for (int c = 1; c < PB; ++c) a[q][c - 1] = lu::fnma(a[q][c], l, u[c]);
            a[q][PB - 1] = make_float2(0.f, 0.f);
        }
    }
    return bad;
}

// Blocks of a batch: entry e of S (factored in place) and perm
struct Batch {
    float2* S; long long stride;     // n x n, row stride n
    int* perm; long long sperm;
    const SweepJob* jobs;
};

template <int W, int RPL>
__global__ void __launch_bounds__(NT) k_lu_panel(Batch B, int n) {
    extern __shared__ __align__(16) float2 lsm[];
    const uint32_t C = lu::cl_size(), rank = lu::cl_rank();
    const int e = blockIdx.x / C, t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int nbk = (n + PB - 1) / PB, bl = (nbk + (int)C - 1) / (int)C, own = (nbk - (int)rank + (int)C - 1) / (int)C;
    float2* F = B.S + e * B.stride;
    float2* V = lsm;                                // local block x: V + x n PB
    float2* lbuf = lsm + (size_t)bl * n * PB;       // the panel in use (C > 1)
    PanelMem& pm = *reinterpret_cast<PanelMem*>(lbuf + (size_t)n * PB);
    int* step = reinterpret_cast<int*>(&pm + 1);
    int* pv = step + n;                             // pivots of the panel this CTA factored
    int* cur = pv + PB;                             // pivots of the panel in use
    for (int q = t; q < own * n * PB; q += NT) {
        const int c = q % PB, x = (q / PB) % own, r = q / (PB * own), col = (x * (int)C + (int)rank) * PB + c;
        V[((size_t)x * n + r) * PB + c] = col < n ? F[(size_t)r * n + col] : make_float2(0.f, 0.f);
    }
    for (int r = t; r < n; r += NT) step[r] = -1;
    __syncthreads();
    if (C > 1) lu::cl_sync();      // S is read everywhere before U rows go over it
    int bad = 0;
    if (rank == 0 && warp < W) bad |= factor_panel<W, RPL>(V, step, n, min(PB, n), pv, pm);
    for (int p = 0; p < nbk; ++p) {
        const int wd = min(PB, n - p * PB), owner = p % (int)C;
        if (C > 1) lu::cl_sync();
        else __syncthreads();
        // the factored panel and its pivots
        const float2* panel = V + (size_t)(p / (int)C) * n * PB;
        const int* ppv = pv;
        if (C > 1) {
            const float4* src = reinterpret_cast<const float4*>(lu::cl_map(V + (size_t)(p / (int)C) * n * PB, (uint32_t)owner));
            ppv = lu::cl_map(pv, (uint32_t)owner);
            if ((int)rank != owner) {
                for (int q = t; q < n * PB / 2; q += NT) reinterpret_cast<float4*>(lbuf)[q] = src[q];
                panel = lbuf;
            }
        }
        if (t < wd) {
            const int r = ppv[t];
            cur[t] = r;
            step[r] = p * PB + t;
        }
        __syncthreads();
        if (p + 1 == nbk) break;
        const bool next = (p + 1) % (int)C == (int)rank;       // this CTA owns the next panel
        const int xn = (p + 1) / (int)C;
        if (next) {
            // the next panel first, a share of its rows per warp
            float2* Q = V + (size_t)xn * n * PB;
            const int share = ((n + 7) / 8 + 3) / 4 * 4;
            update_blocks<1>(V, panel, F, n, cur, step, p, xn, (int)C, (int)rank, warp * share, min(n, (warp + 1) * share), lane);
            __syncthreads();
            if (warp < W) bad |= factor_panel<W, RPL>(Q, step, n, min(PB, n - (p + 1) * PB), pv, pm);
        }
        // blocks past p, but not the next panel again: (block, row chunk) per warp
        const int x0 = next ? xn + 1 : (p + 1 - (int)rank + (int)C - 1) / (int)C;
        const int chunk = n > 64 ? 64 : 32, chunks = (n + chunk - 1) / chunk, left = own - x0;
        const int w0 = next ? (warp + 8 - W) % 8 : warp;       // the factoring warps join last
        for (int q = w0; q < (left + 1) / 2 * chunks; q += 8) {
            const int x = x0 + q / chunks * 2, r0 = q % chunks * chunk, r1 = min(n, r0 + chunk);
            if (x + 1 < own) update_blocks<2>(V, panel, F, n, cur, step, p, x, (int)C, (int)rank, r0, r1, lane);
            else update_blocks<1>(V, panel, F, n, cur, step, p, x, (int)C, (int)rank, r0, r1, lane);
        }
    }
    if (C > 1) lu::cl_sync();      // no CTA leaves while its panels may be read
    // L, and U inside the panels' diagonal blocks
    for (int q = t; q < own * n * PB; q += NT) {
        const int c = q % PB, x = (q / PB) % own, r = q / (PB * own), k0 = (x * (int)C + (int)rank) * PB;
        if (k0 + c < n && step[r] >= k0) F[(size_t)step[r] * n + k0 + c] = V[((size_t)x * PB + c) * n + r];
    }
    if (rank == 0) {
        int* perm = B.perm + e * B.sperm;
        for (int r = t; r < n; r += NT) perm[step[r]] = r;
    }
    if (bad && lane == 0) atomicOr(B.jobs[e].status, PWQT_ST_SINGULAR_PIVOT);
}

// CTAs per energy; 0: none holds the block.  One CTA's updates keep up with the panel chain
// to n = 80; above, they are spread over 4 (measured, 16 energies: n = 128 121 us on one CTA,
// 104 on 2, 92 on 4, 107 on 8; n = 256 293 us on 4, 343 on 8: a larger cluster pays for the
// panel's copy and the cluster barrier; a whole mixed solve of 30 nodes on 4 against 8: 32
// energies n = 256 74.3 and 75.5 ms, n = 320 121 and 138, but one energy 17.0 and 16.7, 26.0
// and 25.5).
// 320 is where the form's tests end, not where it stops paying: with 3 rows a lane and 8 CTAs
// (shared memory holds n <= 440 or so) a mixed solve of 30 nodes takes, against the tensor-core
// form, 16 energies n = 340 96 and 118 ms, n = 384 119 and 151; one energy 29 and 61, 38 and 74.
inline int pick_cluster(int n, int smem_max) {
    if (n > 320) return 0;
    for (int C = n <= 80 ? 1 : 4; C <= 8; C *= 2)
        if (smem_bytes(n, C) <= (size_t)smem_max) return C;
    return 0;
}

inline cudaError_t launch(const Batch& B, int n, int nb, int C, int smem_max, cudaStream_t st) {
    cudaLaunchConfig_t cf{};
    cudaLaunchAttribute at{};
    cf.gridDim = dim3(C * nb);
    cf.blockDim = dim3(NT);
    cf.dynamicSmemBytes = smem_bytes(n, C);
    cf.stream = st;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = C;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cf.attrs = &at;
    cf.numAttrs = 1;
    auto go = [&](auto* f) {
        cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
        return cudaLaunchKernelEx(&cf, f, B, n);
    };
    if (n <= 32) return go(k_lu_panel<1, 1>);
    if (n <= 64) return go(k_lu_panel<2, 1>);
    if (n <= 128) return go(k_lu_panel<4, 1>);
    if (n <= 256) return go(k_lu_panel<4, 2>);
    return go(k_lu_panel<4, 3>);
}

}  // namespace lup
}  // namespace pwqt
