// LU factorisation of one n x n complex128 block per energy by a thread-block cluster (the
// FP64 sweep's; the arithmetic helpers also serve the complex64 panels of lu_panel.cuh).
//
// The block's rows are dealt out over the cluster's C CTAs (row r to CTA r % C) and stay
// in shared memory for the whole factorisation; nothing is exchanged but the pivot: per
// column every CTA proposes its best row (max |re| + |im|), the winner's row is read through
// distributed shared memory, and each CTA updates its own rows.  Rows are not moved: a row that has served as pivot is left alone, and at the end
// row j of the factors is written from where the j-th pivot sat, with perm[j] its index
// (the factors are those of P A, (P x)_j = x[perm[j]]; unit lower triangle).
//
// Bound.  One column is a chain: cluster barrier, choice of the winner, multipliers, update
// of the next column, its search, the reciprocal of its pivot.  Measured on GB300 (cycles):
// cluster barrier 390 at any size, distributed shared-memory read 240, and 64 per FP64
// instruction of a warp whatever its lanes or its dependences do (two lanes per clock and
// SM), so a complex multiply-add is 256 and a reciprocal 430.  Hence: comparisons on the
// integer patterns of the magnitudes (REDUX, not FP64 compares), real and imaginary parts in
// neighbouring lanes on the chain, every row's reciprocal computed beside the search rather
// than after it, and warp 0 updating and searching the next column while the other warps
// update the rest.  The update runs from shared memory as rank-1 steps: FP64-bound (256
// cycles per 32 elements against 12 of shared memory), so panels would gain nothing.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>

#include "pwqt_internal.cuh"

namespace pwqt {
namespace lu {

template <class T2> struct Real;
template <> struct Real<double2> { using t = double; };
template <> struct Real<float2> { using t = float; };

template <class T2> __device__ __forceinline__ T2 make2(typename Real<T2>::t x, typename Real<T2>::t y) {
    T2 r;
    r.x = x;
    r.y = y;
    return r;
}
template <class T2> __device__ __forceinline__ T2 mul(T2 a, T2 b) { return make2<T2>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
// a - b c
template <class T2> __device__ __forceinline__ T2 fnma(T2 a, T2 b, T2 c) {
    a.x = fma(-b.x, c.x, fma(b.y, c.y, a.x));
    a.y = fma(-b.x, c.y, fma(-b.y, c.x, a.y));
    return a;
}
// |a|^2 well inside the range of normal numbers (by its exponent bits)
__device__ __forceinline__ bool plain(double d) { const unsigned e = ((unsigned)__double2hiint(d) >> 20) & 0x7ff; return e - 64u < 1900u; }
__device__ __forceinline__ bool plain(float d) { const unsigned e = (__float_as_uint(d) >> 23) & 0xff; return e - 10u < 230u; }
__device__ __forceinline__ double recip(double d) { return 1.0 / d; }
__device__ __forceinline__ float recip(float d) { return __frcp_rn(d); }
// 1 / a; Smith's form where |a|^2 leaves that range
template <class T2> __device__ __forceinline__ T2 inverse(T2 a) {
    using T = typename Real<T2>::t;
    const T d = fma(a.x, a.x, a.y * a.y);
    if (plain(d)) {
        const T s = recip(d);
        return make2<T2>(a.x * s, -a.y * s);
    }
    if (fabs(a.x) >= fabs(a.y)) {
        const T r = a.y / a.x, q = a.x + a.y * r;
        return make2<T2>(T(1) / q, -r / q);
    }
    const T r = a.x / a.y, q = a.x * r + a.y;
    return make2<T2>(r / q, -T(1) / q);
}

// Magnitudes as integers that compare alike: 0 no row, 1 not comparable (NaN), then the bit
// pattern of |re| + |im| above 1.
__device__ __forceinline__ unsigned long long mag_key(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return b <= 0x7ff0000000000000ull ? b + 2ull : 1ull;
}
// warp-wide: the first lane with the largest key
__device__ __forceinline__ int warp_best(unsigned long long key) {
    const unsigned hi = (unsigned)(key >> 32), lo = (unsigned)key;
    const bool in = hi == __reduce_max_sync(0xffffffffu, hi);
    const unsigned v = in ? lo : 0u, m = __reduce_max_sync(0xffffffffu, v);     // every lane takes part
    return __ffs(__ballot_sync(0xffffffffu, in && v == m)) - 1;
}
__device__ __forceinline__ int warp_best(unsigned key) {
    const unsigned m = __reduce_max_sync(0xffffffffu, key);
    return __ffs(__ballot_sync(0xffffffffu, key == m)) - 1;
}

// a CTA's proposal for one column: two 16-byte words
struct __align__(16) Slot {
    unsigned long long key;      // mag_key of the pivot
    int pos;                     // its place in the CTA's list of rows in use
    int row;                     // local row; bit 30: the pivot is exactly zero
    double2 inv;                 // its reciprocal
};

constexpr int MAX_CLUSTER = 16;

inline size_t smem_bytes(int n, int C) {
    const int rl = (n + C - 1) / C;
    return sizeof(double2) * ((size_t)rl * (n + 2) + n) + 16 + 2 * MAX_CLUSTER * sizeof(Slot) + sizeof(int) * 2 * rl;
}

__device__ __forceinline__ uint32_t cl_rank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ uint32_t cl_size() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ void cl_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// generic address of this CTA's shared object `p` in CTA `rank` of the cluster
template <class T> __device__ __forceinline__ T* cl_map(T* p, uint32_t rank) {
    unsigned long long out;
    asm volatile("mapa.u64 %0, %1, %2;" : "=l"(out) : "l"(reinterpret_cast<unsigned long long>(p)), "r"(rank));
    return reinterpret_cast<T*>(out);
}

// Where(e): {source, destination, row stride, perm, status} of energy e
struct Place { const double2* S; double2* F; int ld; int* perm; int* status; };

constexpr int ZERO_BIT = 1 << 30;

// Warp 0: column c of the rows in use brought up to date (v -= l u over the multipliers lm of
// the previous column; UPDATE false: as it stands), its best row found and proposed to every
// CTA of the cluster.  Lanes 2q, 2q + 1: real and imaginary part of one row.
template <bool UPDATE>
__device__ __forceinline__ void propose(double2* rows, int ldr, int na, const int* ord, const double2* lm, double2 u, int C,
                                        uint32_t rank, int c, Slot* slots, int par) {
    const int lane = threadIdx.x & 31, part = lane & 1;
    unsigned long long bk = 0;
    int bp = 0, br = 0;
    double bx = 1.0, by = 0.0;
    for (int q0 = 0; q0 < na; q0 += 16) {
        const int q = q0 + (lane >> 1);
        const bool in = q < na;
        const int r = ord[in ? q : 0];
        double2* a = rows + (size_t)r * ldr + c;
        double v = part ? a->y : a->x;
        if (UPDATE) {
            const double2 l = lm[r];
            // re: v - l.x u.x + l.y u.y;  im: v - l.x u.y - l.y u.x
            v = part ? fma(-l.x, u.y, fma(-l.y, u.x, v)) : fma(-l.x, u.x, fma(l.y, u.y, v));
            if (in) reinterpret_cast<double*>(a)[part] = v;
        }
        const double o = __shfl_xor_sync(0xffffffffu, v, 1);
        const unsigned long long k = in ? mag_key(fabs(v) + fabs(o)) : 0ull;
        if (q0 == 0 || k > bk) {
            bk = k;
            bp = q;
            br = r;
            bx = part ? o : v;
            by = part ? v : o;
        }
    }
    // the reciprocals of the lanes' own candidates, beside the search
    const bool zero = bx == 0.0 && by == 0.0;
    const double2 inv = inverse(zero ? make_double2(1.0, 0.0) : make_double2(bx, by));
    const int win = warp_best(bk);
    Slot* own = slots + par * MAX_CLUSTER + rank;
    if (lane == win) {
        own->key = bk;
        own->pos = bp;
        own->row = br | (zero ? ZERO_BIT : 0);
        own->inv = inv;
    }
    if (C > 1) {
        __syncwarp();
        const Slot s = *own;
        if (lane < C && lane != (int)rank) *cl_map(own, (uint32_t)lane) = s;
    }
}

template <class Where>
__global__ void __launch_bounds__(256) k_lu(Where where, int n) {
    extern __shared__ __align__(16) unsigned char lu_sm[];
    const uint32_t C = cl_size(), rank = cl_rank();
    const int e = blockIdx.x / C;
    const Place P = where(e);
    const int rl_max = (n + (int)C - 1) / (int)C;
    const int rl = (n - (int)rank + (int)C - 1) / (int)C;      // rows of this CTA
    const int ldr = n + 1, NT = blockDim.x, t = threadIdx.x, warp = t >> 5, lane = t & 31, nw = NT >> 5;
    double2* rows = reinterpret_cast<double2*>(lu_sm);
    double2* urow = rows + (size_t)rl_max * ldr;               // the pivot row
    double2* lm = urow + n;                                    // multipliers of the local rows
    Slot* slots = reinterpret_cast<Slot*>(lu_sm + (sizeof(double2) * ((size_t)rl_max * (ldr + 1) + n) + 15) / 16 * 16);
    int* step = reinterpret_cast<int*>(slots + 2 * MAX_CLUSTER);   // pivot step of a local row
    int* ord = step + rl_max;                                  // the rows not used yet: ord[0 .. na)
    for (int r = warp; r < rl; r += nw)
        for (int c = lane; c < n; c += 32) rows[(size_t)r * ldr + c] = P.S[(size_t)(r * (int)C + (int)rank) * P.ld + c];
    for (int r = t; r < rl; r += NT) ord[r] = r;
    int na = rl;
    __syncthreads();
    if (C > 1) cl_sync();       // every CTA runs before its shared memory is written from outside
    if (warp == 0) propose<false>(rows, ldr, na, ord, lm, make_double2(0.0, 0.0), (int)C, rank, 0, slots, 0);
    int bad = 0;
    for (int j = 0; j < n; ++j) {
        if (C > 1) cl_sync();
        else __syncthreads();
        // the winner, by every warp on its own
        const Slot* set = slots + (j & 1) * MAX_CLUSTER;
        const int w = C > 1 ? warp_best(lane < (int)C ? set[lane].key : 0ull) : 0;
        const int lr = set[w].row & ~ZERO_BIT;
        bad |= set[w].row & ZERO_BIT;
        const double2 inv = set[w].inv;
        const bool mine = w == (int)rank;
        const int wpos = set[w].pos;
        const double2* prow = (C > 1 ? cl_map(rows, (uint32_t)w) : rows) + (size_t)lr * ldr;
        double2 pv[4];          // the pivot row on its way while the multipliers are made (n <= 1024)
#pragma unroll
        for (int x = 0; x < 4; ++x)
            if (j + 1 + t + x * NT < n) pv[x] = prow[j + 1 + t + x * NT];
        // multipliers l = a inv, lanes 2q and 2q + 1 the real and imaginary part of one row's: both
        // read the entry, and the warp, whole in every pass, is past its reads before either
        // part is written (an exchange of the parts by shuffle instead: 0.7 % of a call at n = 64)
        for (int q0 = warp * 16; q0 < na; q0 += NT >> 1) {
            const int q = q0 + (lane >> 1), part = lane & 1, r = ord[min(q, na - 1)];
            double2* a = rows + (size_t)r * ldr + j;
            const double2 v = *a;
            const double l = part ? fma(v.x, inv.y, v.y * inv.x) : fma(v.x, inv.x, -(v.y * inv.y));
            __syncwarp();
            if (q < na && !(mine && r == lr)) {
                reinterpret_cast<double*>(lm + r)[part] = l;
                reinterpret_cast<double*>(a)[part] = l;
            }
        }
#pragma unroll
        for (int x = 0; x < 4; ++x)
            if (j + 1 + t + x * NT < n) urow[j + 1 + t + x * NT] = pv[x];
        __syncthreads();
        if (mine) {
            --na;
            if (t == 0) {
                step[lr] = j;
                ord[wpos] = ord[na];
            }
            __syncthreads();
        }
        if (j + 1 == n) break;
        if (warp == 0) propose<true>(rows, ldr, na, ord, lm, urow[j + 1], (int)C, rank, j + 1, slots, (j + 1) & 1);
        // A[r][c] -= l[r] u[c] over the rows in use and columns past j + 1; warp 0 joins when
        // it has proposed
        const int cols = n - j - 2;
        // items across row ends, so that no lane of a 64-cycle instruction is idle
        for (int q = (warp + nw - 1) % nw * 32 + lane; q < cols * na; q += NT) {
            const int r = ord[q / cols], c = j + 2 + q % cols;
            double2* a = rows + (size_t)r * ldr + c;
            *a = fnma(*a, lm[r], urow[c]);
        }
    }
    if (C > 1) cl_sync();       // no CTA leaves while its rows may be read; all reads of S are done
    for (int r = warp; r < rl; r += nw) {
        const int j = step[r];
        double2* out = P.F + (size_t)j * P.ld;
        for (int c = lane; c < n; c += 32) out[c] = rows[(size_t)r * ldr + c];
        if (lane == 0) P.perm[j] = r * (int)C + (int)rank;
    }
    if (bad && rank == 0 && t == 0) atomicOr(P.status, PWQT_ST_SINGULAR_PIVOT);
}

// Cluster size for nb blocks of n x n: the one with the least waves x max(chain, update).
// 0: no size holds the rows in shared memory.  Chain and update per column in cycles, from
// the measurements above: 1300 on one CTA, 1700 across a cluster, 2 per element of update.
template <class Where> int pick_cluster(int n, int nb, int sms, int smem_max) {
    int best = 0;
    double tb = 0;
    for (int C = 1; C <= MAX_CLUSTER; C *= 2) {
        const size_t sm = smem_bytes(n, C);
        if (sm > (size_t)smem_max || C > n) continue;
        cudaFuncSetAttribute(k_lu<Where>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
        cudaFuncSetAttribute(k_lu<Where>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        cudaLaunchConfig_t cf{};
        cudaLaunchAttribute at{};
        cf.gridDim = dim3(C);
        cf.blockDim = dim3(256);
        cf.dynamicSmemBytes = sm;
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = C;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cf.attrs = &at;
        cf.numAttrs = 1;
        int fit = 0;
        if (cudaOccupancyMaxActiveClusters(&fit, k_lu<Where>, &cf) != cudaSuccess || fit < 1) { cudaGetLastError(); continue; }
        const int run = std::min(nb, fit), waves = (nb + fit - 1) / fit, share = (run * C + sms - 1) / sms;
        const double chain = C == 1 ? 1300 : 1700;
        const double tt = waves * std::max(chain, (double)n * n / (3.0 * C) * 2.0 * share);
        if (!best || tt < tb) { best = C; tb = tt; }
    }
    return best;
}

template <class Where> cudaError_t launch(const Where& where, int n, int nb, int C, cudaStream_t st) {
    cudaLaunchConfig_t cf{};
    cudaLaunchAttribute at{};
    cf.gridDim = dim3(C * nb);
    cf.blockDim = dim3(256);
    cf.dynamicSmemBytes = smem_bytes(n, C);
    cf.stream = st;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = C;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cf.attrs = &at;
    cf.numAttrs = 1;
    return cudaLaunchKernelEx(&cf, k_lu<Where>, where, n);
}

}  // namespace lu
}  // namespace pwqt
