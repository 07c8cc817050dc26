// LU factorisation of one n x n complex block per energy by a thread-block cluster.
//
// The block's rows are dealt out over the cluster's C CTAs (row r to CTA r % C) and stay
// in shared memory for the whole factorisation; nothing is exchanged but the pivot: per
// column every CTA proposes its best row (max |re| + |im|), the winner's row is read through distributed shared memory, and each CTA updates its own
// rows.  Rows are not moved: a row that has served as pivot is left alone, and at the end
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
__device__ __forceinline__ unsigned mag_key(float v) {
    const unsigned b = __float_as_uint(v);
    return b <= 0x7f800000u ? b + 2u : 1u;
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

template <class T2> struct Key;
template <> struct Key<double2> { using t = unsigned long long; };
template <> struct Key<float2> { using t = unsigned; };

// a CTA's proposal for one column: two 16-byte words
template <class T2> struct __align__(16) Slot {
    typename Key<T2>::t key;     // mag_key of the pivot
    int pos;                     // its place in the CTA's list of rows in use
    int row;                     // local row; bit 30: the pivot is exactly zero
    T2 inv;                      // its reciprocal
};

constexpr int MAX_CLUSTER = 16;

template <class T2> size_t smem_bytes(int n, int C) {
    const int rl = (n + C - 1) / C;
    return sizeof(T2) * ((size_t)rl * (n + 2) + n) + 16 + 2 * MAX_CLUSTER * sizeof(Slot<T2>) + sizeof(int) * 2 * rl;
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
template <class T2> struct Place { const T2* S; T2* F; int ld; int* perm; int* status; };

constexpr int ZERO_BIT = 1 << 30;

// Warp 0: column c of the rows in use brought up to date (v -= l u over the multipliers lm of
// the previous column; UPDATE false: as it stands), its best row found and proposed to every
// CTA of the cluster.  Lanes 2q, 2q + 1: real and imaginary part of one row.
template <class T2, bool UPDATE>
__device__ __forceinline__ void propose(T2* rows, int ldr, int na, const int* ord, const T2* lm, T2 u, int C, uint32_t rank, int c,
                                        Slot<T2>* slots, int par) {
    using T = typename Real<T2>::t;
    const int lane = threadIdx.x & 31, part = lane & 1;
    using K = typename Key<T2>::t;
    K bk = 0;
    int bp = 0, br = 0;
    T bx = T(1), by = T(0);
    for (int q0 = 0; q0 < na; q0 += 16) {
        const int q = q0 + (lane >> 1);
        const bool in = q < na;
        const int r = ord[in ? q : 0];
        T2* a = rows + (size_t)r * ldr + c;
        T v = part ? a->y : a->x;
        if (UPDATE) {
            const T2 l = lm[r];
            // re: v - l.x u.x + l.y u.y;  im: v - l.x u.y - l.y u.x
            v = part ? fma(-l.x, u.y, fma(-l.y, u.x, v)) : fma(-l.x, u.x, fma(l.y, u.y, v));
            if (in) reinterpret_cast<T*>(a)[part] = v;
        }
        const T o = __shfl_xor_sync(0xffffffffu, v, 1);
        const K k = in ? mag_key(fabs(v) + fabs(o)) : K(0);
        if (q0 == 0 || k > bk) {
            bk = k;
            bp = q;
            br = r;
            bx = part ? o : v;
            by = part ? v : o;
        }
    }
    // the reciprocals of the lanes' own candidates, beside the search
    const bool zero = bx == T(0) && by == T(0);
    const T2 inv = inverse(zero ? make2<T2>(T(1), T(0)) : make2<T2>(bx, by));
    const int win = warp_best(bk);
    Slot<T2>* own = slots + par * MAX_CLUSTER + rank;
    if (lane == win) {
        own->key = bk;
        own->pos = bp;
        own->row = br | (zero ? ZERO_BIT : 0);
        own->inv = inv;
    }
    if (C > 1) {
        __syncwarp();
        const Slot<T2> s = *own;
        if (lane < C && lane != (int)rank) *cl_map(own, (uint32_t)lane) = s;
    }
}

template <class T2, class Where>
__global__ void __launch_bounds__(256) k_lu(Where where, int n) {
    using T = typename Real<T2>::t;
    extern __shared__ __align__(16) unsigned char lu_sm[];
    const uint32_t C = cl_size(), rank = cl_rank();
    const int e = blockIdx.x / C;
    const Place<T2> P = where(e);
    const int rl_max = (n + (int)C - 1) / (int)C;
    const int rl = (n - (int)rank + (int)C - 1) / (int)C;      // rows of this CTA
    const int ldr = n + 1, NT = blockDim.x, t = threadIdx.x, warp = t >> 5, lane = t & 31, nw = NT >> 5;
    T2* rows = reinterpret_cast<T2*>(lu_sm);
    T2* urow = rows + (size_t)rl_max * ldr;                    // the pivot row
    T2* lm = urow + n;                                         // multipliers of the local rows
    Slot<T2>* slots = reinterpret_cast<Slot<T2>*>(lu_sm + (sizeof(T2) * ((size_t)rl_max * (ldr + 1) + n) + 15) / 16 * 16);
    int* step = reinterpret_cast<int*>(slots + 2 * MAX_CLUSTER);   // pivot step of a local row
    int* ord = step + rl_max;                                  // the rows not used yet: ord[0 .. na)
    for (int r = warp; r < rl; r += nw)
        for (int c = lane; c < n; c += 32) rows[(size_t)r * ldr + c] = P.S[(size_t)(r * (int)C + (int)rank) * P.ld + c];
    for (int r = t; r < rl; r += NT) ord[r] = r;
    int na = rl;
    __syncthreads();
    if (C > 1) cl_sync();       // every CTA runs before its shared memory is written from outside
    if (warp == 0) propose<T2, false>(rows, ldr, na, ord, lm, make2<T2>(T(0), T(0)), (int)C, rank, 0, slots, 0);
    int bad = 0;
    for (int j = 0; j < n; ++j) {
        if (C > 1) cl_sync();
        else __syncthreads();
        // the winner, by every warp on its own
        const Slot<T2>* set = slots + (j & 1) * MAX_CLUSTER;
        using K = typename Key<T2>::t;
        const int w = C > 1 ? warp_best(lane < (int)C ? set[lane].key : K(0)) : 0;
        const int lr = set[w].row & ~ZERO_BIT;
        bad |= set[w].row & ZERO_BIT;
        const T2 inv = set[w].inv;
        const bool mine = w == (int)rank;
        const int wpos = set[w].pos;
        const T2* prow = (C > 1 ? cl_map(rows, (uint32_t)w) : rows) + (size_t)lr * ldr;
        T2 pv[4];               // the pivot row on its way while the multipliers are made (n <= 1024)
#pragma unroll
        for (int x = 0; x < 4; ++x)
            if (j + 1 + t + x * NT < n) pv[x] = prow[j + 1 + t + x * NT];
        // multipliers l = a inv, lanes 2q and 2q + 1 the real and imaginary part of one row's: a
        // lane reads and writes its own part only and has the other by shuffle
        for (int q0 = warp * 16; q0 < na; q0 += NT >> 1) {
            const int q = q0 + (lane >> 1), part = lane & 1, r = ord[min(q, na - 1)];
            T* a = reinterpret_cast<T*>(rows + (size_t)r * ldr + j) + part;
            const T v = q < na ? *a : T(0), o = __shfl_xor_sync(0xffffffffu, v, 1);
            const T l = part ? fma(o, inv.y, v * inv.x) : fma(v, inv.x, -(o * inv.y));
            if (q < na && !(mine && r == lr)) {
                reinterpret_cast<T*>(lm + r)[part] = l;
                *a = l;
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
        if (warp == 0) propose<T2, true>(rows, ldr, na, ord, lm, urow[j + 1], (int)C, rank, j + 1, slots, (j + 1) & 1);
        // A[r][c] -= l[r] u[c] over the rows in use and columns past j + 1; warp 0 joins when
        // it has proposed
        const int cols = n - j - 2;
        if (sizeof(T) == 8) {
            // items across row ends, so that no lane of a 64-cycle instruction is idle
            for (int q = (warp + nw - 1) % nw * 32 + lane; q < cols * na; q += NT) {
                const int r = ord[q / cols], c = j + 2 + q % cols;
                T2* a = rows + (size_t)r * ldr + c;
                *a = fnma(*a, lm[r], urow[c]);
            }
        } else {
            constexpr int RG = 8;       // rows at a time, loads before stores
            const int segs = (cols + 31) / 32, groups = (na + RG - 1) / RG;
            for (int q = (warp + nw - 1) % nw; q < segs * groups; q += nw) {
                const int c = min(j + 2 + q / groups * 32 + lane, n - 1), g = q % groups * RG;
                const bool in = j + 2 + q / groups * 32 + lane < n;
                const T2 u = urow[c];
                T2* a[RG];
                T2 v[RG];
#pragma unroll
                for (int x = 0; x < RG; ++x) {
                    const int r = ord[min(g + x, na - 1)];
                    a[x] = rows + (size_t)r * ldr + c;
                    v[x] = fnma(*a[x], lm[r], u);
                }
#pragma unroll
                for (int x = 0; x < RG; ++x)
                    if (in && g + x < na) *a[x] = v[x];
            }
        }
    }
    if (C > 1) cl_sync();       // no CTA leaves while its rows may be read; all reads of S are done
    for (int r = warp; r < rl; r += nw) {
        const int j = step[r];
        T2* out = P.F + (size_t)j * P.ld;
        for (int c = lane; c < n; c += 32) out[c] = rows[(size_t)r * ldr + c];
        if (lane == 0) P.perm[j] = r * (int)C + (int)rank;
    }
    if (bad && rank == 0 && t == 0) atomicOr(P.status, PWQT_ST_SINGULAR_PIVOT);
}

// Cluster size for nb blocks of n x n: the one with the least waves x max(chain, update).
// 0: no size holds the rows in shared memory.  Chain and update per column in cycles, from
// the measurements above: FP64 1300 on one CTA, 1700 across a cluster, 2 per element of
// update; FP32 450, 900 and 0.16.
template <class T2, class Where> int pick_cluster(int n, int nb, int sms, int smem_max) {
    const bool f64 = sizeof(T2) == 16;
    const double alpha = f64 ? 2.0 : 0.16;
    int best = 0;
    double tb = 0;
    for (int C = 1; C <= MAX_CLUSTER; C *= 2) {
        const size_t sm = smem_bytes<T2>(n, C);
        if (sm > (size_t)smem_max || C > n) continue;
        cudaFuncSetAttribute(k_lu<T2, Where>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
        cudaFuncSetAttribute(k_lu<T2, Where>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
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
        if (cudaOccupancyMaxActiveClusters(&fit, k_lu<T2, Where>, &cf) != cudaSuccess || fit < 1) { cudaGetLastError(); continue; }
        const int run = std::min(nb, fit), waves = (nb + fit - 1) / fit, share = (run * C + sms - 1) / sms;
        const double chain = C == 1 ? (f64 ? 1300 : 450) : (f64 ? 1700 : 900);
        const double tt = waves * std::max(chain, (double)n * n / (3.0 * C) * alpha * share);
        if (!best || tt < tb) { best = C; tb = tt; }
    }
    return best;
}

template <class T2, class Where> cudaError_t launch(const Where& where, int n, int nb, int C, cudaStream_t st) {
    cudaLaunchConfig_t cf{};
    cudaLaunchAttribute at{};
    cf.gridDim = dim3(C * nb);
    cf.blockDim = dim3(256);
    cf.dynamicSmemBytes = smem_bytes<T2>(n, C);
    cf.stream = st;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = C;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cf.attrs = &at;
    cf.numAttrs = 1;
    return cudaLaunchKernelEx(&cf, k_lu<T2, Where>, where, n);
}

}  // namespace lu
}  // namespace pwqt
