// LU factorisation of one n x n complex block per energy by a thread-block cluster.
//
// The block's rows are dealt out over the cluster's C CTAs (row r to CTA r % C) and stay
// in shared memory for the whole factorisation; nothing is exchanged but the pivot: per
// column every CTA proposes its best row (max |re| + |im|, the lower row on ties), the
// winner's row is read through distributed shared memory, and each CTA updates its own
// rows.  Rows are not moved: a row that has served as pivot is left alone, and at the end
// row j of the factors is written from where the j-th pivot sat, with perm[j] its index
// (the factors are those of P A, (P x)_j = x[perm[j]]; unit lower triangle).
//
// Bound.  One column is a chain: pivot search and reciprocal, cluster barrier, remote row
// read, update of the next column.  Warp 0 updates the next column first and searches it
// while the other warps update the rest, so a column costs the larger of the chain and the
// update.  Measured on GB300 (cycles): cluster barrier 390, distributed shared-memory read
// 240, FP64 reciprocal 430, FP64 FMA latency 64 at 1.7 FMA per clock and SM.  An FP64
// update is FMA-bound from shared memory (16 FMA cycles per element and warp against 3
// shared-memory cycles), so unblocked rank-1 steps lose nothing against panels.
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
// 1 / a; Smith's form where |a|^2 leaves the range of normal numbers
template <class T2> __device__ __forceinline__ T2 inverse(T2 a) {
    using T = typename Real<T2>::t;
    const T d = a.x * a.x + a.y * a.y;
    const T lo = sizeof(T) == 8 ? T(1e-290) : T(1e-35), hi = sizeof(T) == 8 ? T(1e290) : T(1e35);
    if (d > lo && d < hi) {
        const T s = T(1) / d;
        return make2<T2>(a.x * s, -a.y * s);
    }
    if (fabs(a.x) >= fabs(a.y)) {
        const T r = a.y / a.x, q = a.x + a.y * r;
        return make2<T2>(T(1) / q, -r / q);
    }
    const T r = a.x / a.y, q = a.x * r + a.y;
    return make2<T2>(r / q, -T(1) / q);
}

// a CTA's proposal for one column
template <class T2> struct Slot {
    typename Real<T2>::t val;   // |re| + |im|; -1: not comparable (NaN), -2: no row left
    int row;                     // local row
    int key;                     // global row
    T2 inv;                      // reciprocal of the pivot
    int zero;                    // the pivot is exactly zero
};

constexpr int MAX_CLUSTER = 16;

template <class T2> size_t smem_bytes(int n, int C) {
    const int rl = (n + C - 1) / C;
    return sizeof(T2) * ((size_t)rl * (n + 1) + 2 * n) + 2 * MAX_CLUSTER * sizeof(Slot<T2>) + sizeof(int) * (rl + 4) + 64;
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

// The best unused row of column c among this CTA's rows, proposed to every CTA of the
// cluster in slot set `par`; called by warp 0.  done: bit-per-row marks of the rows used.
template <class T2>
__device__ __forceinline__ void propose(const T2* rows, int ldr, int rl, int C, uint32_t rank, int c, const int* step, Slot<T2>* slots,
                                        int par) {
    using T = typename Real<T2>::t;
    const int lane = threadIdx.x & 31;
    T best = T(-2);
    int bl = 0;
    for (int r = lane; r < rl; r += 32) {
        if (step[r] >= 0) continue;
        const T2 v = rows[(size_t)r * ldr + c];
        T a = fabs(v.x) + fabs(v.y);
        if (!(a >= T(0))) a = T(-1);
        if (a > best) { best = a; bl = r; }
    }
    for (int o = 16; o > 0; o >>= 1) {
        const T ov = __shfl_xor_sync(0xffffffffu, best, o);
        const int ol = __shfl_xor_sync(0xffffffffu, bl, o);
        if (ov > best || (ov == best && ol < bl)) { best = ov; bl = ol; }
    }
    Slot<T2> s;
    s.val = best;
    s.row = bl;
    s.key = bl * C + (int)rank;
    s.zero = 0;
    s.inv = make2<T2>(T(1), T(0));
    if (best > T(-2)) {
        const T2 p = rows[(size_t)bl * ldr + c];
        if (p.x == T(0) && p.y == T(0)) s.zero = 1;
        else s.inv = inverse(p);
    }
    if (C == 1) {
        if (lane == 0) slots[par * MAX_CLUSTER] = s;
    } else if (lane < C) {
        *cl_map(slots + par * MAX_CLUSTER + rank, (uint32_t)lane) = s;
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
    T2* urow = rows + (size_t)rl_max * ldr;                    // pivot row over the pivot
    T2* invs = urow + n;                                       // reciprocals of the pivots
    Slot<T2>* slots = reinterpret_cast<Slot<T2>*>(invs + n);   // 2 sets of MAX_CLUSTER
    int* step = reinterpret_cast<int*>(slots + 2 * MAX_CLUSTER);   // pivot step of a local row, -1: not yet
    for (int r = warp; r < rl; r += nw)
        for (int c = lane; c < n; c += 32) rows[(size_t)r * ldr + c] = P.S[(size_t)(r * (int)C + (int)rank) * P.ld + c];
    for (int r = t; r < rl_max; r += NT) step[r] = -1;
    __syncthreads();
    if (C > 1) cl_sync();       // every CTA runs before its shared memory is written from outside
    if (warp == 0) propose(rows, ldr, rl, (int)C, rank, 0, step, slots, 0);
    int bad = 0;
    for (int j = 0; j < n; ++j) {
        if (C > 1) cl_sync();
        else __syncthreads();
        // the winner, by every warp on its own
        const Slot<T2>* set = slots + (j & 1) * MAX_CLUSTER;
        int w = lane < (int)C ? lane : 0;
        T best = set[w].val;
        int key = set[w].key;
        for (int o = (int)C >> 1; o > 0; o >>= 1) {
            const T ov = __shfl_xor_sync(0xffffffffu, best, o);
            const int ok = __shfl_xor_sync(0xffffffffu, key, o), ow = __shfl_xor_sync(0xffffffffu, w, o);
            if (ov > best || (ov == best && ok < key)) { best = ov; key = ok; w = ow; }
        }
        w = __shfl_sync(0xffffffffu, w, 0);
        const int lr = set[w].row;
        const T2 inv = set[w].inv;
        bad |= set[w].zero;
        const T2* prow = (C > 1 ? cl_map(rows, (uint32_t)w) : rows) + (size_t)lr * ldr;
        for (int c = j + 1 + t; c < n; c += NT) urow[c] = mul(prow[c], inv);
        if (t == 0) {
            invs[j] = inv;
            if (w == (int)rank) step[lr] = j;
        }
        __syncthreads();
        if (j + 1 == n) break;
        // A[r][c] -= A[r][j] urow[c] over the rows not used yet: warp 0 takes column j + 1
        // and proposes its pivot, the other warps the columns after it, a quarter of the
        // rows at a time
        if (warp == 0) {
            const T2 u = urow[j + 1];
            for (int r = lane; r < rl; r += 32)
                if (step[r] < 0) {
                    T2* a = rows + (size_t)r * ldr;
                    a[j + 1] = fnma(a[j + 1], a[j], u);
                }
            __syncwarp();
            propose(rows, ldr, rl, (int)C, rank, j + 1, step, slots, (j + 1) & 1);
        }
        const int cols = n - j - 2, segs = (cols + 31) / 32;
        const int groups = rl > 4 ? 4 : 1, per = (rl + groups - 1) / groups;
        for (int q = (warp + nw - 1) % nw; q < segs * groups; q += nw) {       // warp 0 joins last
            const int c = j + 2 + (q / groups) * 32 + lane, r0 = (q % groups) * per, r1 = min(rl, r0 + per);
            if (c >= n) continue;
            const T2 u = urow[c];
#pragma unroll 4
            for (int r = r0; r < r1; ++r)
                if (step[r] < 0) {
                    T2* a = rows + (size_t)r * ldr;
                    a[c] = fnma(a[c], a[j], u);
                }
        }
    }
    if (C > 1) cl_sync();       // no CTA leaves while its rows may be read; all reads of S are done
    for (int r = warp; r < rl; r += nw) {
        const int j = step[r];
        T2* out = P.F + (size_t)j * P.ld;
        for (int c = lane; c < n; c += 32) {
            const T2 v = rows[(size_t)r * ldr + c];
            out[c] = c < j ? mul(v, invs[c]) : v;
        }
        if (lane == 0) P.perm[j] = r * (int)C + (int)rank;
    }
    if (bad && rank == 0 && t == 0) atomicOr(P.status, PWQT_ST_SINGULAR_PIVOT);
}

// Cluster size for nb blocks of n x n: the one with the least waves x max(chain, update).
// 0: no size holds the rows in shared memory.  Chain and update per column in cycles, from
// the measurements above: FP64 1100 on one CTA, 1900 across a cluster, 2.4 per element of
// update; FP32 450, 1150 and 0.16.
template <class T2, class Where> int pick_cluster(int n, int nb, int sms, int smem_max) {
    const bool f64 = sizeof(T2) == 16;
    const double alpha = f64 ? 2.4 : 0.16;
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
        const double chain = C == 1 ? (f64 ? 1100 : 450) : (f64 ? 1900 : 1150);
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
