// Complex64 block sweep for blocks whose rows a small cluster holds in shared memory.
#pragma once
#include <cuda_runtime.h>

#include "sweep_common.cuh"

namespace pwqt {

// The arrays of the mixed-precision path that the sweep fills; entry e of X at X + e sX.
struct C64Sweep {
    SweepSys sys;
    const SweepJob* jobs;
    int m, w;                      // uniform column count and row length of [X_i | y_i]
    float2* F; long long sF;       // N n x n factors (row-permuted, unit lower)
    int* perm; long long sP;       // N x n: (P x)_j = x[perm[j]]
    float2* XY; long long sXY;     // N n x w
    float2* Lb; long long sL;      // N n x n couplings L_i = A_{i,i-1}
    double2* C64; long long sC;    // N n x m solution
};

// whether the block size has this form on a device with smem_max bytes of shared memory a CTA
// (25 .. 320, the sizes that its tests cover.  It is the faster one beyond both ends too: mixed
// solve of 60 nodes and 32 energies, tensor-core form and this, n = 8 6.2 and 2.4 ms, n = 16 7.4
// and 3.3, n = 24 8.7 and 4.2; above 320 see lup::pick_cluster)
bool c64_sweep_fits(int n, int smem_max);
// factors, couplings, X_i and the solution of nb energies (jobs; host: the same table on the
// host); returns the number of kernels launched
int c64_sweep(const C64Sweep& S, const SweepJob* host, int nb, int sms, int smem_max, cudaStream_t st);

}  // namespace pwqt
