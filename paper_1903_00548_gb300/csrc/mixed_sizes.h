// Device memory of the mixed-precision path by block size, nodes, energies and injected modes
// (plain C++, no CUDA): what solve_mixed's buffers of a lane take, and whether those that a
// lane keeps hold a group of energies.
#pragma once
#include <algorithm>
#include <cstddef>
#include <cstdint>

namespace pwqt {

namespace oz {
constexpr int SL = 7;                    // slices per operand
constexpr int TM = 128;                  // real rows per tile
constexpr int TN = 32;                   // columns per tile
constexpr int KCH = 32;                  // real K per chunk (one bulk copy per operand)
constexpr uint32_t A_SLICE_BYTES = TM * KCH * 2;          // 8 KB
constexpr uint32_t B_SLICE_BYTES = TN * KCH * 2;          // 2 KB
constexpr uint32_t A_CHUNK_BYTES = SL * A_SLICE_BYTES;    // 56 KB
constexpr uint32_t B_CHUNK_BYTES = SL * B_SLICE_BYTES;    // 14 KB

inline int padded(int n) { return (n + 63) / 64 * 64; }   // n rounded up to a multiple of 64
inline int col_tiles(int ncols) { return (ncols + TN - 1) / TN; }
inline size_t panel_bytes(int n, int items, int nseg) {
    const int n_pad = padded(n);
    return (size_t)items * (2 * n_pad / TM) * nseg * (2 * n_pad / KCH) * A_CHUNK_BYTES;
}
inline size_t panel_item_bytes(int n, int nseg) { return panel_bytes(n, 1, nseg); }
inline size_t rexp_bytes(int n, int items) { return sizeof(int) * (size_t)items * 2 * padded(n); }
inline size_t b_bytes(int n, int N, int ncols) {
    const int n_pad = padded(n), nct = col_tiles(ncols);
    return (size_t)N * nct * (2 * n_pad / KCH) * B_CHUNK_BYTES;
}
}  // namespace oz

constexpr int PW = 32;                // panel width of the tensor-core sweep
constexpr int MV_INTS = 4 * PW + 4;   // per energy: count, then 2 PW destination and 2 PW source rows

inline size_t mixed_bytes_per_energy(int n, int N, int m) {
    // F + XY + L_i (complex64) + pivots + FP64 solution and residual
    constexpr size_t c64 = 8, c128 = 16;
    const size_t w = (size_t)n + m + (m & 1);
    return c64 * ((size_t)N * n * n + (size_t)N * n * w + (size_t)N * n * n) + sizeof(int) * ((size_t)N * n + MV_INTS) + 256 +
           3 * c128 * (size_t)N * n * m +                 // FP64 solution, residual, float-float copy
           2 * oz::panel_item_bytes(n, 1) +               // self-energy slice panels
           oz::b_bytes(n, N, m + 32);                     // solution slices (a column tile of slack)
}

// The buffers of a lane that grow with the group, in bytes.
struct MixedSizes {
    size_t ws = 0;                                        // factors, panels, solution (ws_mixed)
    size_t sig_tab = 0, sig = 0, sig_rexp = 0, B = 0, fexp = 0, act = 0;     // sliced residual (oz_*)
    bool hold(const MixedSizes& need) const {
        return ws >= need.ws && sig_tab >= need.sig_tab && sig >= need.sig && sig_rexp >= need.sig_rexp && B >= need.B &&
               fexp >= need.fexp && act >= need.act;
    }
};

// what a group of g energies of at most m columns (m >= 1) needs
inline MixedSizes mixed_sizes(int n, int N, int g, int m, bool sliced) {
    MixedSizes s;
    s.ws = mixed_bytes_per_energy(n, N, m) * g + 1024 * 4;
    if (sliced) {
        s.sig_tab = sizeof(void*) * 2 * (size_t)g;
        s.sig = oz::panel_bytes(n, 2 * g, 1);
        s.sig_rexp = oz::rexp_bytes(n, 2 * g);
        s.B = oz::b_bytes(n, N, g * m);
        s.fexp = sizeof(int) * (size_t)oz::col_tiles(g * m) * oz::TN;
        s.act = sizeof(int) * (size_t)g;
    }
    return s;
}

// energies of a batch of nb on lane 0; the others run beside them on lane 1
inline int lane_split(int nb) { return nb >= 16 ? nb / 2 : nb; }

// whether buffers of the lanes' sizes hold all nE energies (cols[e] columns each) in one batch
inline bool lanes_hold(const MixedSizes (&lane)[2], int n, int N, int nE, const int* cols, bool sliced) {
    const int at[3] = {0, lane_split(nE), nE};
    for (int q = 0; q < 2; ++q) {
        int m = 1;
        for (int e = at[q]; e < at[q + 1]; ++e) m = std::max(m, cols[e]);
        if (at[q] < at[q + 1] && !lane[q].hold(mixed_sizes(n, N, at[q + 1] - at[q], m, sliced))) return false;
    }
    return true;
}

}  // namespace pwqt
