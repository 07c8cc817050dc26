// Host-only checks of mixed_sizes.h: lanes whose buffers grow as a solve grows them, over calls
// of different block sizes, node and energy counts and residual kinds.  A call is held exactly
// when no buffer of either lane would have to grow for it.
#include <cstdio>
#include <random>
#include <vector>

#include "mixed_sizes.h"

using namespace pwqt;
static int fails = 0;
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); ++fails; } } while (0)

struct Call { int n, N; std::vector<int> cols; bool sliced; };

// grow-only, an eighth of slack; returns whether any buffer grew
static bool grow(size_t& have, size_t need) {
    if (have >= need) return false;
    have = need + need / 8;
    return true;
}
static bool run(MixedSizes (&lane)[2], const Call& c) {
    const int nE = (int)c.cols.size(), a = nE >= 16 ? nE / 2 : nE, lo[2] = {0, a}, hi[2] = {a, nE};
    bool grew = false;
    for (int q = 0; q < 2; ++q) {
        if (lo[q] == hi[q]) continue;
        int m = 1;
        for (int e = lo[q]; e < hi[q]; ++e) m = std::max(m, c.cols[e]);
        const MixedSizes s = mixed_sizes(c.n, c.N, hi[q] - lo[q], m, c.sliced);
        for (auto f : {&MixedSizes::ws, &MixedSizes::sig_tab, &MixedSizes::sig, &MixedSizes::sig_rexp, &MixedSizes::B, &MixedSizes::fexp, &MixedSizes::act})
            grew = grow(lane[q].*f, s.*f) || grew;
    }
    return grew;
}
static bool held(const MixedSizes (&lane)[2], const Call& c) { return lanes_hold(lane, c.n, c.N, (int)c.cols.size(), c.cols.data(), c.sliced); }

int main() {
    // the residual kind changed: the factors' workspace is there, the slices' buffers are not
    {
        MixedSizes lane[2];
        run(lane, {512, 20, std::vector<int>(8, 96), false});
        CHECK(held(lane, {512, 20, std::vector<int>(8, 96), false}));
        CHECK(!held(lane, {512, 20, std::vector<int>(8, 96), true}));
        CHECK(!held(lane, {64, 20, std::vector<int>(2, 10), true}));
    }
    // from a large block to a small one with many columns: the workspace holds it, the slices of
    // the solution do not
    {
        MixedSizes lane[2];
        run(lane, {512, 50, {1, 1}, true});
        const Call small{66, 50, std::vector<int>(15, 40), true};
        CHECK(lane[0].ws >= mixed_sizes(66, 50, 15, 40, true).ws);
        CHECK(lane[0].B < mixed_sizes(66, 50, 15, 40, true).B);
        CHECK(!held(lane, small));
    }
    std::mt19937 rng(7);
    auto pick = [&](int lo, int hi) { return std::uniform_int_distribution<int>(lo, hi)(rng); };
    int yes = 0, no = 0;
    for (int seq = 0; seq < 300; ++seq) {
        MixedSizes lane[2];
        for (int k = 0; k < 8; ++k) {
            Call c{2 * pick(3, 256), pick(2, 60), {}, pick(0, 3) > 0};
            const int nE = pick(1, 40);
            for (int e = 0; e < nE; ++e) c.cols.push_back(pick(0, c.n / 4));
            const bool h = held(lane, c);
            (h ? yes : no)++;
            CHECK(h == !run(lane, c));
            CHECK(held(lane, c));          // the same call again allocates nothing
        }
    }
    CHECK(yes > 100 && no > 100);
    std::printf(fails ? "FAILED\n" : "passed\n");
    return fails != 0;
}
