// FirstUse on the host: threads of several "contexts" fill entries of several block sizes at
// once.  While a first entry is computed nobody else is inside, each size has one first use,
// a failed one is not counted, and fills of known sizes overlap.
#include <atomic>
#include <chrono>
#include <cstdio>
#include <map>
#include <thread>
#include <vector>

#include "first_use.h"

using namespace std::chrono_literals;
static int fails = 0;
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); ++fails; } } while (0)

int main() {
    pwqt::FirstUse gate;
    std::atomic<int> inside{0}, most{0}, shared_with_first{0};
    std::atomic<int> firsts[4] = {};
    std::atomic<bool> fail_next{true};
    auto fill = [&](int ctx, int n) {
        pwqt::FirstUse::Pass p(gate, 0, n);
        const int now = ++inside;
        int m = most.load();
        while (now > m && !most.compare_exchange_weak(m, now)) {}
        if (p.first()) {
            if (now != 1) ++shared_with_first;
            std::this_thread::sleep_for(3ms);
            if (inside.load() != 1) ++shared_with_first;
            if (n == 3 && fail_next.exchange(false)) { --inside; return; }     // its entry fails: known() is not reached
            ++firsts[n];
            --inside;               // others may enter from here on
            p.known();
            ++inside;
        }
        std::this_thread::sleep_for(1ms);
        --inside;
        (void)ctx;
    };
    std::vector<std::thread> th;
    for (int ctx = 0; ctx < 12; ++ctx)
        th.emplace_back([&, ctx] { for (int r = 0; r < 12; ++r) fill(ctx, 1 + (ctx + r) % 3); });
    for (auto& t : th) t.join();
    CHECK(shared_with_first == 0);
    CHECK(firsts[1] == 1 && firsts[2] == 1 && firsts[3] == 1);
    CHECK(most > 1);                // known sizes run side by side
    // another device's first use of a known size is one
    { pwqt::FirstUse::Pass p(gate, 1, 1); CHECK(p.first()); p.known(); CHECK(!p.first()); }
    { pwqt::FirstUse::Pass p(gate, 1, 1); CHECK(!p.first()); }
    // a first use is not kept waiting by a stream of fills
    std::atomic<bool> stop{false};
    std::vector<std::thread> stream;
    for (int k = 0; k < 3; ++k)
        stream.emplace_back([&] { while (!stop) { pwqt::FirstUse::Pass p(gate, 0, 1); std::this_thread::sleep_for(500us); } });
    { pwqt::FirstUse::Pass p(gate, 0, 7); CHECK(p.first()); p.known(); }
    stop = true;
    for (auto& t : stream) t.join();
    std::printf(fails ? "FAILED\n" : "passed\n");
    return fails != 0;
}
