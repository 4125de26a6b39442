// The ticket protocol of the one-kernel scoring on host threads: CTAs take ranges i, i + P, ... of the units, some give up on a
// wait.  Prints a line per failed check; exit status 1 when there was one.
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <thread>
#include <vector>

#include "tickets.h"

struct Case {
    int units, ranges, ctas;
    int fail_cta, fail_at, kind;  // kind 0: nobody fails; 1: its own statistics are never written; 2: its wait for all runs out
};

static int run(const Case &c, std::vector<int> &counters) {
    const finch::Tickets t{counters.data(), counters.data() + c.units, c.ranges};
    std::vector<std::atomic<int>> written(c.units);
    for (auto &w : written) w = 0;
    std::atomic<int> early{0}, passed{0};
    auto cta = [&](int i) {
        bool good = true;
        int step = 0;
        for (int rho = i; rho < c.units * c.ranges; rho += c.ctas, ++step) {
            const int unit = rho / c.ranges;
            const bool hit = i == c.fail_cta && step == c.fail_at;
            good = t.pass(
                unit, good,
                [&]() {
                    if (hit && c.kind == 1) return false;
                    ++written[unit];
                    return true;
                },
                [&](const int *counter, int n) {
                    if (hit && c.kind == 2) return false;
                    for (int spin = 0; spin < 2000000; ++spin) {
                        if (__atomic_load_n(counter, __ATOMIC_ACQUIRE) >= n) {
                            if (written[unit] < n) ++early;
                            return true;
                        }
                        std::this_thread::yield();
                    }
                    return false;
                });
            passed += good;
        }
    };
    std::vector<std::thread> threads;
    for (int i = 0; i < c.ctas; ++i) threads.emplace_back(cta, i);
    for (auto &th : threads) th.join();
    int bad = 0;
    for (int v : counters) bad += v != 0;
    if (c.kind == 0 && (early || passed != c.units * c.ranges)) ++bad;
    if (c.kind != 0 && passed == c.units * c.ranges) ++bad;  // the failure did not happen
    return bad;
}

int main() {
    int bad = 0;
    const int shapes[][3] = {{3, 4, 6}, {5, 1, 2}, {4, 3, 12}, {7, 8, 8}};  // the last two: all ranges of a unit at once
    for (auto &s : shapes) {
        std::vector<int> counters(2 * s[0], 0);
        for (int kind = 0; kind < 3; ++kind)
            for (int cta = 0; cta < s[2]; ++cta) {
                const Case c{s[0], s[1], s[2], cta, kind == 0 ? 0 : (cta % 2 ? 0 : (s[0] * s[1] / s[2] > 1)), kind};
                if (cta + c.fail_at * s[2] >= s[0] * s[1]) continue;
                int b = run(c, counters);
                if (b) std::printf("units %d ranges %d ctas %d: CTA %d at %d, kind %d: %d\n", s[0], s[1], s[2], cta, c.fail_at, kind, b);
                // the next call, with whatever this one left behind
                const Case next{s[0], s[1], s[2], -1, 0, 0};
                const int b2 = run(next, counters);
                if (b2) std::printf("  the call after it: %d\n", b2);
                bad += b + b2;
                counters.assign(counters.size(), 0);
            }
    }
    return bad ? EXIT_FAILURE : EXIT_SUCCESS;
}
