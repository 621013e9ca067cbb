// Host-side check of PpWalk (which places of the item list a CTA of the ping-pong kernel takes):
// CTAs start in every kind of order, some when the kernel begins, the others only when a running one
// has ended or never, because a running CTA cancelled their launch and took over their share; whatever
// the order, every place of the list has to be taken exactly once.  Built and run by
// tests/test_host_logic.py; needs no GPU.
#include <cstdio>
#include <random>
#include <vector>
#include "../../paper_2410_16663_b200/csrc/prefill_pingpong.cuh"

static long long g_runs = 0;

// One launch: deal_ctas CTAs with `rounds` dealt places each and `rest` more places.  `resident` CTAs can
// run at once (while `others` of them are held by another kernel).  order: 0 = CTAs start lowest first,
// 1 = highest first, 2 = in a random order; a claim is declined now and then although CTAs are left.
static bool run(int deal_ctas, int rounds, int rest, int resident, int order, unsigned seed, bool late_starts) {
    const int total = deal_ctas * rounds + rest, grid = (rounds > 0 ? deal_ctas : 0) + rest;
    const int dealing = rounds > 0 ? deal_ctas : 0;
    std::mt19937 rng(seed);
    std::vector<int> waiting(grid), taken(total, 0);
    for (int i = 0; i < grid; ++i) waiting[i] = order == 0 ? grid - 1 - i : i;   // taken from the back
    auto next_waiting = [&]() {
        if (order == 2) std::swap(waiting[rng() % waiting.size()], waiting.back());
        const int x = waiting.back();
        waiting.pop_back();
        return x;
    };
    std::vector<fa::PpWalk> running;
    while (!waiting.empty() || !running.empty()) {
        // the hardware starts CTAs while there is room, and there always is when nothing runs
        while (!waiting.empty() && (int)running.size() < resident && (late_starts || running.empty() || (int)running.size() + (int)waiting.size() == grid))
        {
            running.push_back({dealing, rounds});
            running.back().take(next_waiting());
        }
        const int i = (int)(rng() % running.size());
        fa::PpWalk& w = running[i];
        if (w.used_up()) {
            const bool answered = !waiting.empty() && rng() % 16 != 0;
            if (!answered) {   // the CTA ends
                running[i] = running.back();
                running.pop_back();
                continue;
            }
            w.take(next_waiting());
        }
        const int at = w.next();
        if (at < 0 || at >= total) {
            std::printf("place %d of %d\n", at, total);
            return false;
        }
        ++taken[at];
    }
    ++g_runs;
    for (int i = 0; i < total; ++i)
        if (taken[i] != 1) {
            std::printf("place %d taken %d times: %d CTAs x %d rounds + %d, %d resident, order %d\n", i, taken[i], dealing, rounds, rest, resident, order);
            return false;
        }
    return true;
}

int main() {
    bool ok = true;
    const int ctas = 148;
    for (int rounds = 0; rounds <= 13 && ok; ++rounds)
        for (int rest : {1, 2, 16, 68, 147, 148, 149, 296, 443})
            for (int resident : {1, 2, 100, 116, 132, 147, 148, 1000})
                for (int order = 0; order < 3; ++order)
                    for (int late = 0; late < 2 && ok; ++late)
                        ok = run(ctas, rounds, rest, resident, order, 17u * rounds + rest + resident, late != 0);
    for (int ctas2 : {1, 2, 3, 20})
        for (int rounds = 1; rounds <= 5; ++rounds)
            for (int rest = 0; rest <= 2 * ctas2 && ok; ++rest)
                for (int resident = 1; resident <= ctas2 + 1 && ok; ++resident) ok = run(ctas2, rounds, rest, resident, 2, rest, true);
    std::printf("%s %lld launches\n", ok ? "OK" : "FAILED", g_runs);
    return ok ? 0 : 1;
}
