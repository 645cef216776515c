// Host-side run of the operator-splitting solve's barrier (osbarrier.cuh): threads
// in place of blocks, waits short enough to give up now and then, a round of
// barriers in place of a solve.  Either every thread gets through the last
// barrier of a round or none does.  Then the orders of two arrivals by
// one thread.  Prints "passed given_up disagreed wrong".
#include "../../paper_1107_5719_gb300/csrc/osbarrier.cuh"

#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>

using namespace rt3d;

struct HostWord {
    std::atomic<unsigned long long>* p;
    void arrive(unsigned long long x) { p->fetch_add(x, std::memory_order_release); }
    unsigned long long load() { return p->load(std::memory_order_acquire); }
    unsigned long long cas(unsigned long long seen, unsigned long long x)
    {
        p->compare_exchange_strong(seen, x, std::memory_order_acquire);
        return seen;
    }
};

int main()
{
    constexpr int kRounds = 6000, kBarriers = 4;
    long long passed = 0, gone = 0, disagreed = 0, wrong = 0;
    for (int nblk : {2, 3, 5}) {
        std::vector<std::atomic<unsigned long long>> words((size_t)kRounds * kBarriers);
        for (auto& w : words) w = 0;
        std::vector<std::vector<int>> got(nblk, std::vector<int>(kRounds, -1));
        std::atomic<int> ready{0}, bad{0};
        auto count = [&](int r, int q) {
            int more = 0;
            for (int b = 0; b < nblk; ++b) more += (b + r + q) % 2 == 0;
            return more;
        };
        auto run = [&](int b) {
            unsigned x = 12345u + 977u * b;
            auto rnd = [&] { return x = x * 1664525u + 1013904223u, x >> 16; };
            ready.fetch_add(1);
            while (ready.load() < nblk) std::this_thread::yield();
            for (int r = 0; r < kRounds; ++r)
                for (int q = 0; q < kBarriers; ++q) {
                    const bool last = q + 1 == kBarriers;
                    // short waits at the last barrier of every other round, at all
                    // of them in every eighth
                    const int polls = r % 8 == 0 || (last && r % 2) ? 1 + (int)(rnd() % 3) : 1 << 18;
                    for (unsigned n = rnd() % 64; n > 0; --n) (void)words[0].load();
                    if (rnd() % 256 == 0) std::this_thread::yield();
                    const HostWord w{&words[(size_t)r * kBarriers + q]};
                    int left = bar_wait(w, nblk, (b + r + q) % 2 == 0, polls);
                    if (left < 0 && last) {
                        for (unsigned n = rnd() % 64; n > 0; --n) (void)words[0].load();
                        left = bar_settle(w, nblk);
                    }
                    if (left < 0) break;
                    if (left != count(r, q)) ++bad;
                    if (last) got[b][r] = left;
                }
        };
        std::vector<std::thread> th;
        for (int b = 0; b < nblk; ++b) th.emplace_back(run, b);
        for (auto& t : th) t.join();
        wrong += bad;
        for (int r = 0; r < kRounds; ++r) {
            bool same = true;
            for (int b = 0; b < nblk; ++b) same &= got[b][r] == got[0][r];
            if (!same) ++disagreed;
            else ++(got[0][r] < 0 ? gone : passed);
        }
    }
    {
        // the other arrives after the wait gave up, before or after it is settled
        std::atomic<unsigned long long> a{0}, b{0};
        wrong += bar_wait(HostWord{&a}, 2, true, 3) != -1;
        wrong += bar_wait(HostWord{&a}, 2, true, 3) != 2;
        wrong += bar_settle(HostWord{&a}, 2) != 2;
        wrong += bar_wait(HostWord{&b}, 2, true, 3) != -1;
        wrong += bar_settle(HostWord{&b}, 2) != -1;
        wrong += bar_wait(HostWord{&b}, 2, true, 3) >= 0;
        wrong += bar_settle(HostWord{&b}, 2) >= 0;
    }
    std::printf("%lld %lld %lld %lld\n", passed, gone, disagreed, wrong);
    return 0;
}
